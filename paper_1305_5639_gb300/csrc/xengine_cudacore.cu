// X-engine on CUDA cores (Eq. 2, Section 2): the plain baseline and the FP32 path.
//
// FP32: one CTA per channel and square tile of the lower triangle (Section 4), register
// tiles (fp32_tile.cuh); one CTA per channel for few inputs.
//
// INT8: one CTA computes a 64 x 64 block of input pairs (I-block >= J-block) for one
// channel; 256 threads each own a 4 x 4 register block of pairs. Spectra are staged in
// shared memory in chunks, transposed to [spectrum][input] so that every thread reads
// broadcast / conflict-free.
//   INT8:  complex int8 input, exact INT32 result with dp4a: a 32-bit word holds
//          (re, im) of two consecutive spectra, so
//            Re V_ij += dp4a([re_i im_i ...], [re_j im_j ...])
//            Im V_ij += dp4a([im_i ~re_i ...], [re_j im_j ...]) + sum(im_j)
//          with ~re = -re - 1 (bitwise not), representable for every int8 code
//          including -128 (whose negation is not): the -1 terms sum to -sum(im_j),
//          which a per-column dp4a with [0 1 0 1] adds back.
#include <algorithm>
#include <cmath>

#include "fp32_tile.cuh"
#include "internal.h"

namespace corr {
namespace {

constexpr int TB = 64;          // INT8: inputs per tile side
constexpr int NTH = 256;        // INT8: threads (16 x 16)
constexpr int KC_I = 32;        // INT8: spectra per chunk (16 words)
constexpr int PAD = TB + 1;

__device__ __forceinline__ void tile_of(int t, int &bi, int &bj) {
    // t -> (bi, bj), bi >= bj, row-major over the lower triangle of blocks
    int r = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= t) ++r;
    while (r * (r + 1) / 2 > t) --r;
    bi = r;
    bj = t - r * (r + 1) / 2;
}

// g_i conj(g_j) v
__device__ __forceinline__ float2 apply_gains(float2 v, float2 gi, float2 gj) {
    const float2 w = make_float2(gi.x * gj.x + gi.y * gj.y, gi.y * gj.x - gi.x * gj.y);
    return make_float2(v.x * w.x - v.y * w.y, v.x * w.y + v.y * w.x);
}

// FP32 tiles (fp32_tile.cuh): TB = 16 CT inputs square, CT = 2, 3 or 4, one CTA per
// (channel, lower-triangle tile). On a diagonal tile the warp wholly above the diagonal
// skips its sums and the rows are loaded once for both sides. Measured against one 64 x 64
// tile of 4 x 4 sums per 256-thread CTA with synchronous loads: 158 -> 87 us for 130
// inputs, 64 channels, 500 spectra; 207 -> 60 us for 24 inputs, 256 channels, 1024
// spectra; 1643 -> 1445 us (47.7 TFLOP/s) for 512 inputs, 64 channels, 1024 spectra.
template <int CT>
struct XfCfg {
    static constexpr int RT = 2 * CT, TB = 16 * CT, P = TB + 2;
    static constexpr int kSide = kFtKC * P;  // values of one operand of one stage
    static constexpr size_t smem = sizeof(float2) * 2 * kFtStages * kSide;
};

template <int CT>
__global__ void __launch_bounds__(kFtNth, 4) k_xeng_f32(const float2 *__restrict__ X, float2 *__restrict__ acc,
                                                        const float2 *__restrict__ gains, int n_in, int K,
                                                        long long B, int n_tiles, int store) {
    using C = XfCfg<CT>;
    constexpr int RT = C::RT, TB = C::TB, P = C::P;
    extern __shared__ __align__(16) float2 sm[];  // [stage][I side, J side][KC][P]
    const int chan = (int)(blockIdx.x / (unsigned)n_tiles);
    int bi, bj;
    tile_of((int)(blockIdx.x % (unsigned)n_tiles), bi, bj);
    const bool diag = bi == bj;
    const int I0 = bi * TB, J0 = bj * TB;
    const float2 *Xc = X + (size_t)chan * n_in * K;
    const FtPos<RT, CT> pos;
    const bool live = !(diag && pos.wr < pos.wc);  // this warp's quarter meets the lower triangle

    // loader: spectrum threadIdx.x % 16 of the stage, rows threadIdx.x / 16 + 8 q
    const int ks = threadIdx.x % kFtKC, row = threadIdx.x / kFtKC;
    const int n_st = (K + kFtKC - 1) / kFtKC;
    auto issue = [&](int st) {
        if (st < n_st) {
            float2 *sj = sm + ((st % kFtStages) * 2 + 1) * C::kSide + ks * P + row, *si = sj - C::kSide;
            const int a = st * kFtKC + ks;
#pragma unroll
            for (int q = 0; q < TB / 8; ++q) {
                const int gj = J0 + row + 8 * q, gi = I0 + row + 8 * q;
                const bool lj = gj < n_in && a < K, li = gi < n_in && a < K;
                ft_copy8(sj + 8 * q, lj ? Xc + (size_t)gj * K + a : X, lj);
                if (!diag) ft_copy8(si + 8 * q, li ? Xc + (size_t)gi * K + a : X, li);
            }
        }
        ft_commit();
    };
    float2 sum[RT][CT];
    ft_zero(sum);
#pragma unroll
    for (int st = 0; st < kFtStages - 1; ++st) issue(st);
    for (int st = 0; st < n_st; ++st) {
        ft_wait();
        __syncthreads();  // stage st has landed, and every warp is done with stage st - 1
        issue(st + kFtStages - 1);
        const float2 *sj = sm + ((st % kFtStages) * 2 + 1) * C::kSide, *si = diag ? sj : sj - C::kSide;
        if (live) ft_stage<true, RT, CT, P, P>(sum, si + pos.row0, sj + pos.col0);
    }
    if (!live) return;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const int i = I0 + pos.row(r);
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            const int j = J0 + pos.col(c);
            if (i < n_in && j <= i) {
                float2 v = sum[r][c];
                if (gains) v = apply_gains(v, __ldg(gains + i), __ldg(gains + j));
                const size_t b = (size_t)chan * B + (size_t)i * (i + 1) / 2 + j;
                if (!store) {
                    const float2 o = acc[b];
                    v = make_float2(o.x + v.x, o.y + v.y);
                }
                acc[b] = v;
            }
        }
    }
}

template <int CT>
corr_status launch_f32(const Handle &h, const float2 *X, const float2 *gains, bool store, cudaStream_t st) {
    using C = XfCfg<CT>;
    const int nb = (h.n_in + C::TB - 1) / C::TB;
    const long long n_tiles = (long long)nb * (nb + 1) / 2;
    if (n_tiles * h.n_chan > 0x7fffffffLL) return CORR_EUNSUPPORTED;
    constexpr auto kern = k_xeng_f32<CT>;
    if (const corr_status e = allow_smem<kern>((int)C::smem); e != CORR_OK) return e;
    kern<<<(unsigned)(n_tiles * h.n_chan), kFtNth, C::smem, st>>>(X, static_cast<float2 *>(h.acc), gains, h.n_in,
                                                                 h.n_spectra, h.n_base, (int)n_tiles, store ? 1 : 0);
    return CORR_OK;
}

// Tile edge of the FP32 X-engine: the one whose busiest SM forms the fewest products,
// weighed by each tile's rate (operand reads per FMA grow as the tile shrinks). 130 inputs:
// six tiles of 48 (13,824 products) against six of 64 (24,576) for 8,515 pairs.
int f32_tile_ct(const Handle &h) {
    int best = 4;
    double least = 0.0;
    for (int ct = 4; ct >= 2; --ct) {
        const int tb = 16 * ct, nb = (h.n_in + tb - 1) / tb;
        const double tiles = 0.5 * nb * (nb + 1) - 0.25 * nb;  // diagonal tiles skip a quarter
        const double per_sm = std::ceil(0.5 * nb * (nb + 1) * h.n_chan / h.n_sm) / (0.5 * nb * (nb + 1));
        const double cost = tiles * per_sm * tb * tb * (ct == 4 ? 1.0 : ct == 3 ? 1.08 : 1.3);
        if (ct == 4 || cost < least) best = ct, least = cost;
    }
    return best;
}

// Few inputs (n_in <= kSmallIn): one CTA per channel; a task is a 4 x 4 block of the lower
// triangle over one K range (n_split of them), done by one warp with a lane per pair of
// spectra (per spectrum where K is odd), so that the rows are read straight from global
// memory, 512 contiguous bytes per warp and row, and every load feeds four products. The 32
// sums of a block (16 pairs, Re and Im) are then added over the lanes by a transposing
// butterfly that leaves sum number `lane` in each lane, and over the K ranges in order: a
// fixed order, so the result is run-to-run identical. Bound by the L1 reads (each row is
// read by the n_in / 4 + 1 blocks it meets) and the FP32 pipe: 14 us for 16 inputs, 256
// channels, 1024 spectra (33.5 MB: 5 us of HBM time), against 30.4 us with one thread per
// pair reading both factors of each product from shared memory. Twelve warps, two CTAs per
// SM: three tasks each at 36 blocks, and one CTA's reduction beside the other's loads (16
// inputs: 18.5 us with the dump against 20.8 with 20 warps, one CTA). Above 32 inputs the tiles
// of k_xeng_f32 have the better ratio of sums to reads (24 inputs, 256 channels, 1024
// spectra: 35 us here, 60 us there).
constexpr int kSmallIn = 32;     // at most 36 blocks
constexpr int kSmallWarps = 12;
constexpr int kSmallTasks = 36;  // blocks x K ranges

// the sums v[k] of all lanes: afterwards v[0] holds sum number `lane`
template <typename T>
__device__ __forceinline__ void butterfly32(T (&v)[32], int lane) {
    // after the step of width o, v[k] holds the sum over the lanes differing in bit o of
    // sum k (+ o for lanes with that bit set)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (k >= o) break;
            const bool up = (lane & o) != 0;
            const T send = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(32 * kSmallWarps, 2) k_xeng_f32_small(const float2 *__restrict__ X, float2 *__restrict__ acc,
                                                         const float2 *__restrict__ gains, int n_in, int K,
                                                         long long B, int n_blk, int n_split, int store) {
    __shared__ float part[kSmallTasks][32];
    const int chan = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warp = blockDim.x >> 5;
    const float2 *Xc = X + (size_t)chan * n_in * K;
    const int step = VEC ? 64 : 32;
#pragma unroll 1
    for (int task = warp; task < n_blk * n_split; task += n_warp) {
        int bi, bj;
        tile_of(task % n_blk, bi, bj);
        // rows past the end read the last one; their sums are not written
        const float2 *xi[4], *xj[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            xi[r] = Xc + (size_t)min(4 * bi + r, n_in - 1) * K;
            xj[r] = Xc + (size_t)min(4 * bj + r, n_in - 1) * K;
        }
        float v[32];  // sum 2 (4 r + c) + part of pair (4 bi + r, 4 bj + c)
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = 0.f;
        auto mac = [&](const float2 (&a)[4], const float2 (&b)[4]) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // x_i conj(x_j)
                    const int e = 2 * (4 * r + c);
                    v[e] = fmaf(a[r].x, b[c].x, fmaf(a[r].y, b[c].y, v[e]));
                    v[e + 1] = fmaf(a[r].y, b[c].x, fmaf(-a[r].x, b[c].y, v[e + 1]));
                }
        };
        for (int a = (task / n_blk) * step + (VEC ? 2 * lane : lane); a < K; a += n_split * step) {
            if (VEC) {
                float2 i0[4], i1[4], j0[4], j1[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float4 q = __ldg(reinterpret_cast<const float4 *>(xi[r] + a));
                    i0[r] = make_float2(q.x, q.y), i1[r] = make_float2(q.z, q.w);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float4 q = __ldg(reinterpret_cast<const float4 *>(xj[r] + a));
                    j0[r] = make_float2(q.x, q.y), j1[r] = make_float2(q.z, q.w);
                }
                mac(i0, j0);
                mac(i1, j1);
            } else {
                float2 i0[4], j0[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) i0[r] = __ldg(xi[r] + a), j0[r] = __ldg(xj[r] + a);
                mac(i0, j0);
            }
        }
        butterfly32(v, lane);
        part[task][lane] = v[0];
    }
    __syncthreads();
    for (int blk = warp; blk < n_blk; blk += n_warp) {
        int bi, bj;
        tile_of(blk, bi, bj);
        float s = part[blk][lane];
        for (int q = 1; q < n_split; ++q) s += part[blk + q * n_blk][lane];
        const float other = __shfl_xor_sync(0xffffffffu, s, 1);
        const int i = 4 * bi + (lane >> 3), j = 4 * bj + ((lane >> 1) & 3);
        if ((lane & 1) || i >= n_in || j > i) continue;
        float2 w = make_float2(s, other);
        if (gains) w = apply_gains(w, __ldg(gains + i), __ldg(gains + j));
        const size_t b = (size_t)chan * B + (size_t)i * (i + 1) / 2 + j;
        if (!store) {
            const float2 o = acc[b];
            w = make_float2(o.x + w.x, o.y + w.y);
        }
        acc[b] = w;
    }
}

__device__ __forceinline__ uint32_t rot_word(uint32_t w) {
    // bytes [re0 im0 re1 im1] -> [im0 ~re0 im1 ~re1] (~re = -re - 1)
    const uint32_t sw = __byte_perm(w, 0u, 0x2301);  // [im0 re0 im1 re1]
    return sw ^ 0xff00ff00u;
}
// dp4a weights picking the imaginary bytes of a word: [0 1 0 1]
constexpr int kImOnes = 0x01000100;

// INT8 with few inputs (n_in <= kSmallIn), as k_xeng_f32_small: a lane takes W words of two
// spectra per row and step (W = 4 where a row is whole 16-byte pieces, 1 for an even K; W = 0:
// single spectra), every word feeding four dp4a pairs. Reads the complex int8 layout
// directly, where the tensor cores need a conversion pass and spend a 128 x 128 tile on the
// few pairs. X-engine and dump, tensor cores -> here (us): 16 inputs, 256 channels, 1024
// spectra 39 -> 13; 8 inputs, 1024 channels, 512 spectra 70 -> 12; 32 inputs, 1024 channels,
// 4096 spectra 471 -> 233.
template <int W>
__global__ void __launch_bounds__(32 * kSmallWarps, 2) k_xeng_i8_small(const char2 *__restrict__ X, int2 *__restrict__ acc,
                                                                    int n_in, int K, long long B, int n_blk,
                                                                    int n_split, int store) {
    __shared__ int part[kSmallTasks][32];
    const int chan = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warp = blockDim.x >> 5;
    const char2 *Xc = X + (size_t)chan * n_in * K;
    constexpr int NW = W ? W : 1, S = W ? 2 * W : 1;  // words and spectra per lane and step
#pragma unroll 1
    for (int task = warp; task < n_blk * n_split; task += n_warp) {
        int bi, bj;
        tile_of(task % n_blk, bi, bj);
        const char2 *xi[4], *xj[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            xi[r] = Xc + (size_t)min(4 * bi + r, n_in - 1) * K;
            xj[r] = Xc + (size_t)min(4 * bj + r, n_in - 1) * K;
        }
        int v[32], cim[4] = {0, 0, 0, 0};
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = 0;
        auto load = [](const char2 *p, uint32_t (&w)[NW]) {
            if constexpr (W == 4) {
                const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p));
                w[0] = q.x, w[1] = q.y, w[2] = q.z, w[3] = q.w;
            } else if constexpr (W == 1) {
                w[0] = __ldg(reinterpret_cast<const unsigned int *>(p));
            } else {
                w[0] = __ldg(reinterpret_cast<const unsigned short *>(p));
            }
        };
        for (int a = ((task / n_blk) * 32 + lane) * S; a < K; a += n_split * 32 * S) {
            uint32_t wi[4][NW], wj[4][NW];
#pragma unroll
            for (int r = 0; r < 4; ++r) load(xi[r] + a, wi[r]);
#pragma unroll
            for (int r = 0; r < 4; ++r) load(xj[r] + a, wj[r]);
#pragma unroll
            for (int q = 0; q < NW; ++q) {
#pragma unroll
                for (int c = 0; c < 4; ++c) cim[c] = __dp4a((int)wj[c][q], kImOnes, cim[c]);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    // (a zero upper half rotates to (0, ~0): ~0 times the zero of x_j)
                    const int x = (int)wi[r][q], rx = (int)rot_word(wi[r][q]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int e = 2 * (4 * r + c);
                        v[e] = __dp4a(x, (int)wj[c][q], v[e]);
                        v[e + 1] = __dp4a(rx, (int)wj[c][q], v[e + 1]);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) v[2 * e + 1] += cim[e & 3];
        butterfly32(v, lane);
        part[task][lane] = v[0];
    }
    __syncthreads();
    for (int blk = warp; blk < n_blk; blk += n_warp) {
        int bi, bj;
        tile_of(blk, bi, bj);
        int s = part[blk][lane];
        for (int q = 1; q < n_split; ++q) s += part[blk + q * n_blk][lane];
        const int other = __shfl_xor_sync(0xffffffffu, s, 1);
        const int i = 4 * bi + (lane >> 3), j = 4 * bj + ((lane >> 1) & 3);
        if ((lane & 1) || i >= n_in || j > i) continue;
        int2 w = make_int2(s, other);
        const size_t b = (size_t)chan * B + (size_t)i * (i + 1) / 2 + j;
        if (!store) {
            const int2 o = acc[b];
            w = make_int2(o.x + w.x, o.y + w.y);
        }
        acc[b] = w;
    }
}

__global__ void __launch_bounds__(NTH) k_xeng_i8(const char2 *__restrict__ X, int2 *__restrict__ acc,
                                                 int n_in, int K, long long B, int store) {
    constexpr int KW = KC_I / 2;  // words per row per chunk
    __shared__ uint32_t si[KW][PAD];
    __shared__ uint32_t sr[KW][PAD];
    __shared__ uint32_t sj[KW][PAD];
    int bi, bj;
    tile_of(blockIdx.x, bi, bj);
    const int chan = blockIdx.y;
    const int I0 = bi * TB, J0 = bj * TB;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const char2 *Xc = X + (size_t)chan * n_in * K;

    int ar[4][4], ai[4][4];
    int cim[4] = {0, 0, 0, 0};  // sum of Im x_j over the spectra, per column
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) ar[r][c] = ai[r][c] = 0;

    for (int a0 = 0; a0 < K; a0 += KC_I) {
#pragma unroll
        for (int q = 0; q < (TB * KW) / NTH; ++q) {
            int e = threadIdx.x + NTH * q;
            int row = e / KW, w = e % KW;
            int gi = I0 + row, gj = J0 + row, ga = a0 + 2 * w;
            uint32_t vi = 0, vj = 0;
            if (gi < n_in) {
                const char2 *p = Xc + (size_t)gi * K + ga;
                char2 c0 = ga < K ? p[0] : make_char2(0, 0);
                char2 c1 = ga + 1 < K ? p[1] : make_char2(0, 0);
                vi = (uint32_t)(uint8_t)c0.x | ((uint32_t)(uint8_t)c0.y << 8) | ((uint32_t)(uint8_t)c1.x << 16) |
                     ((uint32_t)(uint8_t)c1.y << 24);
            }
            if (gj < n_in) {
                const char2 *p = Xc + (size_t)gj * K + ga;
                char2 c0 = ga < K ? p[0] : make_char2(0, 0);
                char2 c1 = ga + 1 < K ? p[1] : make_char2(0, 0);
                vj = (uint32_t)(uint8_t)c0.x | ((uint32_t)(uint8_t)c0.y << 8) | ((uint32_t)(uint8_t)c1.x << 16) |
                     ((uint32_t)(uint8_t)c1.y << 24);
            }
            si[w][row] = vi;
            sr[w][row] = rot_word(vi);
            sj[w][row] = vj;
        }
        __syncthreads();
#pragma unroll 4
        for (int w = 0; w < KW; ++w) {
            int xi[4], xr[4], xj[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                xi[r] = (int)si[w][ty + 16 * r];
                xr[r] = (int)sr[w][ty + 16 * r];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                xj[c] = (int)sj[w][tx + 16 * c];
                cim[c] = __dp4a(xj[c], kImOnes, cim[c]);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    ar[r][c] = __dp4a(xi[r], xj[c], ar[r][c]);
                    ai[r][c] = __dp4a(xr[r], xj[c], ai[r][c]);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        int i = I0 + ty + 16 * r;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            int j = J0 + tx + 16 * c;
            if (i < n_in && j <= i) {
                size_t b = (size_t)chan * B + (size_t)i * (i + 1) / 2 + j;
                const int im = ai[r][c] + cim[c];
                if (store) {
                    acc[b] = make_int2(ar[r][c], im);
                } else {
                    int2 o = acc[b];
                    acc[b] = make_int2(o.x + ar[r][c], o.y + im);
                }
            }
        }
    }
}

}  // namespace

bool xengine_i8_small(const Handle &h) {
    if (h.precision != CORR_PREC_INT8 || h.xengine != CORR_XENG_AUTO ||
        (h.flags & (CORR_FLAG_PLANAR | CORR_FLAG_FUSED_DUMP)))
        return false;
    // Where the two sides measure equal (X-engine with dump, us, here / tensor cores, 64 and
    // 1024 channels): 16-byte loads win up to 32 inputs (32 x 4000 spectra 39 / 60 and 235 /
    // 438). 4-byte loads win up to 28 inputs (28 x 4002: 57 / 60, 412 / 421), above that up to
    // 1000 spectra (32 x 1002: 25 / 25, 117 / 122; 32 x 4002: 68 / 60, 524 / 438). Single
    // spectra win up to 16 inputs (16 x 4001: 45 / 58, 319 / 379), up to 20 for 1500 spectra
    // (20 x 1001: 24 / 24, 95 / 112; 20 x 4001: 65 / 60, 455 / 399), up to 24 for 500 (24 x 401:
    // 17 / 19, 60 / 62; 24 x 1001: 28 / 25, 126 / 115; 24 x 4001: 81 / 60, 604 / 419).
    const int n = h.n_in, K = h.n_spectra;
    if (K % 8 == 0) return n <= kSmallIn;
    if (K % 2 == 0) return n <= 28 || (n <= kSmallIn && K <= 1000);
    return n <= 16 || (n <= 20 && K <= 1500) || (n <= 24 && K < 500);
}

corr_status launch_xengine_cudacore(const Handle &h, const void *chan_in, const float2 *gains, bool store,
                                    cudaStream_t st) {
    StageScope sc(h, CORR_STAGE_XENGINE, st);
    corr_status s = CORR_OK;
    const float2 *X = static_cast<const float2 *>(chan_in);
    if (h.n_in <= kSmallIn) {
        const int nb = (h.n_in + 3) / 4, n_blk = nb * (nb + 1) / 2;
        const bool i8 = h.precision == CORR_PREC_INT8;
        const int W = !i8 ? 0 : h.n_spectra % 8 == 0 ? 4 : h.n_spectra % 2 == 0 ? 1 : 0;
        // K ranges: as many tasks as warps, as long as each range has a few rounds
        const int round = i8 ? 32 * (W ? 2 * W : 1) : 64;
        const int n_split = std::max(1, std::min(kSmallWarps / n_blk, h.n_spectra / (4 * round)));
        const int threads = 32 * std::min(kSmallWarps, n_blk * n_split);
        if (i8) {
            auto kern = W == 4 ? k_xeng_i8_small<4> : W == 1 ? k_xeng_i8_small<1> : k_xeng_i8_small<0>;
            kern<<<h.n_chan, threads, 0, st>>>(static_cast<const char2 *>(chan_in), static_cast<int2 *>(h.acc), h.n_in,
                                               h.n_spectra, h.n_base, n_blk, n_split, store ? 1 : 0);
        } else {
            auto kern = (h.n_spectra % 2) == 0 ? k_xeng_f32_small<true> : k_xeng_f32_small<false>;
            kern<<<h.n_chan, threads, 0, st>>>(X, static_cast<float2 *>(h.acc), gains, h.n_in, h.n_spectra, h.n_base,
                                               n_blk, n_split, store ? 1 : 0);
        }
    } else if (h.precision == CORR_PREC_INT8) {
        const int nb = (h.n_in + TB - 1) / TB;
        dim3 grid(nb * (nb + 1) / 2, h.n_chan);
        k_xeng_i8<<<grid, NTH, 0, st>>>(static_cast<const char2 *>(chan_in), static_cast<int2 *>(h.acc), h.n_in,
                                        h.n_spectra, h.n_base, store ? 1 : 0);
    } else {
        const int ct = f32_tile_ct(h);
        s = ct == 2 ? launch_f32<2>(h, X, gains, store, st)
                    : ct == 3 ? launch_f32<3>(h, X, gains, store, st) : launch_f32<4>(h, X, gains, store, st);
        if (s != CORR_OK) return s;
    }
    return check_launch("k_xeng_cudacore");
}

}  // namespace corr
