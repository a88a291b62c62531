// Adjoint of the gained X-engine for gradient-based gain calibration.
//
// Forward (per channel f): V'_ij = g_i conj(g_j) sum_a X_ia conj(X_ja), i >= j.
// Given G = dL/dV' (PyTorch convention, packed i >= j) and its Hermitian
// completion G^ (G^_ij = G_ij for i > j, G^_ji = conj G_ij, G^_ii = 2 Re G_ii):
//     Y      = G^ diag(g) X                      (complex GEMM, n_in x n_in x K)
//     dL/dX  = diag(conj g) Y
//     dL/dg_m = sum_f sum_a conj(X_ma) Y_ma      (= sum_f sum_j G^_mj g_j V_jm)
// The dg reduction is fused into the GEMM epilogue: each CTA writes one partial
// per row into a workspace, and a second kernel sums the partials in a fixed
// order (bit-reproducible).
#include "fp32_tile.cuh"
#include "internal.h"

namespace corr {
namespace {

constexpr int CT = 4, TA = 16 * CT;  // spectra per tile (fp32_tile.cuh)

// G^_mj from the packed entry that holds it (G_mj, or G_jm above the diagonal)
__device__ __forceinline__ float2 ghat_load(const float2 *__restrict__ G, int m, int j, int n_in) {
    if (m >= n_in || j >= n_in) return make_float2(0.f, 0.f);
    const int r = max(m, j), c = min(m, j);
    return __ldg(G + (size_t)r * (r + 1) / 2 + c);
}
__device__ __forceinline__ float2 ghat_of(float2 v, int m, int j) {
    return m == j ? make_float2(2.0f * v.x, 0.0f) : make_float2(v.x, m > j ? v.y : -v.y);
}

// One CTA: TM = 8 RT rows m x 64 spectra a of Y for one channel (RT = 4, 6 or 8),
// operands A_mj = G^_mj g_j (through registers) and X_ja (asynchronous copies) staged in
// shared memory (fp32_tile.cuh). Rows of G^ left of the tile's rows are read along j
// (packed rows), those right of them along m (the packed rows of the conjugate), so both
// are contiguous. Measured against 64 x 64 tiles of 4 x 4 sums per 256-thread CTA with
// synchronous loads: 207 -> 132 us for 130 inputs, 64 channels, 500 spectra (48-row
// tiles), 3594 -> 2746 us (50 TFLOP/s) for 512 inputs, 64 channels, 1024 spectra.
template <int RT>
struct AdjCfg {
    static constexpr int TM = 8 * RT, PG = TM + 2, PZ = TA + 2;
    static constexpr int kBuf = kFtKC * (PG + PZ);  // values of one stage
    static constexpr size_t smem = sizeof(float2) * kFtStages * kBuf;
};

template <int RT>
__global__ void __launch_bounds__(kFtNth, 4) k_adj(const float2 *__restrict__ Gp, const float2 *__restrict__ X,
                                                   const float2 *__restrict__ gains, float2 *__restrict__ dX,
                                                   float2 *__restrict__ part, int n_in, int K, long long B, int nM,
                                                   int nA) {
    using C = AdjCfg<RT>;
    constexpr int TM = C::TM, PG = C::PG, PZ = C::PZ;
    extern __shared__ __align__(16) float2 sm[];  // [stage]{ A[KC][PG], X[KC][PZ] }
    const unsigned t = blockIdx.x / (unsigned)nM;
    const int M0 = (int)(blockIdx.x % (unsigned)nM) * TM;
    const int ab = (int)(t % (unsigned)nA), chan = (int)(t / (unsigned)nA);
    const int A0 = ab * TA;
    const float2 *Gc = Gp + (size_t)chan * B;
    const float2 *Xc = X + (size_t)chan * n_in * K;
    const FtPos<RT, CT> pos;
    const int n_st = (n_in + kFtKC - 1) / kFtKC;

    auto issue = [&](int st) {
        if (st < n_st) {
            float2 *sz = sm + (st % kFtStages) * C::kBuf + kFtKC * PG;
            const int col = threadIdx.x % TA, a = A0 + col;
#pragma unroll
            for (int q = 0; q < kFtKC * TA / kFtNth; ++q) {
                const int jj = threadIdx.x / TA + (kFtNth / TA) * q, j = st * kFtKC + jj;
                const bool live = j < n_in && a < K;
                ft_copy8(sz + jj * PZ + col, live ? Xc + (size_t)j * K + a : X, live);
            }
        }
        ft_commit();
    };
    // element q of this thread: row ml and contraction step jj of stage st's A tile
    float2 gv[RT];
    auto g_at = [&](int st, int q, int &ml, int &jj) {
        const int e = threadIdx.x + kFtNth * q;
        const bool along_j = (st + 1) * kFtKC <= M0 + TM;
        ml = along_j ? e / kFtKC : e % TM;
        jj = along_j ? e % kFtKC : e / TM;
    };
    auto fetch = [&](int st) {
        if (st >= n_st) return;
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            int ml, jj;
            g_at(st, q, ml, jj);
            gv[q] = ghat_load(Gc, M0 + ml, st * kFtKC + jj, n_in);
        }
    };
    // the arithmetic on the loaded entries waits until they are stored, a stage later
    auto put = [&](int st) {
        if (st >= n_st) return;
        float2 *sg = sm + (st % kFtStages) * C::kBuf;
#pragma unroll
        for (int q = 0; q < RT; ++q) {
            int ml, jj;
            g_at(st, q, ml, jj);
            const int j = st * kFtKC + jj;
            const float2 v = ghat_of(gv[q], M0 + ml, j);
            const float2 g = gains && j < n_in ? __ldg(gains + j) : make_float2(1.f, 0.f);
            sg[jj * PG + ml] = make_float2(v.x * g.x - v.y * g.y, v.x * g.y + v.y * g.x);
        }
    };
    float2 y[RT][CT];
    ft_zero(y);
#pragma unroll
    for (int st = 0; st < kFtStages - 1; ++st) issue(st);
    fetch(0);
    put(0);
    fetch(1);
    for (int st = 0; st < n_st; ++st) {
        ft_wait();
        __syncthreads();  // stage st is complete, and every warp is done with stage st - 1
        issue(st + kFtStages - 1);
        put(st + 1);
        fetch(st + 2);
        const float2 *sg = sm + (st % kFtStages) * C::kBuf;
        ft_stage<false, RT, CT, PG, PZ>(y, sg + pos.row0, sg + kFtKC * PG + pos.col0);
    }

    // epilogue: dX = conj(g_m) Y, partial dg_m = sum_a conj(X_ma) Y_ma
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const int m = M0 + pos.row(r);
        float pr = 0.f, pi = 0.f;
        if (m < n_in) {
            const float2 g = gains ? __ldg(gains + m) : make_float2(1.f, 0.f);
#pragma unroll
            for (int c = 0; c < CT; ++c) {
                const int a = A0 + pos.col(c);
                if (a < K) {
                    const float2 x = __ldg(Xc + (size_t)m * K + a);
                    const float2 v = y[r][c];
                    // conj(x) y
                    pr = fmaf(x.x, v.x, fmaf(x.y, v.y, pr));
                    pi = fmaf(x.x, v.y, fmaf(-x.y, v.x, pi));
                    if (dX) {
                        // conj(g) y
                        dX[((size_t)chan * n_in + m) * K + a] =
                            make_float2(g.x * v.x + g.y * v.y, g.x * v.y - g.y * v.x);
                    }
                }
            }
        }
        if (part) {
            // the 8 lanes of one row; one partial per column half of the tile
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) {
                pr += __shfl_xor_sync(0xffffffffu, pr, off);
                pi += __shfl_xor_sync(0xffffffffu, pi, off);
            }
            if ((threadIdx.x & 7) == 0 && m < n_in)
                part[(((size_t)chan * nA + ab) * 2 + pos.wc) * n_in + m] = make_float2(pr, pi);
        }
    }
}

template <int RT>
corr_status launch_adj(const Handle &h, const float2 *G, const float2 *X, const float2 *gains, float2 *dX,
                       float2 *part, cudaStream_t st) {
    using C = AdjCfg<RT>;
    const int nM = (h.n_in + C::TM - 1) / C::TM, nA = (h.n_spectra + TA - 1) / TA;
    const long long n = (long long)nM * nA * h.n_chan;
    if (n > 0x7fffffffLL) return CORR_EUNSUPPORTED;
    constexpr auto kern = k_adj<RT>;
    if (const corr_status e = allow_smem<kern>((int)C::smem); e != CORR_OK) return e;
    kern<<<(unsigned)n, kFtNth, C::smem, st>>>(G, X, gains, dX, part, h.n_in, h.n_spectra, h.n_base, nM, nA);
    return check_launch("k_adj");
}

// dL/dg = sum of n_part per-row partials, in two fixed-order levels (bit-reproducible):
// level 1 sums the partials of kRedSplit contiguous ranges in FP64, level 2 the ranges.
constexpr int kRedSplit = 64;

__global__ void k_adj_reduce1(const float2 *__restrict__ part, double2 *__restrict__ mid, int n_in, long long n_part) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n_in) return;
    const long long per = (n_part + kRedSplit - 1) / kRedSplit;
    const long long p0 = per * blockIdx.y, p1 = min(n_part, p0 + per);
    double sr = 0.0, si = 0.0;
    // 8 loads in flight, added in order
    long long q = p0;
    for (; q + 8 <= p1; q += 8) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldg(part + (q + u) * n_in + m);
#pragma unroll
        for (int u = 0; u < 8; ++u) sr += v[u].x, si += v[u].y;
    }
    for (; q < p1; ++q) {
        const float2 v = __ldg(part + q * n_in + m);
        sr += v.x;
        si += v.y;
    }
    mid[(size_t)blockIdx.y * n_in + m] = make_double2(sr, si);
}

// 8 lanes per row, each adding every 8th range in order, then the lanes by a butterfly
// (FP64 adds are slow: one thread per row took 8 us, most of it 128 adds in a chain)
__global__ void __launch_bounds__(128) k_adj_reduce2(const double2 *__restrict__ mid, float2 *__restrict__ dg, int n_in) {
    const int m = blockIdx.x * 16 + (threadIdx.x >> 3), u = threadIdx.x & 7;
    double sr = 0.0, si = 0.0;
    if (m < n_in)
#pragma unroll
        for (int s = u; s < kRedSplit; s += 8) {
            const double2 v = mid[(size_t)s * n_in + m];
            sr += v.x;
            si += v.y;
        }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (u == 0 && m < n_in) dg[m] = make_float2((float)sr, (float)si);
}

}  // namespace

size_t backward_workspace_bytes(const Handle &h) {
    const int nA = (h.n_spectra + TA - 1) / TA;
    return align16(sizeof(float2) * (size_t)h.n_chan * nA * 2 * h.n_in) + adj_reduce_scratch_bytes(h.n_in);
}

size_t adj_reduce_scratch_bytes(int n_in) { return sizeof(double2) * (size_t)kRedSplit * n_in; }

corr_status launch_backward_ws(const Handle &h, const float2 *grad_vis, const float2 *chan_in,
                               const float2 *gains, float2 *grad_chan, float2 *grad_gains, float2 *ws,
                               cudaStream_t st) {
    const int nA = (h.n_spectra + TA - 1) / TA;
    if (h.n_chan > 65535) return CORR_EUNSUPPORTED;
    corr_status s;
    {
        StageScope sc(h, CORR_STAGE_ADJ_GEMM, st);
        // rows per tile: the one that pads the inputs least, the largest on a tie
        int rt = 8, rows = (h.n_in + 63) / 64 * 64;
        for (int c : {6, 4}) {
            const int padded = (h.n_in + 8 * c - 1) / (8 * c) * (8 * c);
            // smaller tiles read more operand bytes per product: worth it for 8 % (48 rows)
            // or 25 % (32 rows) less padding
            if (padded * (c == 6 ? 1.08 : 1.25) < rows) rt = c, rows = padded;
        }
        float2 *part = grad_gains ? ws : nullptr;
        s = rt == 8 ? launch_adj<8>(h, grad_vis, chan_in, gains, grad_chan, part, st)
                    : rt == 6 ? launch_adj<6>(h, grad_vis, chan_in, gains, grad_chan, part, st)
                              : launch_adj<4>(h, grad_vis, chan_in, gains, grad_chan, part, st);
    }
    if (s != CORR_OK || !grad_gains) return s;
    const long long n_part = (long long)h.n_chan * nA * 2;
    double2 *scratch = reinterpret_cast<double2 *>(reinterpret_cast<char *>(ws) +
                                                   align16(sizeof(float2) * (size_t)n_part * h.n_in));
    StageScope sc(h, CORR_STAGE_ADJ_REDUCE, st, 2);
    return launch_adj_reduce(ws, scratch, grad_gains, h.n_in, n_part, st);
}

corr_status launch_adj_reduce(const float2 *part, double2 *scratch, float2 *dg, int n_in, long long n_part,
                              cudaStream_t st) {
    const unsigned nb = (unsigned)((n_in + 127) / 128);
    k_adj_reduce1<<<dim3(nb, kRedSplit), 128, 0, st>>>(part, scratch, n_in, n_part);
    corr_status s = check_launch("k_adj_reduce1");
    if (s != CORR_OK) return s;
    k_adj_reduce2<<<(unsigned)((n_in + 15) / 16), 128, 0, st>>>(scratch, dg, n_in);
    return check_launch("k_adj_reduce2");
}

}  // namespace corr
