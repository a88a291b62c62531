// F-engine: per-input channelisation by an unnormalised forward DFT (Eq. 1,
// Section 2), 8-bit re-packing of the spectra and corner turn to channel-major
// order, in one pass.
//
// Each N = T1 x T2 point FFT is computed by a group of T2 threads (twice as many where two
// of them share a column) in two register passes (four-step / Cooley-Tukey split
// n = t + T2 m, k = k1 + T1 k2):
//   pass 1: thread t < T2 holds x[t + T2 m], m < T1, and computes the T1-point DFT
//           over m; the result is multiplied by W_N^(t k1) (twiddle table copied
//           to shared memory per CTA)
//   exchange through shared memory (padded rows, conflict-free)
//   pass 2: thread k1 < T1 holds Y[t][k1], t < T2, and computes the T2-point DFT
//           over t, giving X[k1 + T1 k2].
// Square lengths (16, 64, 256, 1024) take one thread per column and per row. For T2 = 2 T1
// (128, 512, 2048) two threads share each row's T2-point DFT, and for 64 x 64 (4096) each
// column's and each row's (dft_shared): every thread is busy in both passes and holds at
// most 32 values, so that 16 warps fit on an SM (the power pass at 4096 excepted: FCfg::ONE).
// A CTA handles one input and SB consecutive spectra; the outputs are staged in
// shared memory as [channel][spectrum] so that every (channel, input) row segment
// of SB spectra is written to global memory contiguously (the corner turn). Raw
// int8 frames of the plain front end arrive by asynchronous copies into the FFT's
// exchange buffer while the previous frame's pass 2 runs, and enter pass 1 scaled by
// 256 on an offset that the first butterflies cancel (i8_to_f2_scaled).
//
// This header holds the kernel template; the per-feature translation units
// (fengine_plain.cu, fengine_delay.cu, fengine_pfb4.cu, fengine_pfb8.cu,
// fengine_pfb_power.cu) instantiate it, so that the instantiations compile in
// parallel, and fengine.cu holds the host entry points.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cuda_fp16.h>

#include "fft_common.cuh"
#include "internal.h"
#include "requant.cuh"

namespace corr {

// Shape and twiddle table of one F-engine launch.
struct FShape {
    int n_in, n_chan, n_spectra;
    bool i8;
    const float2 *tw;  // [k1][t] table for n_chan = T1 x T2
    int i0 = 0, n_run = -1;  // inputs [i0, i0 + n_run) of the n_in (n_run < 0: all)
    const int *dint = nullptr;     // per-input integer advance (delay compensation), or null
    const float2 *dph = nullptr;   // per-input phase tables [n_in][T1 + T2]: c[k1], then d[k2]
    int n_sm = 152;
};

namespace {


enum Mode { kFloatOut = 0, kRequant = 1, kPower = 2, kRequantPlanar = 3 };

// Front-end features of one F-engine instantiation: none, delay compensation (an integer
// advance of the frames and / or the per-channel fractional phase), or the polyphase
// filter bank formed in shared memory (with or without delays).
enum Feat { kPlain = 0, kDelay = 1, kPfb = 2 };

template <int N, bool I8, int MODE, int FEAT = kPlain>
struct FCfg {
    static constexpr int T2 = fengine_t2(N);  // pass-1 threads = pass-2 DFT length
    static constexpr int T1 = N / T2;         // pass-1 DFT length = pass-2 threads
    static_assert(T2 > 0 && T1 * T2 == N && T1 <= T2 && T2 <= 64, "unsupported F-engine length");
    // The power pass at N = 4096 without delays has no staging rows, and 64 values per thread
    // fit its registers: one thread per DFT, in CTAs of two FFTs, two to an SM, beats shared
    // DFTs in CTAs of 256 threads (int8, us: 128 inputs x 1024 spectra 1268 -> 1002, 16 x 256
    // 65.7 -> 53.2, 16 x 128 41.1 -> 34.1; FP32 16 x 128 45.2 -> 36.0; with delays 1471 -> 1873:
    // those share).
    static constexpr bool ONE = N == 4096 && MODE == kPower && FEAT == kPlain;
    static constexpr int H1 = T1 == 64 && !ONE ? 2 : 1;               // threads per column in pass 1
    static constexpr int H2 = T2 == 2 * T1 || (T1 == 64 && !ONE) ? 2 : 1;  // threads per row in pass 2
    static constexpr int TG = T2 * H1;        // threads per FFT group
    static_assert(TG == T1 * H2, "every thread takes part in both passes");
    static constexpr bool RQ = MODE == kRequant || MODE == kRequantPlanar;
    // long re-packed transforms read the twiddles through L1 instead of a shared-memory copy,
    // so that two CTAs fit on an SM at N = 2048 (one's copy-out beside the other's FFTs: 370
    // -> 324 us below) and twice the staging rows at N = 4096
    static constexpr bool TWG = N >= 2048 && RQ && FEAT != kPfb;
    // threads per CTA: 256, or 512 where the shared memory leaves room for one CTA only
    static constexpr int NT = (N >= 2048 && RQ && !TWG) || (N == 4096 && RQ) ? 512 : ONE ? 128 : 256;
    static constexpr int G = NT / TG;         // FFTs in flight per CTA
    // Exchange buffer of one FFT: T1 rows of EXS floats; row k1 receives Y[0..T2-1][k1]
    // (one column per writing thread) and is read back as float4. EXS and the per-FFT
    // stride GS keep both the scalar writes and the float4 reads free of bank conflicts:
    // 4 EXS / 4 odd per quarter warp, and GS = TG (mod 32) so that the FFTs sharing a
    // warp write to disjoint banks.
    static constexpr int EXS = T2 == 4 ? 8 : T2 + 4;
    // The filter bank's frames (complex FP32) are formed in the same per-FFT slots, read
    // by pass 1 before the exchange overwrites them.
    static constexpr int GS = (FEAT == kPfb ? 2 * N : T1 * EXS) + (TG >= 32 ? 0 : TG);
    static_assert(GS >= T1 * EXS, "the exchange fits into a slot");
    // spectra per CTA: the re-packing modes take 32 up to N = 1024 (64-byte row
    // segments of the planar FP16 planes, 2 CTAs/SM at N = 1024), 16 for longer
    // transforms: whole 32-byte sectors per row (with 8 at N = 4096, whose staging rows
    // then leave room for two CTAs, the planar layout took 674 us against 489 for 64
    // inputs x 512 spectra)
    // (the FP32 and power modes take at least the G spectra that are in flight at once: with
    // 8 spectra per CTA half the threads of N = 256 had no FFT, 15.4 -> 11.5 us for 16
    // inputs x 1024 spectra)
    static constexpr int SB = MODE == kFloatOut ? (N <= 1024 ? (G > 8 ? G : 8) : 8192 / N)
                                                : (RQ ? (FEAT == kPfb && N == 1024 ? 16 : N <= 1024 ? 32 : (N == 4096 && FEAT != kPfb) ? 16 : 32768 / N)
                                                      : (G > 16 ? G : 16));
    // The long transforms may take fewer spectra per CTA than SB (see launch_one_); for the
    // others the variable loop bound cost more (1 to 4 %) than a fuller chip gains.
    static constexpr bool VARSB = RQ && N >= 2048;
    // The power pass runs over many blocks of SB spectra per CTA (see launch_one_): its
    // channel sums stay in shared memory as FP64. A thread adds PQ of its spectra in FP32 and
    // the FW FFTs of a warp join in FP32, 16 spectra at most and 8 in a row, what an FP32 sum
    // in order over 16 spectra may lose; the warps' sums join without a rounding.
    // (Modelled with exponentially distributed powers, rms error against that sum's: 0.66 at
    // N = 16, 0.68 at 64, 0.75 up to 256, 0.73 up to 1024, 0.83 above.)
    static constexpr bool POW = MODE == kPower;
    static constexpr int FW = TG < 32 ? 32 / TG : 1;  // FFTs per warp
    static constexpr int PQ = FW > 2 ? 16 / FW : 8;
    // blocks of SB spectra per CTA at most, and whether they join more than once
    static constexpr int POWB = N * SB < 1 << 16 ? (1 << 16) / (N * SB) : 1;
    static constexpr bool PSUM = POW && POWB * SB > PQ * G;
    // staging row stride in 32-bit words. The re-packing modes stage one 16-bit code
    // pair per (channel k, spectrum s): a row of SB / 2 words whose word index is
    // XOR-swizzled with (k >> SW) & (ROWW - 1), SW = log2(32 / ROWW), so that the
    // 16-bit writes of one warp (32 consecutive rows) and the 4-word row reads of the
    // copy-out are free of bank conflicts. The FP32 mode stages float2 values in
    // padded rows.
    static constexpr int ROWW = RQ ? SB / 2 : (MODE == kFloatOut ? 2 * SB + 2 : 0);
    static constexpr int SW = RQ ? ilog2(32 / ROWW) : 0;
    static_assert(!RQ || (ROWW >= 4 && ROWW <= 16), "swizzle assumes 4..16-word rows");
    static constexpr size_t ex_bytes = sizeof(float) * (size_t)G * GS;
    static constexpr size_t pw_bytes = PSUM ? sizeof(double) * N : 0;  // FP64 channel sums
    static constexpr size_t tw_bytes = TWG ? 0 : sizeof(float2) * (size_t)N;  // twiddle table copy
    static constexpr size_t dl_bytes = sizeof(float2) * 64;         // delay phases d[k2] (T2 <= 64)
    static constexpr size_t st_bytes = sizeof(uint32_t) * (size_t)N * ROWW;
    static constexpr size_t smem = ex_bytes + pw_bytes + tw_bytes + dl_bytes + st_bytes;
    static_assert(smem <= 232448, "shared memory");
};

// complex int8 sample (16 bits: re in the low byte) -> float2, exactly:
// (0x4B400000 | (x + 128)) is the float 12582912 + x + 128.
__device__ __forceinline__ float2 i8_to_f2(uint32_t w) {
    const uint32_t u = w ^ 0x8080u;
    return f2_sub(make_float2(__uint_as_float(__byte_perm(u, 0x4B400000u, 0x7650)),
                              __uint_as_float(__byte_perm(u, 0x4B400000u, 0x7651))),
                  make_float2(kMagic + 128.0f, kMagic + 128.0f));
}

// complex int8 sample x (16 bits: re in the low byte) -> float2 (c + 256 re, c + 256 im)
// with the constant c = 2^23 + 2^15, exactly: the float with bits 0x4B00 (x + 128) 00
// is 2^23 + 256 (x + 128). The offset needs no subtraction here: the first radix-2
// stage's differences cancel it exactly, and along the all-sums path (DFT bin 0 of
// pass 1) every partial sum j c + 256 s stays exact (a multiple of 256 below 2^29,
// where the spacing of floats is at most 32), so that bin is corrected once per FFT
// (kOffsetFix). The factor 256 leaves every rounding unchanged (a power of two); it
// is divided out by the inter-pass twiddles, stored divided by 256.
__device__ __forceinline__ float2 i8_to_f2_scaled(uint32_t w) {
    const uint32_t u = w ^ 0x8080u;
    return make_float2(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7404)),
                       __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7414)));
}
constexpr float kI8Scale = 256.0f;
constexpr float kI8OffsetOverScale = 32896.0f;  // (2^23 + 2^15) / 256

// pass-1 bin 0 of T scaled samples (T c + 256 sum x, exact below 2^31: every partial
// sum is a multiple of 256) -> sum x, exactly
template <int T>
__device__ __forceinline__ float2 kOffsetFix(float2 v) {
    constexpr float k = -(float)T * kI8OffsetOverScale;
    return f2_fma(v, make_float2(1.0f / kI8Scale, 1.0f / kI8Scale), make_float2(k, k));
}

// 16-byte global -> shared copy that bypasses the registers (cp.async, L2 only)
__device__ __forceinline__ void cp_async16(void *sdst, const void *gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(sdst)),
                 "l"(gsrc)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// a + b rounded; err gains what the rounding left out (Knuth's two-sum, exact)
__device__ __forceinline__ float add_err(float a, float b, float &err) {
    const float s = a + b, bb = s - a;
    err += (a - (s - bb)) + (b - bb);
    return s;
}

// Polyphase filter-bank parameters of one launch (see pfb_frames).
struct PfbArgs {
    const float *win = nullptr;  // [taps][N]
    int taps = 0;
};

// Where sample n of a filter-bank frame lies in its slot: the 16-byte units of two
// samples are exchanged in pairs by bit 3 of the unit, so that lanes storing units
// 2 l, 2 l + 1 of consecutive quads meet every bank once (and pass 1's reads do too).
__host__ __device__ constexpr int pfb_at(int n) { return n ^ (((n >> 4) & 1) << 1); }

// byte b of u (an offset-binary code x + 128) as the float 12582912 + x + 128
template <int B>
__device__ __forceinline__ float ob_float(uint32_t u) {
    return __uint_as_float(__byte_perm(u, 0x4B400000u, 0x7650 + B));
}

// The FIR stage of the fused filter bank: frames s0 .. s0 + G - 1 of this CTA into the
// FFT slots, y_a[n] = sum_{p < taps} h[p][n] s'[(a + p) N + n], taps <= P, int8 voltages.
// A thread takes four consecutive positions of FR consecutive spectra: each raw quad is
// loaded (8 bytes) and converted once for all the spectra it enters, the window once.
// The sums run over p in order with one FMA per tap, as k_pfb_fir's, whose frames these
// equal bit for bit. At N = 1024 with 4 taps it adds 620 warp instructions per frame to the
// FFT's 1540 and 96 shared-memory wavefronts to its 290; what bounds the whole is latency:
// issue 50 % active, the raw loads of a round exposed between two CTA-wide barriers.
template <int N, int P, int G, int GS, int NT>
__device__ __forceinline__ void pfb_frames(float *slots, const char2 *__restrict__ in, const PfbArgs &f, long long D,
                                           long long n_rec, int a_first) {
    // spectra per thread and round (a longer window leaves registers for fewer)
    constexpr int FR = N >= 1024 ? (P <= 4 ? G : G / 2) : (G * N / 1024 > 0 ? G * N / 1024 : 1);
    constexpr int NQ = N / 4, UNITS = NQ * (G / FR);
    static_assert(UNITS % NT == 0, "whole rounds");
    const bool vec = (D & 3) == 0;
    auto quad = [&](int b, int n) {  // samples n .. n + 3 of frame b of the advanced stream
        const long long t = (long long)b * N + n + D;
        uint2 w = make_uint2(0u, 0u);
        if (t >= n_rec || t + 4 <= 0) return w;
        if (vec) {  // n_rec and t are multiples of 4: wholly inside
            w = __ldg(reinterpret_cast<const uint2 *>(in + t));
        } else {
            const unsigned short *s = reinterpret_cast<const unsigned short *>(in) + t;
            uint32_t e[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) e[x] = t + x >= 0 && t + x < n_rec ? (uint32_t)__ldg(s + x) : 0u;
            w = make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
        }
        return w;
    };
#pragma unroll 1
    for (int u = threadIdx.x; u < UNITS; u += NT) {
        const int n = 4 * (u % NQ), g0 = (u / NQ) * FR, a0 = a_first + g0;
        // every load of the round in flight together
        float4 h[P];
#pragma unroll
        for (int p = 0; p < P; ++p)
            h[p] = p < f.taps ? __ldg(reinterpret_cast<const float4 *>(f.win + (size_t)p * N + n)) : make_float4(0.f, 0.f, 0.f, 0.f);
        uint2 raw[FR + P - 1];
        const long long t0 = (long long)a0 * N + n + D;
        if (vec && t0 >= 0 && t0 + (long long)(FR + P - 2) * N < n_rec) {
            const char2 *src = in + t0;
#pragma unroll
            for (int q = 0; q < FR + P - 1; ++q) raw[q] = __ldg(reinterpret_cast<const uint2 *>(src + q * N));
        } else {
#pragma unroll
            for (int q = 0; q < FR + P - 1; ++q) raw[q] = quad(a0 + q, n);
        }
        float2 y[FR][4];
#pragma unroll
        for (int r = 0; r < FR; ++r)
#pragma unroll
            for (int x = 0; x < 4; ++x) y[r][x] = make_float2(0.f, 0.f);
        // raw quad q enters spectra r = q - p: converted once, p ascending for every r
#pragma unroll
        for (int q = 0; q < FR + P - 1; ++q) {
            const uint32_t a = raw[q].x ^ 0x80808080u, b = raw[q].y ^ 0x80808080u;
            const float2 off = make_float2(kMagic + 128.0f, kMagic + 128.0f);
            const float2 x0 = f2_sub(make_float2(ob_float<0>(a), ob_float<1>(a)), off);
            const float2 x1 = f2_sub(make_float2(ob_float<2>(a), ob_float<3>(a)), off);
            const float2 x2 = f2_sub(make_float2(ob_float<0>(b), ob_float<1>(b)), off);
            const float2 x3 = f2_sub(make_float2(ob_float<2>(b), ob_float<3>(b)), off);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const int r = q - p;
                if (r < 0 || r >= FR) continue;
                y[r][0] = f2_fma(make_float2(h[p].x, h[p].x), x0, y[r][0]);
                y[r][1] = f2_fma(make_float2(h[p].y, h[p].y), x1, y[r][1]);
                y[r][2] = f2_fma(make_float2(h[p].z, h[p].z), x2, y[r][2]);
                y[r][3] = f2_fma(make_float2(h[p].w, h[p].w), x3, y[r][3]);
            }
        }
#pragma unroll
        for (int r = 0; r < FR; ++r) {
            float2 *slot = reinterpret_cast<float2 *>(slots + (size_t)(g0 + r) * GS);
            *reinterpret_cast<float4 *>(slot + pfb_at(n)) = make_float4(y[r][0].x, y[r][0].y, y[r][1].x, y[r][1].y);
            *reinterpret_cast<float4 *>(slot + pfb_at(n + 2)) = make_float4(y[r][2].x, y[r][2].y, y[r][3].x, y[r][3].y);
        }
    }
}

// One L-point DFT shared by two threads of a warp, the lanes of which differ in bit HB:
// thread h holds x[q h + i] (lo[i]) and x[L/2 + q h + i] (hi[i]), i < q = L/4, and returns in
// v[bitrev(k')] the outputs k = 2 k' + h. The first radix-2 stage pairs what a thread holds;
// thread 0 then goes on with the sums and thread 1 with the differences, of which each gets
// the other half from its partner (in the second stage the two halves meet: the thread that
// holds the upper ones subtracts the wrong way round, put right by an exact factor -1). The
// butterflies, factors and roundings are fft_dif<L>'s: the results are the same. 64 inputs,
// int8 layout (us): N = 2048 x 1024 spectra 555 -> 324 (the T2-point DFTs ran on one of two
// warps, at 212 registers and 8 warps per SM), N = 4096 x 512 527 -> 445 (8 -> 16 warps), N =
// 512 x 4096 346 -> 258 and N = 128 x 16384 338 -> 267 (half of each warp idle).
template <int L, int HB, bool PACK>
__device__ __forceinline__ void dft_shared(const float2 (&lo)[L / 4], const float2 (&hi)[L / 4], int h,
                                           float2 (&v)[L / 2]) {
    constexpr int q = L / 4;
    const float2 sgn = h ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
    sfor<0, q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        const float2 s = f2_add(lo[i], hi[i]);
        float2 d = f2_sub(lo[i], hi[i]);
        if constexpr (i == 0) {
            d = h ? make_float2(d.y, -d.x) : d;  // W^q = -j, W^0 = 1
        } else {
            // W_L^(q h + i), as mul_w multiplies by it
            constexpr float c0 = (float)cos2pi(i, L), s0 = (float)sin2pi(i, L);
            constexpr float c1 = (float)cos2pi(q + i, L), s1 = (float)sin2pi(q + i, L);
            const float c = h ? c1 : c0, sn = h ? s1 : s0;
            d = make_float2(fmaf(d.x, c, d.y * sn), fmaf(d.y, c, -(d.x * sn)));
        }
        const float2 keep = h ? d : s, give = h ? s : d;
        const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, HB), __shfl_xor_sync(0xffffffffu, give.y, HB));
        v[i] = f2_add(keep, got);
        v[i + q] = mul_w<i, L / 2, PACK>(f2_mul(f2_sub(keep, got), sgn));
    });
    fft_dif<L / 2, L / 2, 1, PACK>(v);
}

// CTAs per SM the register allocation aims at. The shorter transforms hold 8 or 16 values per
// thread and wait on loads and barriers, so more warps in flight pay for as long as nothing
// spills; the delay form, which converts its samples with synchronous loads, gains most.
// 128 inputs, int8 layout, us (3 CTAs, or 2 at N = 512, before): delays N = 512 x 8192 spectra
// 1252 -> 1101 with 4, N = 256 x 16384 1079 -> 1002 with 4, 951 with 5 and 1096 with 6, N =
// 128 x 16384 661 -> 566 with 5, 547 with 6, N = 64 x 32768 597 -> 554 with 5, 537 with 6;
// no delays N = 256 848 -> 842 with 4 (planar 952 -> 923), 849 with 5, N = 128 528 -> 503
// with 5 and 504 with 6, N = 64 476 -> 453 with 6. FP32 voltages gain from 6 up to N = 128
// (334 -> 313 for 8192 spectra) and nothing above. The filter bank keeps its FIR quads in
// registers: more CTAs help at N = 64 only (4 taps 729 -> 669 with 6; 8 taps 935 -> 823 with
// 4, 983 with 5). The power pass has no staging rows: N = 1024 with delays 1604 -> 1104 with 2.
template <int N, bool I8, int MODE, int FEAT, int P>
constexpr int fengine_ctas() {
    if (N >= 2048) return FCfg<N, I8, MODE, FEAT>::NT == 512 ? 1 : 2;
    if (MODE == kPower && FEAT != kPfb) return N == 1024 ? 2 : N >= 512 ? 3 : N == 256 ? 4 : 5;
    if (N >= 1024) return 2;
    if (FEAT == kPfb) return N >= 512 ? 2 : N != 64 ? 3 : P <= 4 ? 6 : 4;
    if (N == 512) return I8 && FEAT == kDelay ? 4 : 2;
    if (N == 256) return !I8 ? 3 : FEAT == kDelay ? 5 : 4;
    if (N == 128) return I8 && FEAT == kPlain ? 5 : 6;
    return N == 64 ? 6 : 3;
}

template <int N, bool I8, int MODE, int FEAT, int P = 0>
__global__ void __launch_bounds__(FCfg<N, I8, MODE, FEAT>::NT, fengine_ctas<N, I8, MODE, FEAT, P>()) k_fengine(const void *__restrict__ volt,
                                                      const float *__restrict__ scale,
                                                      void *__restrict__ out,
                                                      double *__restrict__ power, int n_in, int K,
                                                      const float2 *__restrict__ tw_glob, int i0, int vec_out,
                                                      const int *__restrict__ dint,
                                                      const float2 *__restrict__ dph, int async_raw,
                                                      const PfbArgs pfb, int sb_run) {
    using C = FCfg<N, I8, MODE, FEAT>;
    constexpr int T1 = C::T1, T2 = C::T2, TG = C::TG, G = C::G, EXS = C::EXS, SB = C::SB, ROWW = C::ROWW;
    constexpr int NT = C::NT, H1 = C::H1, H2 = C::H2;
    constexpr int R1 = T1 / H1, R2 = T2 / H2;  // values per thread in each pass
    constexpr int TV = R1 > R2 ? R1 : R2;
    constexpr bool PACK = N == 512 || N == 1024 || (N == 4096 && FEAT != kDelay);  // packed factors pay (see mul_w)
    constexpr int HB = T1 < 16 ? T1 : 16;      // lane bit between two threads that share a DFT
    // square 32-point passes read the exchange into float arrays and do pass 2's
    // first stage in scalar arithmetic (no register moves into the (re, im) pairs); the
    // smaller lengths keep the in-place reads, which fit their register budgets
    constexpr bool kScalarStage = T1 == T2 && T2 >= 32;
    constexpr bool PFB = FEAT == kPfb;
    constexpr bool DLY = FEAT != kPlain;  // delay code compiled in
    // int8 samples enter the plain FFT scaled by 256 on an offset (i8_to_f2_scaled); the
    // delay instantiation converts them exactly (measured faster there)
    constexpr bool SCALED = I8 && !DLY;
    // the integer advance and the phase are separate: the filter-bank path applies the
    // advance in its FIR pass and only the phase here
    const bool has_shift = DLY && dint != nullptr, has_dly = DLY && dph != nullptr;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *ex = reinterpret_cast<float *>(smem_raw);                                 // [G][T1][EXS]
    double *psum = reinterpret_cast<double *>(smem_raw + C::ex_bytes);               // [N] (power)
    float2 *tws = reinterpret_cast<float2 *>(smem_raw + C::ex_bytes + C::pw_bytes);  // [k1][t] twiddles
    float2 *dsm = reinterpret_cast<float2 *>(smem_raw + C::ex_bytes + C::pw_bytes + C::tw_bytes);  // [k2] phases
    uint32_t *stg = reinterpret_cast<uint32_t *>(smem_raw + C::ex_bytes + C::pw_bytes + C::tw_bytes +
                                                 C::dl_bytes);  // staging
    // 16-bit slot of code (k, s) in the swizzled staging rows
    auto slot = [](int k, int s) {
        return k * (2 * ROWW) + 2 * ((s >> 1) ^ ((k >> C::SW) & (ROWW - 1))) + (s & 1);
    };
    // the threads of one FFT group meet: a warp (or part of one), or the whole CTA
    auto group_sync = [] {
        if constexpr (TG <= 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / TG), "n"(TG) : "memory");  // (warps of this group)
    };

    const int i = i0 + blockIdx.y;
    const int sb = C::VARSB || C::POW ? sb_run : SB;  // spectra per CTA
    const int a0 = blockIdx.x * sb;
    // Raw int8 frames without delays are copied asynchronously into the FFT's exchange
    // buffer (free between exchanges): the copy for the next frame is issued after the
    // current frame's exchange and lands while its pass 2 and re-packing run. Each of
    // the TG threads moves N / (8 TG) 16-byte pieces of the 2 N-byte frame.
    constexpr bool kAsync = I8 && !DLY && N / (8 * TG) >= 1;
    static_assert(!kAsync || sizeof(float) * C::GS >= 2 * N, "exchange buffer holds one raw frame");
    const bool use_async = kAsync && async_raw;
    // copy of frame s_ of this CTA into the exchange buffer of FFT slot s_ % G
    auto issue_raw = [&](int s_) {
        const int a_ = a0 + s_, t_ = threadIdx.x % TG;
        if (s_ < sb && a_ < K) {
            const char *src = reinterpret_cast<const char *>(volt) + ((size_t)i * K + a_) * (size_t)N * 2;
            char *dst = reinterpret_cast<char *>(ex + (size_t)(s_ % G) * C::GS);
#pragma unroll
            for (int c = 0; c < N / (8 * TG); ++c) cp_async16(dst + (c * TG + t_) * 16, src + (c * TG + t_) * 16);
        }
        cp_async_commit();
    };
    if (use_async) issue_raw(threadIdx.x / TG);
    // Delay compensation: the frames are read D samples later in input i's stream
    // (samples outside the record are zero) and channel k = k1 + T1 k2 is multiplied by
    // c[k1] d[k2] = exp(+j 2 pi k f / N): c is folded into the inter-pass twiddles
    // (it is common to thread k1's pass-2 DFT), d applied to the outputs.
    const long long n_rec = (long long)K * N;  // samples per input
    const int D = has_shift ? __ldg(dint + i) : 0;
    // Warm L2 with the raw block of spectra [a_lo, a_hi) of input i (one contiguous range):
    // the loads of the later spectra then hit L2 instead of HBM.
    auto warm = [&](long long a_lo, long long a_hi) {
        constexpr int BPS = I8 ? 2 : 8;  // bytes per complex sample
        const long long lo = max(0LL, a_lo * N + D);
        const long long hi = min(n_rec, min((long long)K, a_hi) * N + D);
        if (hi > lo) {
            const char *blk = reinterpret_cast<const char *>(volt) + ((size_t)i * n_rec + lo) * BPS;
            const int lines = (int)(((hi - lo) * BPS + 127) / 128);
            for (int l = threadIdx.x; l < lines; l += NT)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(blk + (size_t)l * 128));
        }
    };
    warm(a0, (long long)a0 + min(SB, sb));
    // per-CTA copy of the twiddle table (shared-memory loads in the FFT loop; measured
    // faster than L1 lookups, while the channel scales are faster from L1)
    const bool tw_async = PFB && !has_dly;  // as it stands: in flight while the first frames form
    if (tw_async) {
        for (int m = 2 * threadIdx.x; m < N; m += 2 * NT) cp_async16(tws + m, tw_glob + m);
        cp_async_commit();
    }
    if (C::TWG && has_dly && threadIdx.x < T2) dsm[threadIdx.x] = __ldg(dph + (size_t)i * (T1 + T2) + T1 + threadIdx.x);
    for (int m = threadIdx.x; m < N && !tw_async && !C::TWG; m += NT) {
        float2 w = __ldg(tw_glob + m);
        if (DLY && has_dly) {
            w = cmul(w, __ldg(dph + (size_t)i * (T1 + T2) + m / T2));  // table [k1][t]: c[k1]
            if (m < T2) dsm[m] = __ldg(dph + (size_t)i * (T1 + T2) + T1 + m);
        }
        if constexpr (SCALED) w = make_float2(w.x * (1.0f / kI8Scale), w.y * (1.0f / kI8Scale));
        tws[m] = w;
    }
    if constexpr (!PFB) __syncthreads();

    const int g = threadIdx.x / TG;
    const int t = threadIdx.x % TG;
    // the column this thread takes in pass 1 and the row in pass 2, and which half of a
    // shared DFT (the threads HB lanes apart)
    const int half = (t / HB) & 1, pair = (t % HB) + (t / (2 * HB)) * HB;
    const int col = H1 == 2 ? pair : t, row = H2 == 2 ? pair : t;
    const int h1 = H1 == 2 ? half : 0, h2 = H2 == 2 ? half : 0;
    float *exg = ex + (size_t)g * C::GS;
    const float4 *exrow = reinterpret_cast<const float4 *>(exg + row * EXS);
    float pw[R2];
    if constexpr (MODE == kPower) {
#pragma unroll
        for (int q = 0; q < R2; ++q) pw[q] = 0.0f;
    }

    for (int s0 = 0; s0 < (C::POW ? sb : SB); s0 += G) {
        if (C::VARSB && s0 >= sb) break;  // (sb is a multiple of G)
        if (C::POW && s0 % SB == 0) warm((long long)a0 + s0 + SB, a0 + min(s0 + 2LL * SB, (long long)sb));
        const bool join = C::POW && ((s0 / G) % C::PQ == C::PQ - 1 || s0 + G >= sb);  // partial sums meet below
        const int s = s0 + g;
        const int a = a0 + s;
        const bool valid = (s < (C::POW ? sb : SB)) && (a < K);
        float2 v[TV];
        // ---- pass 1: column col takes x[col + T2 m]: value m of the R1 this thread holds is
        // sample mm(m) of the column
        // twiddle W_N^(col k1) (with the delay phase c[k1]; / 256 for scaled samples)
        auto tw_at = [&](int k1) {
            if constexpr (!C::TWG) return tws[k1 * T2 + col];
            float2 w = __ldg(tw_glob + k1 * T2 + col);
            if (DLY && has_dly) w = cmul(w, __ldg(dph + (size_t)i * (T1 + T2) + k1));
            if constexpr (SCALED) w = make_float2(w.x * (1.0f / kI8Scale), w.y * (1.0f / kI8Scale));
            return w;
        };
        auto mm = [&](int m) { return H1 == 1 ? m : (m < R1 / 2 ? 0 : T1 / 2 - R1 / 2) + (T1 / 4) * h1 + m; };
        // sample offset of this frame in input i's stream (shifted by D with delays)
        const long long off = (long long)(valid ? a : 0) * N + D;
        const long long base = (long long)i * n_rec + off + col;
        // with delays, frames that reach outside the record take the checked loads
        const bool inside = !DLY || (off >= 0 && off + N <= n_rec);
        if constexpr (PFB) {
            if (s0 > 0) __syncthreads();  // every FFT has left its slot
            pfb_frames<N, P, G, C::GS, NT>(ex, reinterpret_cast<const char2 *>(volt) + (size_t)i * n_rec, pfb, D, n_rec,
                                       a0 + s0);
            cp_async_wait_all();
            __syncthreads();
            const float2 *frame = reinterpret_cast<const float2 *>(exg);
#pragma unroll
            for (int m = 0; m < R1; ++m) v[m] = valid ? frame[pfb_at(col + T2 * mm(m))] : make_float2(0.f, 0.f);
            group_sync();  // read before the exchange overwrites the slot
        } else if constexpr (I8) {
            const unsigned short *src = reinterpret_cast<const unsigned short *>(volt) + base;
            if (use_async) {
                cp_async_wait_all();
                group_sync();  // every thread's pieces of the frame have landed
                const unsigned short *raw = reinterpret_cast<const unsigned short *>(exg) + col;
#pragma unroll
                for (int m = 0; m < R1; ++m) v[m] = i8_to_f2_scaled(valid ? (uint32_t)raw[T2 * mm(m)] : 0u);
                group_sync();  // read before the exchange overwrites the buffer
            } else if (inside) {
#pragma unroll
                for (int m = 0; m < R1; ++m) {
                    const uint32_t w = valid ? (uint32_t)__ldg(src + (size_t)T2 * mm(m)) : 0u;
                    v[m] = SCALED ? i8_to_f2_scaled(w) : i8_to_f2(w);
                }
            } else {
#pragma unroll
                for (int m = 0; m < R1; ++m) {
                    const long long n = off + col + T2 * mm(m);
                    const uint32_t w = (valid && n >= 0 && n < n_rec) ? (uint32_t)__ldg(src + (long long)T2 * mm(m)) : 0u;
                    v[m] = SCALED ? i8_to_f2_scaled(w) : i8_to_f2(w);
                }
            }
        } else {
            const float2 *src = reinterpret_cast<const float2 *>(volt) + base;
            if (inside) {
#pragma unroll
                for (int m = 0; m < R1; ++m) v[m] = valid ? __ldg(src + (size_t)T2 * mm(m)) : make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int m = 0; m < R1; ++m) {
                    const long long n = off + col + T2 * mm(m);
                    v[m] = (valid && n >= 0 && n < n_rec) ? __ldg(src + (long long)T2 * mm(m)) : make_float2(0.f, 0.f);
                }
            }
        }
        // v[bitrev(k')] = Y[col][k1], k1 = H1 k' + h1 (x 256, bin 0 offset, for int8 input)
        if constexpr (H1 == 1) {
            fft_dif<T1, TV, 0, PACK>(v);
        } else {
            float2 lo[R1 / 2], hi[R1 / 2];
#pragma unroll
            for (int m = 0; m < R1 / 2; ++m) lo[m] = v[m], hi[m] = v[m + R1 / 2];
            dft_shared<T1, HB, PACK>(lo, hi, h1, v);
        }
        if constexpr (SCALED) v[0] = h1 == 0 ? kOffsetFix<T1>(v[0]) : v[0];
        sfor<0, R1>([&](auto K1) {
            constexpr int k1 = decltype(K1)::value;
            // twiddle W_N^(col k1), table laid out [k1][col]
            float2 &x = v[bitrev(k1, ilog2(R1))];
            if constexpr (H1 == 1) {
                if constexpr (k1 != 0) x = cmul(x, tw_at(k1));
            } else {
                const float2 y = cmul(x, tw_at(2 * k1 + h1));
                x = k1 == 0 && h1 == 0 ? x : y;
            }
        });
        // ---- exchange (Re, then Im; the other half stays in place) and pass 2: this thread
        // now takes Y[tt][row]
        sfor<0, R1>([&](auto K1) {
            constexpr int k1 = decltype(K1)::value;
            exg[(H1 * k1 + h1) * EXS + col] = v[bitrev(k1, ilog2(R1))].x;
        });
        group_sync();
        if constexpr (H2 == 2) {
            // tt = q h2 + i and T2 / 2 + q h2 + i, i < q
            constexpr int q = T2 / 4;
            float2 lo[q], hi[q];
#pragma unroll
            for (int j = 0; j < q / 4; ++j) {
                const float4 a = exrow[q / 4 * h2 + j], b = exrow[T2 / 8 + q / 4 * h2 + j];
                lo[4 * j].x = a.x, lo[4 * j + 1].x = a.y, lo[4 * j + 2].x = a.z, lo[4 * j + 3].x = a.w;
                hi[4 * j].x = b.x, hi[4 * j + 1].x = b.y, hi[4 * j + 2].x = b.z, hi[4 * j + 3].x = b.w;
            }
            group_sync();
            sfor<0, R1>([&](auto K1) {
                constexpr int k1 = decltype(K1)::value;
                exg[(H1 * k1 + h1) * EXS + col] = v[bitrev(k1, ilog2(R1))].y;
            });
            group_sync();
#pragma unroll
            for (int j = 0; j < q / 4; ++j) {
                const float4 a = exrow[q / 4 * h2 + j], b = exrow[T2 / 8 + q / 4 * h2 + j];
                lo[4 * j].y = a.x, lo[4 * j + 1].y = a.y, lo[4 * j + 2].y = a.z, lo[4 * j + 3].y = a.w;
                hi[4 * j].y = b.x, hi[4 * j + 1].y = b.y, hi[4 * j + 2].y = b.z, hi[4 * j + 3].y = b.w;
            }
            group_sync();
            if (use_async && s0 + G < sb && !join) issue_raw(s0 + G + g);  // next frame into the free buffer
            dft_shared<T2, HB, PACK>(lo, hi, h2, v);  // v[bitrev(k')] = X[row + T1 k2], k2 = 2 k' + h2
        } else if constexpr (kScalarStage) {
            // the rows are read into plain float arrays (a 16-byte load fills four
            // consecutive registers, which the (re, im) register pairs of v cannot offer)
            float rin[T2], iin[T2];
            {
#pragma unroll
                for (int j = 0; j < T2 / 4; ++j) {
                    const float4 r = exrow[j];
                    rin[4 * j] = r.x, rin[4 * j + 1] = r.y, rin[4 * j + 2] = r.z, rin[4 * j + 3] = r.w;
                }
            }
            group_sync();
            sfor<0, T1>([&](auto K1) {
                constexpr int k1 = decltype(K1)::value;
                exg[k1 * EXS + t] = v[bitrev(k1, ilog2(T1))].y;
            });
            group_sync();
            {
#pragma unroll
                for (int j = 0; j < T2 / 4; ++j) {
                    const float4 r = exrow[j];
                    iin[4 * j] = r.x, iin[4 * j + 1] = r.y, iin[4 * j + 2] = r.z, iin[4 * j + 3] = r.w;
                }
            }
            group_sync();
            if (use_async && s0 + G < sb && !join) issue_raw(s0 + G + g);  // next frame into the free buffer
            // pass 2: its first radix-2 stage in scalar arithmetic, from the float arrays
            // into the (re, im) pairs, then the remaining stages on the pairs
            sfor<0, T2 / 2>([&](auto J) {
                constexpr int a = decltype(J)::value, b = a + T2 / 2;
                const float ar = rin[a], ai = iin[a], br = rin[b], bi = iin[b];
                v[a] = make_float2(ar + br, ai + bi);
                if constexpr (4 * a == T2)
                    v[b] = make_float2(ai - bi, br - ar);  // (x - y)(-j)
                else
                    v[b] = mul_w<a, T2, PACK>(make_float2(ar - br, ai - bi));
            });
            fft_dif<T2, TV, 1, PACK>(v);  // v[bitrev(k2)] = X[t + T1 k2]
        } else {
            {
#pragma unroll
                for (int j = 0; j < T2 / 4; ++j) {
                    const float4 r = exrow[j];
                    v[4 * j].x = r.x, v[4 * j + 1].x = r.y, v[4 * j + 2].x = r.z, v[4 * j + 3].x = r.w;
                }
            }
            group_sync();
            sfor<0, T1>([&](auto K1) {
                constexpr int k1 = decltype(K1)::value;
                exg[k1 * EXS + t] = v[bitrev(k1, ilog2(T1))].y;
            });
            group_sync();
            {
#pragma unroll
                for (int j = 0; j < T2 / 4; ++j) {
                    const float4 r = exrow[j];
                    v[4 * j].y = r.x, v[4 * j + 1].y = r.y, v[4 * j + 2].y = r.z, v[4 * j + 3].y = r.w;
                }
            }
            group_sync();
            if (use_async && s0 + G < sb && !join) issue_raw(s0 + G + g);  // next frame into the free buffer
            fft_dif<T2, TV, 0, PACK>(v);  // v[bitrev(k2)] = X[t + T1 k2]
        }
        if (PFB && has_dly) {
            // delay phases exp(+j 2 pi T1 k2 f / N), in a block of their own: without delays
            // the plain filter bank skips it as a whole
            sfor<0, R2>([&](auto K2) {
                constexpr int k2 = decltype(K2)::value;
                float2 &x = v[bitrev(k2, ilog2(R2))];
                const float2 y = cmul(x, dsm[H2 * k2 + h2]);
                x = k2 == 0 && h2 == 0 ? x : y;
            });
        }
        if (valid) {
            sfor<0, R2>([&](auto K2) {
                constexpr int k2 = decltype(K2)::value;
                [[maybe_unused]] const int k = row + T1 * (H2 * k2 + h2);
                float2 x = v[bitrev(k2, ilog2(R2))];
                if constexpr (FEAT == kDelay && (k2 != 0 || H2 == 2)) {
                    // delay phase exp(+j 2 pi T1 k2 f / N)
                    if (has_dly && (k2 != 0 || h2 != 0)) x = cmul(x, dsm[H2 * k2 + h2]);
                }
                if constexpr (MODE == kRequant || MODE == kRequantPlanar) {
                    const uint32_t q = pack_q<MODE == kRequantPlanar>(x, __ldg(scale + k));
                    reinterpret_cast<uint16_t *>(stg)[slot(k, s)] = (uint16_t)q;
                } else if constexpr (MODE == kFloatOut) {
                    reinterpret_cast<float2 *>(stg)[(size_t)k * (ROWW / 2) + s] = x;
                } else {
                    pw[k2] += x.x * x.x + x.y * x.y;
                }
            });
        }
        if (C::POW && join) {
            // The FP32 sums of the FFTs that share a warp are added (shuffles), each FFT's
            // lanes writing their share of the channels to the warp's part of the exchange
            // buffer; then a thread per channel adds the warps' sums as FP32 pairs of sum and
            // error, and the result to the FP64 sum (each warp's sum added in FP64: N = 1024, 16
            // inputs x 256 spectra 28.9 us against 23.0; two of them are two conversions and one
            // add either way).
            constexpr int FW = C::FW, PARTS = G / FW;  // FFTs per warp; partial sums
            const int fft = (threadIdx.x % 32) / TG;
            float *part = ex + (size_t)(g / FW * FW) * C::GS;
            sfor<0, R2>([&](auto K2) {
                constexpr int k2 = decltype(K2)::value;
                float p = pw[k2];
#pragma unroll
                for (int x = 1; x < FW; x *= 2) p += __shfl_xor_sync(0xffffffffu, p, x * TG);
                if (FW == 1 || fft == k2 % FW) part[row + T1 * (H2 * k2 + h2)] = p;
                pw[k2] = 0.0f;
            });
            __syncthreads();
            for (int m = threadIdx.x; m < N; m += NT) {
                float d[PARTS];
#pragma unroll
                for (int x = 0; x < PARTS; ++x) d[x] = ex[(size_t)(x * FW) * C::GS + m];
                double sum;
                if constexpr (PARTS == 2) {
                    sum = (double)d[0] + (double)d[1];
                } else {
                    float err = 0.0f;
#pragma unroll
                    for (int h = PARTS / 2; h > 0; h /= 2)
#pragma unroll
                        for (int x = 0; x < h; ++x) d[x] = add_err(d[x], d[x + h], err);
                    // (the error of an infinite sum is no number)
                    sum = (double)d[0] + (err == err ? (double)err : 0.0);
                }
                if (C::PSUM && s0 / G >= C::PQ) sum += psum[m];  // not the first time
                if (C::PSUM && s0 + G < sb) psum[m] = sum;
                else atomicAdd(&power[m], sum);
            }
            __syncthreads();
            if (use_async && s0 + G < sb) issue_raw(s0 + G + g);
        }
    }

    if constexpr (MODE != kPower) {
        __syncthreads();
        // ---- corner turn: row (k, i) gets spectra a0 .. a0 + nv - 1
        const int nv = min(sb, K - a0);
        if constexpr (MODE == kRequantPlanar || MODE == kRequant) {
            uint16_t *dst = reinterpret_cast<uint16_t *>(out);
            // planar FP16 layout [k][plane][i][a]; int8 layout [k][i][a] (complex int8)
            constexpr int PL = MODE == kRequantPlanar ? 2 : 1;
            if (vec_out && (C::VARSB || nv == SB)) {  // nv is a multiple of 8: sb and K are
                // each thread moves 8 spectra of one channel row: 4 staged words
                // (the code pairs of 2 spectra each) -> one 16-byte store per plane
                constexpr int CPR = SB / 8;          // 8-spectrum chunks per row
                constexpr int RPI = NT / CPR;  // rows per iteration
                const int q = threadIdx.x % CPR;
                int k = threadIdx.x / CPR;
                // physical words of logical words 4q .. 4q + 3 in row k; the swizzle
                // (k >> SW) & (ROWW - 1) is the same for k + RPI
                static_assert((RPI >> C::SW) % ROWW == 0 || RPI >= N, "");
                const int h = (k >> C::SW) & (ROWW - 1);
                const int o0 = (4 * q) ^ h, o1 = (4 * q + 1) ^ h, o2 = (4 * q + 2) ^ h, o3 = (4 * q + 3) ^ h;
                const uint32_t *src = stg + (size_t)k * ROWW;
                uint4 *d = reinterpret_cast<uint4 *>(dst + ((size_t)(PL * k) * n_in + i) * K + a0 + 8 * q);
                const size_t dstep = (size_t)PL * RPI * n_in * K / 8, dplane = (size_t)n_in * K / 8;
                const int k_end = !C::VARSB || 8 * q < nv ? N : 0;
                for (; k < k_end; k += RPI, src += RPI * ROWW, d += dstep) {
                    const uint32_t w0 = src[o0], w1 = src[o1], w2 = src[o2], w3 = src[o3];
                    if constexpr (MODE == kRequantPlanar) {
                        uint4 re, im;
                        ob_codes_to_f16_planes(w0, re.x, im.x);
                        ob_codes_to_f16_planes(w1, re.y, im.y);
                        ob_codes_to_f16_planes(w2, re.z, im.z);
                        ob_codes_to_f16_planes(w3, re.w, im.w);
                        d[0] = re;
                        d[dplane] = im;
                    } else {
                        d[0] = make_uint4(w0, w1, w2, w3);
                    }
                }
            } else {
                // unaligned rows or a short last block: a thread per code, whole rows per store
                // instruction (one write request per row), U staged codes in flight
                constexpr int U = 8, RPI = NT / SB;  // rows per round
                const uint16_t *sh = reinterpret_cast<const uint16_t *>(stg);
                const size_t plane = (size_t)n_in * K;
                const int c = threadIdx.x % SB;
                for (int k0 = threadIdx.x / SB; c < nv && k0 < N; k0 += U * RPI) {
                    uint32_t code[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) code[u] = k0 + u * RPI < N ? sh[slot(k0 + u * RPI, c)] : 0u;
                    uint16_t *d = dst + ((size_t)(PL * k0) * n_in + i) * K + a0 + c;
#pragma unroll
                    for (int u = 0; u < U; ++u, d += PL * RPI * plane) {
                        if (k0 + u * RPI >= N) break;
                        if constexpr (MODE == kRequantPlanar) {
                            uint32_t re, im;
                            ob_codes_to_f16_planes(code[u], re, im);
                            d[0] = (uint16_t)re;
                            d[plane] = (uint16_t)im;
                        } else {
                            d[0] = (uint16_t)code[u];
                        }
                    }
                }
            }
        } else {
            float2 *dst = reinterpret_cast<float2 *>(out);
            const float2 *sh = reinterpret_cast<const float2 *>(stg);
            for (int e = threadIdx.x; e < N * SB; e += NT) {
                int k = e / SB, c = e % SB;
                if (c < nv) dst[((size_t)k * n_in + i) * K + a0 + c] = sh[(size_t)k * (ROWW / 2) + c];
            }
        }
    }
}

template <int N, bool I8, int MODE, int FEAT, int P = 0>
corr_status launch_one_(const FShape &f, const void *volt, const float *scale, void *out, double *power,
                       cudaStream_t st, const PfbArgs &pfb = {}) {
    using C = FCfg<N, I8, MODE, FEAT>;
    constexpr auto kern = k_fengine<N, I8, MODE, FEAT, P>;
    if (const corr_status s = allow_smem<kern>((int)C::smem); s != CORR_OK) return s;
    // 16-byte row stores need 16-byte aligned rows: an aligned buffer and 8 | n_spectra
    const int vec_out = (reinterpret_cast<uintptr_t>(out) % 16 == 0) && (f.n_spectra % 8 == 0);
    // blockIdx.x (the spectra block) varies fastest, so the CTAs resident at one time
    // write neighbouring segments of the same output rows
    // spectra per CTA: SB, or half of it (whole rounds of the G FFTs in flight, whole 16-byte
    // pieces of a row) while the launch has fewer CTAs than the chip has SMs:
    // few inputs and spectra then take the time of one round instead of SB / G of them (7
    // inputs x 80 spectra at N = 4096, one launch per input: 487 -> 396 us
    // for the host pipeline's call)
    const int n_rows = f.n_run < 0 ? f.n_in : f.n_run;
    int sb = C::SB;
    while (C::VARSB && sb / 2 >= C::G && sb / 2 >= 8 && (long long)((f.n_spectra + sb - 1) / sb) * n_rows < f.n_sm) sb /= 2;
    // The power pass: blocks of SB spectra per CTA up to 2^16 samples, while 16 CTAs are left
    // for each SM (a CTA ends with one FP64 atomic per channel, and atomics to one address take
    // 16 ns each: with one CTA per block they were all the time of short transforms); parts
    // of a block, whole rounds of the G FFTs in flight, while there are not two CTAs per SM
    // (one at N = 4096, whose atomics weigh more: 16 inputs x 60 spectra, shared DFTs, 31.8 -> 27.8
    // us, but 36.3 with one CTA per block).
    // 128 inputs, int8, us: N = 16 x 32768 spectra 1213 -> 118, N = 64 x 32768 2094 -> 354, N =
    // 256 x 16384 2095 -> 668, N = 512 x 8192 2018 -> 818, N = 1024 x 4096 1332 -> 728, N =
    // 2048 x 2048 1891 -> 996, N = 4096 x 1024 1319 -> 1002.
    if (C::POW) {
        const long long blocks = (f.n_spectra + C::SB - 1) / C::SB, want = 16LL * f.n_sm;
        sb *= (int)std::min(std::min(blocks, (long long)C::POWB), std::max(1LL, blocks * n_rows / want));
        while (sb <= C::SB && sb / 2 >= C::G && (long long)((f.n_spectra + sb - 1) / sb) * n_rows < (N >= 4096 ? 1LL : 2LL) * f.n_sm) sb /= 2;
    }
    dim3 grid((f.n_spectra + sb - 1) / sb, n_rows);
    // asynchronous raw copies need 16-byte aligned frames (2 N bytes each, N >= 64); the
    // public entry points only accept 16-byte aligned voltages, so this is a safeguard
    const int async_raw = reinterpret_cast<uintptr_t>(volt) % 16 == 0;
    kern<<<grid, C::NT, C::smem, st>>>(volt, scale, out, power, f.n_in, f.n_spectra, f.tw, f.i0, vec_out,
                                          f.dint, f.dph, async_raw, pfb, sb);
    return check_launch("k_fengine");
}

template <int MODE, int FEAT>
corr_status launch_mode(const FShape &f, const void *volt, const float *scale, void *out, double *power,
                        cudaStream_t st) {
#define CORR_F_CASE(NN)                                                                      \
    case NN:                                                                                 \
        return f.i8 ? launch_one_<NN, true, MODE, FEAT>(f, volt, scale, out, power, st)      \
                    : launch_one_<NN, false, MODE, FEAT>(f, volt, scale, out, power, st);
    switch (f.n_chan) {
        CORR_F_CASE(16)
        CORR_F_CASE(64)
        CORR_F_CASE(128)
        CORR_F_CASE(256)
        CORR_F_CASE(512)
        CORR_F_CASE(1024)
        CORR_F_CASE(2048)
        CORR_F_CASE(4096)
        default: return CORR_EUNSUPPORTED;
    }
#undef CORR_F_CASE
}

// The fused filter bank of up to P taps: int8 voltages, re-packed output.
template <int P>
corr_status launch_pfb(bool planar, const FShape &f, const PfbArgs &pfb, const void *volt, const float *scale, void *out,
                       cudaStream_t st) {
#define CORR_F_CASE(NN)                                                                                           \
    case NN:                                                                                                      \
        return planar ? launch_one_<NN, true, kRequantPlanar, kPfb, P>(f, volt, scale, out, nullptr, st, pfb)     \
                      : launch_one_<NN, true, kRequant, kPfb, P>(f, volt, scale, out, nullptr, st, pfb);
    switch (f.n_chan) {
        CORR_F_CASE(64)
        CORR_F_CASE(128)
        CORR_F_CASE(256)
        CORR_F_CASE(512)
        CORR_F_CASE(1024)
        CORR_F_CASE(2048)
        CORR_F_CASE(4096)
        default: return CORR_EUNSUPPORTED;
    }
#undef CORR_F_CASE
}

// The power pass of the fused filter bank of up to P taps.
template <int P>
corr_status launch_pfb_power(const FShape &f, const PfbArgs &pfb, const void *volt, double *power, cudaStream_t st) {
#define CORR_F_CASE(NN) \
    case NN: return launch_one_<NN, true, kPower, kPfb, P>(f, volt, nullptr, nullptr, power, st, pfb);
    switch (f.n_chan) {
        CORR_F_CASE(64)
        CORR_F_CASE(128)
        CORR_F_CASE(256)
        CORR_F_CASE(512)
        CORR_F_CASE(1024)
        CORR_F_CASE(2048)
        CORR_F_CASE(4096)
        default: return CORR_EUNSUPPORTED;
    }
#undef CORR_F_CASE
}

// Every (mode, n_chan, input type) of one front-end feature.
template <int FEAT>
corr_status launch_feature(int mode, const FShape &f, const void *volt, const float *scale, void *out,
                           double *power, cudaStream_t st) {
    switch (mode) {
        case kFloatOut: return launch_mode<kFloatOut, FEAT>(f, volt, scale, out, power, st);
        case kRequant: return launch_mode<kRequant, FEAT>(f, volt, scale, out, power, st);
        case kPower: return launch_mode<kPower, FEAT>(f, volt, scale, out, power, st);
        case kRequantPlanar: return launch_mode<kRequantPlanar, FEAT>(f, volt, scale, out, power, st);
        default: return CORR_EINVAL;
    }
}

}  // namespace

// Per-feature entry points, one translation unit each.
corr_status fengine_run_plain(int mode, const FShape &f, const void *volt, const float *scale, void *out,
                              double *power, cudaStream_t st);
corr_status fengine_run_delay(int mode, const FShape &f, const void *volt, const float *scale, void *out,
                              double *power, cudaStream_t st);
// Fused filter bank, win [taps][n_chan]: taps <= 4 and <= 8.
corr_status fengine_run_pfb4(bool planar, const FShape &f, const float *win, int taps, const void *volt,
                             const float *scale, void *out, cudaStream_t st);
corr_status fengine_run_pfb8(bool planar, const FShape &f, const float *win, int taps, const void *volt,
                             const float *scale, void *out, cudaStream_t st);
corr_status fengine_run_pfb_power(const FShape &f, const float *win, int taps, const void *volt, double *power,
                                  cudaStream_t st);

}  // namespace corr
