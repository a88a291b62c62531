// Register-tiled complex products on the FP32 pipe, shared by the CUDA-core X-engine
// (xengine_cudacore.cu) and the CUDA-core adjoint (adjoint.cu).
//
// A CTA of 128 threads forms a tile of (8 RT) rows x (16 CT) columns; its four warps
// take the quarters (2 x 2), and in a warp 4 x 8 lanes own RT x CT complex sums each.
// Both operands lie in shared memory as [k][row] complex values, filled by asynchronous
// copies kFtStages deep. A lane's rows (and its columns, for even CT) are neighbours in
// pairs, so one 16-byte load brings two operands. The sums are packed (Re, Im):
//     acc += a (br, br);   acc += a' (bi, bi)     with a' = a rotated by -j (conj) or +j
// two fma.rn.f32x2 per product, the rotation and the duplicates built in registers.
// What bounds it: per k a warp issues 2 RT CT packed FMAs of two cycles, 2 RT + 4 CT
// moves and (RT + CT) / 2 loads, 128 FMA cycles against about 100 issue slots and 96 of
// the shared-memory pipe at RT = 8, CT = 4. Measured forms that lost: scalar FMAs (no
// moves, but three operand reads per cycle: dispatch stalls held the FMA pipe at 60 %)
// and duplicated operands in shared memory (16 bytes per value: the loads took twice the
// FMAs' time).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_common.cuh"

namespace corr {

constexpr int kFtNth = 128;    // threads per CTA
constexpr int kFtKC = 16;      // contraction steps per shared-memory stage
constexpr int kFtStages = 3;   // stages in flight

// 8-byte asynchronous global -> shared copy, zeros if !live (the source is not read then)
__device__ __forceinline__ void ft_copy8(float2 *dst, const float2 *src, bool live) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(live ? 8 : 0)
                 : "memory");
}
__device__ __forceinline__ void ft_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest group have landed (for this thread's copies)
__device__ __forceinline__ void ft_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kFtStages - 2) : "memory"); }

// Position of this thread in the 2 x 2 warps x (4 x 8) lanes grid.
template <int RT, int CT>
struct FtPos {
    static_assert(RT % 2 == 0, "rows are loaded in pairs");
    int wr, wc, row0, col0;
    __device__ __forceinline__ FtPos() {
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        wr = w >> 1;
        wc = w & 1;
        row0 = wr * 4 * RT + 2 * (lane >> 3);
        col0 = wc * 8 * CT + (CT % 2 == 0 ? 2 : 1) * (lane & 7);
    }
    // tile row of sum r, tile column of sum c
    __device__ __forceinline__ int row(int r) const { return row0 + 8 * (r / 2) + r % 2; }
    __device__ __forceinline__ int col(int c) const { return CT % 2 == 0 ? col0 + 16 * (c / 2) + c % 2 : col0 + 8 * c; }
};

template <int RT, int CT>
__device__ __forceinline__ void ft_zero(float2 (&acc)[RT][CT]) {
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < CT; ++c) acc[r][c] = make_float2(0.f, 0.f);
}

// acc += a b (CONJ: a conj(b)) over one stage: operands a[k * AP + row], b[k * BP + col]
// from the thread's first row and column on (both 16-byte aligned where loaded in pairs).
template <bool CONJ, int RT, int CT, int AP, int BP>
__device__ __forceinline__ void ft_stage(float2 (&acc)[RT][CT], const float2 *a, const float2 *b) {
    static_assert(AP % 2 == 0 && (CT % 2 != 0 || BP % 2 == 0), "pairs are 16-byte aligned");
#pragma unroll 4
    for (int k = 0; k < kFtKC; ++k) {
        float2 bv[CT];
        if constexpr (CT % 2 == 0) {
#pragma unroll
            for (int c = 0; c < CT; c += 2) {
                const float4 q = *reinterpret_cast<const float4 *>(b + k * BP + 8 * c);
                bv[c] = make_float2(q.x, q.y);
                bv[c + 1] = make_float2(q.z, q.w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < CT; ++c) bv[c] = b[k * BP + 8 * c];
        }
#pragma unroll
        for (int r = 0; r < RT; r += 2) {
            const float4 q = *reinterpret_cast<const float4 *>(a + k * AP + 4 * r);
            const float2 av[2] = {make_float2(q.x, q.y), make_float2(q.z, q.w)};
#pragma unroll
            for (int e = 0; e < 2; ++e) {
#pragma unroll
                for (int c = 0; c < CT; ++c)
                    acc[r + e][c] = f2_fma(av[e], make_float2(bv[c].x, bv[c].x), acc[r + e][c]);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 rot = CONJ ? make_float2(av[e].y, -av[e].x) : make_float2(-av[e].y, av[e].x);
#pragma unroll
                for (int c = 0; c < CT; ++c)
                    acc[r + e][c] = f2_fma(rot, make_float2(bv[c].y, bv[c].y), acc[r + e][c]);
            }
        }
    }
}

}  // namespace corr
