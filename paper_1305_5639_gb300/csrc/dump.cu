// Integration dump: the long-integration FP64 buffer receives the integration
// accumulator (INT32 pairs for INT8, FP32 pairs otherwise) in one streaming pass
// (read 8 B + read/write 16 B per visibility), with the FP64 pipe doing at most the
// add itself (exact_add.cuh: INT32 sums are added in integers, FP32 sums converted
// in integers). The accumulator is not
// rewritten with zeros: the handle marks it clear, so the next X-engine launch
// overwrites it instead of adding to it and corr_get_accum returns zeros meanwhile.
#include "exact_add.cuh"
#include "internal.h"

namespace corr {
namespace {

// COPY: the new long integration also goes to out (corr_dump with vis_out), instead of a
// device copy after the pass: 16 bytes per visibility less, and a launch (16 inputs x 64
// channels: 3.6 us of a 20.7 us step).
template <typename AccT, bool COPY>
__global__ void __launch_bounds__(256) k_dump(const AccT *__restrict__ acc, double2 *__restrict__ vis, long long n,
                                              double2 *__restrict__ out) {
    // four visibilities per thread and round, all loads before any store (more bytes in
    // flight per thread for the read-modify-write of the FP64 buffer)
    constexpr int U = 4;
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; e + (U - 1) * stride < n; e += U * stride) {
        AccT a[U];
        double2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = __ldcs(acc + e + u * stride);
            v[u] = vis[e + u * stride];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const double2 s = add_exact(v[u], a[u]);
            vis[e + u * stride] = s;
            if (COPY) __stcs(out + e + u * stride, s);
        }
    }
    for (; e < n; e += stride) {
        const double2 s = add_exact(vis[e], __ldcs(acc + e));
        vis[e] = s;
        if (COPY) __stcs(out + e, s);
    }
}

template <typename AccT>
void launch_k(unsigned blocks, const void *acc, double2 *vis, long long n, double2 *out, cudaStream_t st) {
    const AccT *a = static_cast<const AccT *>(acc);
    if (out) k_dump<AccT, true><<<blocks, 256, 0, st>>>(a, vis, n, out);
    else k_dump<AccT, false><<<blocks, 256, 0, st>>>(a, vis, n, nullptr);
}

// n visibilities of acc into vis (and the sums to out)
corr_status dump_pass(const Handle &h, const void *acc, double2 *vis, long long n, double2 *out, cudaStream_t st) {
    if (n <= 0) return CORR_OK;
    StageScope sc(h, CORR_STAGE_DUMP, st);
    long long blocks = (n + 255) / 256;
    const long long cap = (long long)h.n_sm * 16;
    if (blocks > cap) blocks = cap;
    if (h.precision == CORR_PREC_INT8) launch_k<int2>((unsigned)blocks, acc, vis, n, out, st);
    else launch_k<float2>((unsigned)blocks, acc, vis, n, out, st);
    return check_launch("k_dump");
}

}  // namespace

corr_status launch_dump_src(const Handle &h, const void *acc, double2 *out, cudaStream_t st) {
    return dump_pass(h, acc, h.vis64, (long long)h.n_chan * h.n_base, out, st);
}

corr_status launch_dump_range(const Handle &h, int c0, int c1, cudaStream_t st) {
    const long long off = (long long)c0 * h.n_base;
    // (8 bytes per accumulator entry in every precision)
    return dump_pass(h, static_cast<const char *>(h.acc) + 8 * off, h.vis64 + off, (long long)(c1 - c0) * h.n_base,
                     nullptr, st);
}

}  // namespace corr
