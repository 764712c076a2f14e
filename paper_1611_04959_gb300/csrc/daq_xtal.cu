// Per-crystal full-resolution fill sum (Table 2, fill-by-fill sum kernel, in
// the form its thread count suggests: one term per crystal and sample):
//
//   Qx[c][x][t] += s[f][c][x][t] - P[f][c][x]   for every fill f and t < len_f
//
// with P the per-crystal pedestal of Table 2's pedestal kernel (the first
// min(ped_samples, len) samples, rounded half up).  Q stays on the device and
// accumulates over calls.  Two kernels: pedestals (one warp per crystal row),
// then a streaming pass in which each thread owns groups of 8 consecutive samples
// of the rows taken as one flat sequence, adds every fill of the call in registers
// and read-modify-writes the 8 int64 accumulators once.  HBM traffic per call: the samples once
// (2 bytes each) and Q once each way (16 bytes per crystal-sample).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "daq.h"

namespace daq_xtal {

constexpr int kThreads = 256;

struct XLayout {
    size_t status, lens, ped, total;
};

XLayout xlayout(int64_t n_fills, int64_t n_rows)
{
    auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
    XLayout l;
    l.status = 0;
    l.lens = 256;
    l.ped = up(l.lens + sizeof(int32_t) * (size_t)std::max<int64_t>(n_fills, 1));
    l.total = up(l.ped + sizeof(int32_t) * (size_t)std::max<int64_t>(n_rows, 1));
    return l;
}

__device__ __forceinline__ long long floor_div_ll(long long a, long long b)
{
    long long q = a / b;
    if ((a % b != 0) && ((a < 0) != (b < 0))) --q;
    return q;
}

// Fill lengths (clamped; out-of-range ones flagged in *status, cleared by the
// host before the launch) and every row's pedestal.
__global__ void __launch_bounds__(kThreads) xtal_prepare_kernel(const int16_t *samples, int n_fills, int n_calo,
                                                                int n_xtal, int64_t pitch, const int32_t *fill_len,
                                                                int ped_samples, int32_t *lens, int32_t *ped,
                                                                unsigned long long *status)
{
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * kThreads) >> 5;
    for (long long f = (long long)blockIdx.x * kThreads + threadIdx.x; f < n_fills; f += (long long)gridDim.x * kThreads) {
        long long len = fill_len ? (long long)fill_len[f] : pitch;
        if (len < 0 || len > pitch) {
            atomicOr(status, (unsigned long long)DAQ_DEV_BAD_FILL_LEN);
            len = len < 0 ? 0 : pitch;
        }
        lens[f] = (int32_t)len;
    }
    const long long n_rows = (long long)n_fills * n_calo * n_xtal;
    for (long long r = gw; r < n_rows; r += nw) {
        const long long f = r / ((long long)n_calo * n_xtal);
        long long len = fill_len ? (long long)fill_len[f] : pitch;
        len = len < 0 ? 0 : (len > pitch ? pitch : len);
        const long long n = len < ped_samples ? len : ped_samples;
        const int16_t *row = samples + r * pitch;
        long long sum = 0;
        for (long long t = lane; t < n; t += 32) sum += row[t];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
        if (lane == 0) ped[r] = n > 0 ? (int32_t)floor_div_ll(sum + n / 2, n) : 0;
    }
}

__device__ __forceinline__ void load_q(const long long *p, long long (&v)[8], bool wide)
{
    if (wide) {  // 32 bytes an access: every lane takes whole sectors
#pragma unroll
        for (int k = 0; k < 8; k += 4)
            asm volatile("ld.global.v4.s64 {%0, %1, %2, %3}, [%4];"
                         : "=l"(v[k]), "=l"(v[k + 1]), "=l"(v[k + 2]), "=l"(v[k + 3])
                         : "l"(p + k)
                         : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            const longlong2 t = *reinterpret_cast<const longlong2 *>(p + k);
            v[k] = t.x;
            v[k + 1] = t.y;
        }
    }
}

__device__ __forceinline__ void store_q(long long *p, const long long (&v)[8], bool wide)
{
    if (wide) {
#pragma unroll
        for (int k = 0; k < 8; k += 4)
            asm volatile("st.global.v4.s64 [%0], {%1, %2, %3, %4};" ::"l"(p + k), "l"(v[k]), "l"(v[k + 1]), "l"(v[k + 2]),
                         "l"(v[k + 3])
                         : "memory");
    } else {
#pragma unroll
        for (int k = 0; k < 8; k += 2) __stcs(reinterpret_cast<longlong2 *>(p + k), make_longlong2(v[k], v[k + 1]));
    }
}

// Bound by HBM: 2 bytes a sample, 16 bytes a cell.  A thread owns 8 consecutive
// cells of the whole array [n_calo][n_xtal][pitch], whatever the pitch, so that its
// accumulators are 64-byte aligned and (where one fill's samples are a multiple of
// 8, or there is one fill) its samples 16-byte aligned; a group of 8 may hold the
// end of one row and the start of the next.  Accumulators move 32 bytes a lane and
// access, whole sectors: 24 x 54 x 560,000 cells take 1.94 ms (6.75 TB/s, the copy
// rate) against 2.17 with accesses of 16 bytes, 64 apart from lane to lane, and
// 3.03 with lanes on consecutive 16 bytes and 4-byte sample loads.  Groups within a
// row, taken sample by sample where the pitch is odd, took 1.70 ms for three fills of
// 24 x 54 x 99,999; these take 0.45.  A sample past its fill's length is not read:
// eight fills of 24 x 54 x 70,000 cut to 7,000 take 262 us, 465 if it is.  Four CTAs an
// SM: at five the 64 registers do not suffice (2.22 ms).
// kVec: aligned 16-byte sample loads, of kAhead fills at once (two: 721 us for four
// fills of 140,000 samples against 731 with one and 748 with four, whose registers
// cost a CTA); wide: q is 32-byte aligned.  I: the type of rows and places in them, 32
// bits where the cells allow (one division a group, and the compares with every
// fill's length: those four fills take 674 us so).
template <bool kVec, int kAhead, typename I>
__global__ void __launch_bounds__(kThreads, 4) xtal_sum_kernel(const int16_t *samples, int n_fills, int n_calo,
                                                            int n_xtal, int64_t pitch, const int32_t *lens,
                                                            const int32_t *ped, long long *q, bool wide)
{
    const long long n_rows = (long long)n_calo * n_xtal;
    const long long cells = n_rows * pitch;
    const long long groups = (cells + 7) / 8;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < groups; i += (long long)gridDim.x * kThreads) {
        const long long at = 8 * i;
        const I row = (I)at / (I)pitch;
        const I t0 = (I)at - row * (I)pitch;
        const bool full = at + 8 <= cells;
        const bool one_row = full && (long long)t0 + 8 <= pitch;
        long long acc[8];
        if (full) {  // the accumulators' loads go out before the samples'
            load_q(q + at, acc, wide);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = at + k < cells ? q[at + k] : 0;
        }
        for (int f0 = 0; f0 < n_fills; f0 += kAhead) {
            int4 v[kAhead];
            if (kVec && one_row) {
#pragma unroll
                for (int u = 0; u < kAhead; ++u)
                    if (f0 + u < n_fills && t0 + 8 <= (I)lens[f0 + u])
                        v[u] = __ldcs(reinterpret_cast<const int4 *>(samples + (long long)(f0 + u) * cells + at));  // read once
            }
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int f = f0 + u;
                if (f >= n_fills) break;
                const I len = (I)lens[f];
                const int32_t *P = ped + (long long)f * n_rows + row;
                if (kVec && one_row && t0 + 8 <= len) {
                    const int p = P[0];
                    const uint32_t w[4] = {(uint32_t)v[u].x, (uint32_t)v[u].y, (uint32_t)v[u].z, (uint32_t)v[u].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {  // a sample less a pedestal fits 32 bits
                        acc[2 * k] += (int)(int16_t)(w[k] & 0xffffu) - p;
                        acc[2 * k + 1] += (int)(int16_t)(w[k] >> 16) - p;
                    }
                } else if (!one_row || t0 < len) {
                    // the end of a row, of the fill or of the array
                    const int16_t *src = samples + (long long)f * cells + at;
                    I t = t0;
                    int r = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        if (at + k < cells && t < len) acc[k] += (int)src[k] - P[r];
                        if (++t == (I)pitch) {
                            t = 0;
                            ++r;
                        }
                    }
                }
            }
        }
        if (full) {
            store_q(q + at, acc, wide);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (at + k < cells) q[at + k] = acc[k];
        }
    }
}

using SumKernel = void (*)(const int16_t *, int, int, int, int64_t, const int32_t *, const int32_t *, long long *, bool);
template <int kAhead> SumKernel pick(bool vec, bool small)
{
    if (vec) return small ? xtal_sum_kernel<true, kAhead, uint32_t> : xtal_sum_kernel<true, kAhead, unsigned long long>;
    return small ? xtal_sum_kernel<false, kAhead, uint32_t> : xtal_sum_kernel<false, kAhead, unsigned long long>;
}

int grid_for(long long work)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long want = (work + kThreads - 1) / kThreads;
    return (int)std::max<long long>(1, std::min<long long>(want, (long long)std::max(sms, 1) * 8));
}

}  // namespace daq_xtal

using namespace daq_xtal;

extern "C" {

int daq_crystal_sum_workspace_size(int n_calo, int n_xtal, int n_fills, size_t *bytes)
{
    if (!bytes || n_calo < 0 || n_xtal < 1 || n_fills < 0) return DAQ_EINVAL;
    *bytes = xlayout(n_fills, (int64_t)n_fills * n_calo * n_xtal).total;
    return DAQ_OK;
}

int daq_crystal_sum(const int16_t *samples, int n_calo, int n_xtal, int64_t n_samples, int n_fills,
                    const daq_params *params, int64_t *q_xtal)
{
    if (!params || n_calo < 0 || n_xtal < 1 || n_samples < 0 || n_fills < 0 || params->ped_samples < 1)
        return DAQ_EINVAL;
    const int64_t n_rows = (int64_t)n_fills * n_calo * n_xtal;
    const XLayout l = xlayout(n_fills, n_rows);
    if (!params->workspace || params->workspace_bytes < l.total ||
        (reinterpret_cast<uintptr_t>(params->workspace) & 15))
        return DAQ_EINVAL;
    const int64_t cells = (int64_t)n_calo * n_xtal * n_samples;
    if (cells > 0 && (!q_xtal || (reinterpret_cast<uintptr_t>(q_xtal) & 15))) return DAQ_EINVAL;
    if (n_rows * n_samples > 0 && !samples) return DAQ_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(params->stream);
    unsigned char *ws = static_cast<unsigned char *>(params->workspace);
    unsigned long long *status = reinterpret_cast<unsigned long long *>(ws + l.status);
    int32_t *lens = reinterpret_cast<int32_t *>(ws + l.lens);
    int32_t *ped = reinterpret_cast<int32_t *>(ws + l.ped);
    if (cudaMemsetAsync(status, 0, sizeof(*status), s) != cudaSuccess) return DAQ_ECUDA;
    xtal_prepare_kernel<<<grid_for(std::max<int64_t>(n_rows * 32, n_fills)), kThreads, 0, s>>>(
        samples, n_fills, n_calo, n_xtal, n_samples, params->fill_len, params->ped_samples, lens, ped, status);
    if (cudaGetLastError() != cudaSuccess) return DAQ_ECUDA;
    if (cells > 0 && n_fills > 0) {
        const bool vec = (cells % 8 == 0 || n_fills == 1) && (reinterpret_cast<uintptr_t>(samples) & 15) == 0;
        const bool wide = (reinterpret_cast<uintptr_t>(q_xtal) & 31) == 0, small = cells <= (int64_t)0xffffffff;
        const auto kernel = n_fills == 1 ? pick<1>(vec, small) : pick<2>(vec, small);
        kernel<<<grid_for((cells + 7) / 8), kThreads, 0, s>>>(samples, n_fills, n_calo, n_xtal, n_samples, lens, ped,
                                                              reinterpret_cast<long long *>(q_xtal), wide);
        if (cudaGetLastError() != cudaSuccess) return DAQ_ECUDA;
    }
    if (params->flags & DAQ_SYNC) {
        unsigned long long st = 0;
        if (cudaMemcpyAsync(&st, status, sizeof(st), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return DAQ_ECUDA;
        if (st & DAQ_DEV_BAD_FILL_LEN) return DAQ_EINVAL;
    }
    return DAQ_OK;
}

}  // extern "C"
