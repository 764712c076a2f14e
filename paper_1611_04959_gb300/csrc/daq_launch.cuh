// Launch of the two-pass form: its plan, and the count, scan and compact
// kernels of one tile width.  Included by the source files that instantiate
// them, one for tensor-box loads and one for row copies.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "daq_twopass.cuh"

namespace daq {

struct Plan {
    int tw, hl, hr, ew, rs, boxw, nbox, box_stride, slot_bytes, need_sarr, mode;
    int halo_free;  // two-pass form: the count pass loads the tile proper only
    int boxw_b, nbox_b, box_stride_b, slot_bytes_b, rs_b;  // compact pass (two-pass mode)
    size_t smem, smem_b;                                   // tile (or count) kernel, compact kernel
    int str_meta, str_stages;                              // streaming / single-read forms: tile records, row stages per CTA
    int pk_slots, pk_cols;                                 // single-read form: park slots, Tensor Memory columns per slot
    int count_ns;                                          // two-pass form: tile slots of the count kernel (2 or 3)
    int64_t max_tiles;
    int64_t ws_tiles;  // tiles the workspace is laid out for: also covers the two-pass plan a call may fall back to
};

template <typename K> static cudaError_t ensure_smem(K kernel, size_t bytes, size_t *configured)
{
    static std::mutex mu;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> g(mu);
    if (dev >= 0 && dev < 64 && configured[dev] < bytes) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
        configured[dev] = bytes;
    }
    return cudaSuccess;
}

// Launch with programmatic stream serialization: the kernel may be scheduled
// while the previous kernel of the stream drains; it waits for it in-kernel
// (pdl_wait) before reading its outputs.
template <typename K>
static cudaError_t launch_pdl(K kernel, int grid, int block, size_t smem, cudaStream_t s, const KArgs &a)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return cudaErrorUnknown;
    cfg.attrs = attr;
    cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// The count kernel for NS slots, halo-free or not, grids from occupancy when
// grid <= 0.
template <int TW, int NS, bool HF, bool ROWS>
static cudaError_t launch_count(const KArgs &a, const Plan &pl, int grid, int sms, int64_t tiles, cudaStream_t s)
{
    static size_t conf[64] = {0};
    cudaError_t e = ensure_smem(daq_count_kernel<TW, NS, HF, ROWS>, pl.smem, conf);
    if (e != cudaSuccess) return e;
    if (grid <= 0) {
        int per = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, daq_count_kernel<TW, NS, HF, ROWS>, count_threads<NS>(), pl.smem);
        if (e != cudaSuccess) return e;
        if (per < 1) return cudaErrorInvalidConfiguration;
        grid = per * sms;
    }
    grid = (int)std::min<int64_t>(grid, tiles);
    return launch_pdl(daq_count_kernel<TW, NS, HF, ROWS>, grid, count_threads<NS>(), pl.smem, s, a);
}

// The compact kernel (DAQ_SPARSE: the form that passes over tiles without a
// marked sample), grids from occupancy when grid <= 0.
template <int TW, bool kSparse, bool ROWS>
static cudaError_t launch_compact(const KArgs &a, const Plan &pl, int grid, int sms, int64_t tiles, cudaStream_t s)
{
    static size_t conf[64] = {0};
    cudaError_t e = ensure_smem(daq_compact_kernel<TW, kSparse, ROWS>, pl.smem_b, conf);
    if (e != cudaSuccess) return e;
    if (grid <= 0) {
        int per = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, daq_compact_kernel<TW, kSparse, ROWS>, 256, pl.smem_b);
        if (e != cudaSuccess) return e;
        if (per < 1) return cudaErrorInvalidConfiguration;
        grid = per * sms;
    }
    grid = (int)std::min<int64_t>(grid, tiles);
    return launch_pdl(daq_compact_kernel<TW, kSparse, ROWS>, grid, 256, pl.smem_b, s, a);
}

// Count pass, scan, compact pass.  Events (optional): [2] after the count
// kernel, [3] after the scan, [4] after the compact kernel.
template <int TW, bool ROWS>
static cudaError_t launch_twopass(const KArgs &a, const Plan &pl, int grid, int sms, bool skip_isl,
                                  cudaEvent_t const *ev, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    const int64_t tiles = std::max<int64_t>(1, pl.max_tiles);
    e = pl.halo_free             ? launch_count<TW, 2, true, ROWS>(a, pl, grid, sms, tiles, s)
        : pl.count_ns == 3       ? launch_count<TW, 3, false, ROWS>(a, pl, grid, sms, tiles, s)
                                 : launch_count<TW, 2, false, ROWS>(a, pl, grid, sms, tiles, s);
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[2], s)) != cudaSuccess) return e;
    const int scan_blocks = (int)((tiles + kScanChunk - 1) / kScanChunk);
    e = pl.halo_free ? launch_pdl(daq_scan_kernel<TW, true>, scan_blocks, kScanThreads, 0, s, a)
                     : launch_pdl(daq_scan_kernel<TW, false>, scan_blocks, kScanThreads, 0, s, a);
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return e;
    if (!skip_isl) {
        e = (a.flags & DAQ_SPARSE) ? launch_compact<TW, true, ROWS>(a, pl, grid, sms, tiles, s)
                                   : launch_compact<TW, false, ROWS>(a, pl, grid, sms, tiles, s);
        if (e != cudaSuccess) return e;
    }
    if (ev && (e = cudaEventRecord(ev[4], s)) != cudaSuccess) return e;
    return cudaSuccess;
}

// Every tile width of the two-pass form, loaded by row copies (a.use_tma ==
// kLoadRows) or not.
cudaError_t launch_twopass_rows(const KArgs &a, const Plan &pl, int grid, int sms, bool skip_isl, cudaEvent_t const *ev,
                                cudaStream_t s);

template <bool ROWS>
static cudaError_t launch_twopass_any(const KArgs &a, const Plan &pl, int grid, int sms, bool skip_isl,
                                      cudaEvent_t const *ev, cudaStream_t s)
{
    switch (pl.tw) {
    case 128: return launch_twopass<128, ROWS>(a, pl, grid, sms, skip_isl, ev, s);
    case 224: return launch_twopass<224, ROWS>(a, pl, grid, sms, skip_isl, ev, s);
    case 384: return launch_twopass<384, ROWS>(a, pl, grid, sms, skip_isl, ev, s);
    default: return launch_twopass<448, ROWS>(a, pl, grid, sms, skip_isl, ev, s);
    }
}

}  // namespace daq
