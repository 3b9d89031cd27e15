// Definitions shared by the tensor-core layout build and the tensor-core kernels.
#pragma once

#include "life_internal.cuh"

namespace life {

constexpr int SUB = 32;                  // atoms per WC segment (offset granularity of the WC streams)
constexpr int DKC = 128;                 // atoms per DSC K chunk (offset granularity of the DSC stream)
constexpr int ZW = 33;                   // row stride (floats) of a WC scatter warp's 32 x 32 Z tile
constexpr uint16_t CONT = 0x8000;        // entry continues the previous entry's (atom, row)

// Device decision state of the live-entry DSC stream.
struct SparseCtl {
    unsigned long long n_live;        // real slots with x != 0 seen by this call's gather
    unsigned long long n_live_cmp;    // that count when the compacted stream was built
    unsigned long long n_compactions; // compacted-stream rebuilds so far
    unsigned long long n_compact_calls;  // DSC calls that streamed the compacted entries
    unsigned long long n_calls;       // DSC calls that went through the decision
    uint32_t stale;                   // some slot with x != 0 lies outside L
    uint32_t mode;                    // DSC_MODE_* of the current call
    uint32_t compact_now;             // the current call rebuilds the compacted stream
    uint32_t have;                    // a compacted stream exists
    uint32_t gather_done;             // blocks of the gather finished (the last one decides)
    uint32_t since;                   // decisions since the last rebuild
    uint32_t gap;                     // decisions a rebuild for a stale live set must wait (backoff)
};

// Tensor-memory columns the FP32-storage WC needs: D's FP16 hi and lo parts for
// each 128-atom block (np/2 columns each) and three 64-column Z slots.
__host__ __device__ inline int wc32_tmem_cols(int np, int kp) { return (kp / 128) * np + 3 * 64; }

}  // namespace life
