// Indexed row copies (device side), shared by the gather / scatter / cache-store kernel and by the
// kernel that moves everything a region step moves between its partition and its attention.
//
// Rows are byte strings whose length is a multiple of 16; a thread moves kUnroll 16-byte chunks that
// are blockDim apart, so a warp always touches 512 contiguous bytes per request, all loads of a thread
// are issued before its first store, and source data (read once) bypasses L1.
#pragma once

#include "common.cuh"

namespace regione {

constexpr int kCopyThreads = 256;
constexpr int kUnroll = 8;

struct RowCopyPair {
    const uint4* src;
    uint4* dst;
};

constexpr int kMaxPairs = 4;                 // tensors sharing one index list in one launch
struct RowCopyPairs {
    RowCopyPair p[kMaxPairs];
};

// GATHER: dst[b, j] = src[b, idx[b, j]];  !GATHER: dst[b, idx[b, j]] = src[b, j].
// `idx_rows` bounds the indexed side, `cap` the dense side; `block` = place among the blocks of request b.
template <bool GATHER>
__device__ __forceinline__ void copy_rows(const RowCopyPair p, int b, unsigned block, const int32_t* __restrict__ idx,
                                          const int32_t* __restrict__ n, long long idx_rows, long long idx_stride,
                                          long long cap, int cpr, int32_t* dev_status) {
    long long live = n[b];
    if (live < 0 || live > cap) {
        if (threadIdx.x == 0 && block == 0) record_status(dev_status, REGIONE_DEV_BOUNDS);
        live = live < 0 ? 0 : cap;
    }
    // 32-bit chunk arithmetic: the host guarantees cap * cpr < 2^31.
    const unsigned total = (unsigned)live * (unsigned)cpr;
    const unsigned base = block * (unsigned)(kCopyThreads * kUnroll) + threadIdx.x;
    if (base >= total) return;
    const uint4* __restrict__ src = p.src + (size_t)b * (GATHER ? idx_rows : cap) * cpr;
    uint4* __restrict__ dst = p.dst + (size_t)b * (GATHER ? cap : idx_rows) * cpr;
    const int32_t* __restrict__ my_idx = idx + (size_t)b * idx_stride;

    // (row j, chunk c) of the first element; later elements advance by kCopyThreads chunks.
    unsigned j = base / (unsigned)cpr;
    unsigned c = base - j * (unsigned)cpr;
    const unsigned step_rows = (unsigned)kCopyThreads / (unsigned)cpr;
    const unsigned step_chunks = (unsigned)kCopyThreads - step_rows * (unsigned)cpr;

    // All indexes first, then all rows: two round trips for the block instead of one per chunk (with the partition's
    // own trips cut, a region step of 1024 tokens 25.8 -> 24.1 us, of 4096 with 205 queries 56.6 -> 53.9).
    unsigned row[kUnroll], chunk[kUnroll];
    int at[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
        row[u] = j;
        chunk[u] = c;
        at[u] = base + (unsigned)u * kCopyThreads < total ? my_idx[j] : -1;
        j += step_rows;
        c += step_chunks;
        if (c >= (unsigned)cpr) { c -= (unsigned)cpr; ++j; }
    }
    uint4 val[kUnroll];
    bool bad = false;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
        if (at[u] >= 0 && at[u] < idx_rows) {
            val[u] = ld_stream128(src + ((GATHER ? (long long)at[u] : (long long)row[u]) * cpr + chunk[u]));
        } else {
            bad |= base + (unsigned)u * kCopyThreads < total;
            at[u] = -1;
        }
    }
    if (bad) record_status(dev_status, REGIONE_DEV_BOUNDS);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
        if (at[u] >= 0) dst[(GATHER ? (long long)row[u] : (long long)at[u]) * cpr + chunk[u]] = val[u];
}

}  // namespace regione
