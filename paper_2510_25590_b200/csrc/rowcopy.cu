// Indexed row copies: token gather / scatter (Algorithm 1: X[E_index] and the
// re-gathering by spatial position) and the Region-Instruction KV cache store
// (Sec. 4 "Stabilization Stage": K and V of every attention layer are saved).
// All three are pure HBM traffic.
#include "rowcopy.cuh"

namespace regione {

// blockIdx.z picks the tensor pair.
template <bool GATHER>
__global__ void __launch_bounds__(kCopyThreads)
row_copy_kernel(const __grid_constant__ RowCopyPairs pairs, const int32_t* __restrict__ idx,
                const int32_t* __restrict__ n, long long idx_rows, long long idx_stride,
                long long cap, int cpr, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    copy_rows<GATHER>(pairs.p[blockIdx.z], blockIdx.y, blockIdx.x, idx, n, idx_rows, idx_stride, cap, cpr, dev_status);
}

template <bool GATHER>
static int launch_row_copy(const RowCopyPairs& ps, int pairs, const int32_t* idx,
                           const int32_t* n, int B, long long idx_rows, long long idx_stride,
                           long long cap, long long row_bytes, int32_t* dev_status, void* stream) {
    const long long cpr = row_bytes / 16;
    const long long per_block = (long long)kCopyThreads * kUnroll;
    const long long blocks = (cap * cpr + per_block - 1) / per_block;
    if (cap * cpr + per_block >= 0x7fffffffLL) return REGIONE_UNSUPPORTED;
    dim3 grid((unsigned)blocks, (unsigned)B, (unsigned)pairs);
    return launch_status(launch_overlapped(row_copy_kernel<GATHER>, grid, dim3(kCopyThreads), 0,
                                           (cudaStream_t)stream, ps, idx, n, idx_rows, idx_stride,
                                           cap, (int)cpr, dev_status));
}

}  // namespace regione

using namespace regione;

static int check_rows(const void* src, const void* idx, const void* n, const void* dst, int B,
                      int64_t a, int64_t stride, int64_t c, int64_t row_bytes) {
    if (!src || !idx || !n || !dst) return REGIONE_INVALID_ARG;
    if (B < 0 || a < 0 || c < 0 || stride < 0 || row_bytes <= 0) return REGIONE_INVALID_ARG;
    if (!aligned16(src) || !aligned16(dst)) return REGIONE_INVALID_ARG;
    if (row_bytes % 16 != 0 || B > 65535) return REGIONE_UNSUPPORTED;
    return REGIONE_OK;
}

extern "C" int regione_gather(const void* src, const int32_t* idx, const int32_t* n, int B,
                              int64_t src_rows, int64_t idx_stride, int64_t dst_rows_cap,
                              int64_t row_bytes, void* dst, int32_t* dev_status, void* stream) {
    int s = check_rows(src, idx, n, dst, B, src_rows, idx_stride, dst_rows_cap, row_bytes);
    if (s != REGIONE_OK) return s;
    if (idx_stride < dst_rows_cap) return REGIONE_INVALID_ARG;
    if (B == 0 || dst_rows_cap == 0) return REGIONE_OK;
    RowCopyPairs ps = {};
    ps.p[0] = RowCopyPair{(const uint4*)src, (uint4*)dst};
    return launch_row_copy<true>(ps, 1, idx, n, B, src_rows, idx_stride, dst_rows_cap, row_bytes,
                                 dev_status, stream);
}

extern "C" int regione_scatter(const void* src, const int32_t* idx, const int32_t* n, int B,
                               int64_t src_rows_cap, int64_t idx_stride, int64_t dst_rows,
                               int64_t row_bytes, void* dst, int32_t* dev_status, void* stream) {
    int s = check_rows(src, idx, n, dst, B, dst_rows, idx_stride, src_rows_cap, row_bytes);
    if (s != REGIONE_OK) return s;
    if (idx_stride < src_rows_cap) return REGIONE_INVALID_ARG;
    if (B == 0 || src_rows_cap == 0) return REGIONE_OK;
    RowCopyPairs ps = {};
    ps.p[0] = RowCopyPair{(const uint4*)src, (uint4*)dst};
    return launch_row_copy<false>(ps, 1, idx, n, B, dst_rows, idx_stride, src_rows_cap, row_bytes,
                                  dev_status, stream);
}

extern "C" int regione_rikv_store(const regione_bf16* k_full, const regione_bf16* v_full,
                                  const int32_t* keep_rows, const int32_t* n_keep, int B,
                                  int N_full, int Nc_cap, int H, int D, regione_bf16* k_cache,
                                  regione_bf16* v_cache, int32_t* dev_status, void* stream) {
    if (!k_full || !v_full || !keep_rows || !n_keep || !k_cache || !v_cache)
        return REGIONE_INVALID_ARG;
    if (B < 0 || N_full < 0 || Nc_cap < 0 || H < 1 || D < 1) return REGIONE_INVALID_ARG;
    if (!aligned16(k_full) || !aligned16(v_full) || !aligned16(k_cache) || !aligned16(v_cache))
        return REGIONE_INVALID_ARG;
    const long long row_bytes = (long long)H * D * 2;
    if (row_bytes % 16 != 0 || B > 65535) return REGIONE_UNSUPPORTED;
    if (B == 0 || Nc_cap == 0) return REGIONE_OK;
    RowCopyPairs ps = {};
    ps.p[0] = RowCopyPair{(const uint4*)k_full, (uint4*)k_cache};
    ps.p[1] = RowCopyPair{(const uint4*)v_full, (uint4*)v_cache};
    return launch_row_copy<true>(ps, 2, keep_rows, n_keep, B, N_full, Nc_cap, Nc_cap, row_bytes,
                                 dev_status, stream);
}

extern "C" int regione_gather_multi(const void* const* srcs, void* const* dsts, int n_tensors,
                                    const int32_t* idx, const int32_t* n, int B, int64_t src_rows,
                                    int64_t idx_stride, int64_t dst_rows_cap, int64_t row_bytes,
                                    int32_t* dev_status, void* stream) {
    if (!srcs || !dsts || n_tensors < 1 || n_tensors > kMaxPairs) return REGIONE_INVALID_ARG;
    RowCopyPairs ps = {};
    for (int i = 0; i < n_tensors; ++i) {
        int s = check_rows(srcs[i], idx, n, dsts[i], B, src_rows, idx_stride, dst_rows_cap, row_bytes);
        if (s != REGIONE_OK) return s;
        ps.p[i] = RowCopyPair{(const uint4*)srcs[i], (uint4*)dsts[i]};
    }
    if (idx_stride < dst_rows_cap) return REGIONE_INVALID_ARG;
    if (B == 0 || dst_rows_cap == 0) return REGIONE_OK;
    return launch_row_copy<true>(ps, n_tensors, idx, n, B, src_rows, idx_stride, dst_rows_cap, row_bytes,
                                 dev_status, stream);
}
