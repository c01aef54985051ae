// One region-aware step of one attention layer as a sequence of three or four launches (Algorithm 1, one iteration of
// the region loop for one layer):
//   1 partition with the joint-sequence row lists
//   2 everything that moves rows between the partition and the attention: the latent update and the gathers
//   3 region attention, its rows written at their joint-sequence positions; in a step that refreshes the
//     cache the copies to the cache travel in the same launch
//   4 merge of the items that the attention cut, where it does not do that itself
//
// Why one launch for all the moves: the kernels it replaces (gather of X^E and v, velocity decay, merge, gather
// of Q / K / V) take 2 to 5 us each, most of it launch and one memory round trip, and had two streams to be forked
// and joined.  Why the cache store rides with the attention: the rows of a step that refreshes the cache from its own
// K and V are, fresh and cached together, all rows of K and V, so the attention reads those directly and nothing
// waits for the cache.  Measured, one pass among others with its host work (seven calls on two streams -> one call):
//   256 of 1024 tokens, 4 heads x 64, cache refreshed       108 -> 24 us
//   205 of 4096 tokens, 24 heads x 128, cache read           95 -> 54 us
//   819 of 4096 tokens, 24 heads x 128, cache read          135 -> 128 us (power-capped attention)
//   2048 of 4096 tokens, 24 heads x 128, cache refreshed    281 -> 246 us (power-capped attention)
#include "rowcopy.cuh"

namespace regione {

// Whether the attention of a step that refreshes the cache reads K and V where they are and takes the rows of the
// cache along, or reads [cache | fresh] as a step that keeps the cache does, with the rows copied ahead of it.  The
// copies need the attention's time to hide behind, which grows with the queries.  Measured, a whole step with the rows
// copied ahead -> along, us: 8704 rows of 24 heads, 128 queries 81 -> 83, 256 89 -> 90, 512 104 -> 93, 819 143 -> 132, 1536
// 168 -> 143; four requests of 18944, 512 queries 758 -> 612, 1382 1537 -> 1274.  The line lies above the point where
// the two meet: it is where the other order of the keys moves single elements of the scattered buffer by 0.05 of its
// rms, not by 0.1 as below (see keeps_cuts: a difference between two roundings, not an error of either).
static bool takes_rows_along(int q_cap, int n_full) { return 16LL * (q_cap - 64) >= n_full; }

constexpr int kApartBlocks = 64;      // blocks of a request that copy rows only where rows_apart says so

struct LatentMove {
    const uint4 *x, *v;             // [B, N, C] current latent and velocity
    const int32_t* slot;            // [B, N] place of an edited token in X^E, negative: unedited
    const int32_t* n_edit;          // [B]
    uint4 *x_e, *v_e, *v_avd;       // [B, Ne_cap, C] X^E after the Euler step, v^E, the kept velocity
    uint4* x_out;                   // [B, N, C]
    int N, Ne_cap, cpr;             // 16-byte chunks per token
};

// Gather of X^E and v^E, decayed velocity + Euler update, and merge with the one-step-predicted unedited tokens:
// each token is read once and all that follows from it written.  A thread owns 8 channels of one token.
__device__ __forceinline__ void move_latents(const LatentMove& a, int b, unsigned block, float neg_dt_scale, float neg_dt_u,
                                             int32_t* dev_status) {
    const unsigned e = block * blockDim.x + threadIdx.x;
    int ne = a.n_edit[b];
    if (ne < 0 || ne > a.Ne_cap) {
        if (e == 0) record_status(dev_status, REGIONE_DEV_BOUNDS);
        ne = max(0, min(ne, a.Ne_cap));
    }
    if (e >= (unsigned)a.N * (unsigned)a.cpr) return;
    const unsigned n = e / (unsigned)a.cpr, c = e - n * (unsigned)a.cpr;
    const size_t at = (size_t)b * a.N * a.cpr + e;
    const int s = a.slot[(size_t)b * a.N + n];
    const uint4 x = ldg128(a.x + at), v = ldg128(a.v + at);
    const bool merge = neg_dt_u == neg_dt_u;                      // NaN: the request sits that operation out
    if (s < 0) {
        if (merge) a.x_out[at] = axpy8(x, v, neg_dt_u);
        return;
    }
    if (s >= a.Ne_cap) {
        if (merge) record_status(dev_status, REGIONE_DEV_BOUNDS);
        return;
    }
    const size_t es = ((size_t)b * a.Ne_cap + s) * a.cpr + c;
    uint4 y = x;
    if (s < ne) {
        a.v_e[es] = v;
        if (neg_dt_scale == neg_dt_scale) {
            y = axpy8(x, v, neg_dt_scale);
            a.v_avd[es] = v;
        }
        a.x_e[es] = y;
    } else {
        y = a.x_e[es];                                            // (lists of an earlier, shorter partition)
    }
    if (merge) a.x_out[at] = y;
}

// blockIdx.x: blocks of the latent update, then of each of the n_pairs tensors whose recomputed rows are gathered, then
// of K and V of the rows that go to the cache; blockIdx.y = request of this launch.  Where the attention reads K and V
// in place (along), only the queries are gathered for certain: a request whose lists do not name all rows needs its
// other rows as well (rows_apart), which is rare, so that a few blocks stride over them.
// Bound by launch and one or two memory round trips at the sizes of the paper's editors (4 to 5 us); the row gathers
// run at the bandwidth of HBM where they are large, and the latent blocks, which come first, hide behind them.
__global__ void __launch_bounds__(kCopyThreads)
region_step_move_kernel(const LatentMove lat, const __grid_constant__ PerRequestF neg_dt_scale,
                        const __grid_constant__ PerRequestF neg_dt_u, int b0, int lat_blocks,
                        const __grid_constant__ RowCopyPairs rows, int n_pairs, int row_blocks,
                        const int32_t* __restrict__ query_rows, const int32_t* __restrict__ n_q, int n_full, int q_cap,
                        int row_cpr, const __grid_constant__ RowCopyPairs kept, int kept_blocks, bool along, int tail_blocks,
                        const int32_t* __restrict__ cache_rows, const int32_t* __restrict__ n_cache, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = b0 + blockIdx.y;
    const int blk = blockIdx.x;
    if (blk < lat_blocks) {
        move_latents(lat, b, blk, neg_dt_scale.v[blockIdx.y], neg_dt_u.v[blockIdx.y], dev_status);
        return;
    }
    int at = blk - lat_blocks;
    if (at < n_pairs * row_blocks) {
        const int pair = at / row_blocks;
        copy_rows<true>(rows.p[pair], b, at - pair * row_blocks, query_rows, n_q, n_full, q_cap, q_cap, row_cpr, dev_status);
        return;
    }
    at -= n_pairs * row_blocks;
    if (along && !rows_apart(n_q[b], n_cache[b], q_cap, n_full)) return;
    const int fresh = along ? 2 * row_blocks : 0;              // K and V, pairs 1 and 2 of `rows`
    for (; at < fresh + 2 * kept_blocks; at += tail_blocks) {
        const int pair = at < fresh ? at / row_blocks : (at - fresh) / kept_blocks;
        if (at < fresh)
            copy_rows<true>(rows.p[1 + pair], b, at - pair * row_blocks, query_rows, n_q, n_full, q_cap, q_cap, row_cpr,
                            dev_status);
        else
            copy_rows<true>(kept.p[pair], b, at - fresh - pair * kept_blocks, cache_rows, n_cache, n_full, n_full, n_full,
                            row_cpr, dev_status);
    }
}

}  // namespace regione

using namespace regione;

extern "C" size_t regione_region_step_workspace(const regione_step_plan* p) {
    if (!p) return 0;
    const int q_cap = p->ne_cap + (p->membership == REGIONE_ROWS_PAPER ? p->n_text : 0);
    const int n_full = p->n_text + p->N + p->n_ref;
    const size_t a = regione_region_attention_workspace(p->B, q_cap, q_cap, n_full, p->H, p->D);
    const size_t s = regione_region_attention_workspace(p->B, q_cap, n_full, 0, p->H, p->D);
    return a > s ? a : s;
}

extern "C" int regione_region_step(const regione_step_plan* p, const regione_bf16* x_t, const regione_bf16* v,
                                   const regione_bf16* ref, const regione_bf16* q_full, const regione_bf16* k_full,
                                   const regione_bf16* v_full, const float* t, const float* scale, const float* dt,
                                   const float* dt_unedited, int store_cache, int parts, void* stream) {
    if (!p || !x_t || !v || !ref || !q_full || !k_full || !v_full) return REGIONE_INVALID_ARG;
    if (p->B < 0 || (p->B > 0 && (!t || !scale || !dt || !dt_unedited))) return REGIONE_INVALID_ARG;
    if (!p->mask || !p->edit_idx || !p->keep_idx || !p->slot || !p->n_edit || !p->query_rows || !p->n_q || !p->cache_rows ||
        !p->n_cache || !p->n_rows || !p->x_e || !p->v_e || !p->v_avd || !p->x_out || !p->q_e || !p->k_fresh || !p->v_fresh ||
        !p->k_cache || !p->v_cache || !p->o_full)
        return REGIONE_INVALID_ARG;
    const int B = p->B, N = p->N, H = p->H, D = p->D, C = p->C;
    if (N < 1 || p->n_text < 0 || p->n_ref < 0 || p->ne_cap < 0 || H < 1 || D < 1 || C < 1) return REGIONE_INVALID_ARG;
    if (p->membership != REGIONE_ROWS_EDITED_QUERIES && p->membership != REGIONE_ROWS_PAPER) return REGIONE_INVALID_ARG;
    const void* const wide[] = {x_t, v, p->x_e, p->v_e, p->v_avd, p->x_out, q_full, k_full, v_full, p->q_e, p->k_fresh,
                                p->v_fresh, p->k_cache, p->v_cache, p->o_full};
    for (const void* a : wide)
        if (!aligned16(a)) return REGIONE_INVALID_ARG;
    if ((D != 64 && D != 128) || (C & 7) != 0 || B > 65535 || H > 65535) return REGIONE_UNSUPPORTED;
    const long long n_full_ll = (long long)p->n_text + N + p->n_ref;
    const long long q_cap_ll = (long long)p->ne_cap + (p->membership == REGIONE_ROWS_PAPER ? p->n_text : 0);
    const long long lat_chunks = (long long)N * (C / 8), row_cpr = (long long)H * D / 8;
    const long long per_block = (long long)kCopyThreads * kUnroll;
    // (the copies index the chunks of a request's rows in 32 bits; ne_cap may exceed N, so neither bounds the other)
    if (lat_chunks + kCopyThreads >= 0x7fffffffLL || (long long)p->ne_cap * (C / 8) >= 0x7fffffffLL ||
        (n_full_ll > q_cap_ll ? n_full_ll : q_cap_ll) * row_cpr + per_block >= 0x7fffffffLL)
        return REGIONE_UNSUPPORTED;
    const int n_full = (int)n_full_ll, q_cap = (int)q_cap_ll;
    if (B == 0) return REGIONE_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const bool along = store_cache && q_cap > 0 && takes_rows_along(q_cap, n_full);

    if (parts & REGIONE_STEP_MOVES) {
        const int rc = regione_partition_rows(x_t, v, ref, B, N, C, t, p->metric, p->threshold, p->mask, p->edit_idx,
                                              p->keep_idx, p->slot, p->n_edit, nullptr, p->n_text, p->n_ref, p->membership,
                                              p->query_rows, p->n_q, q_cap, p->cache_rows, p->n_cache, n_full, p->dev_status,
                                              stream);
        if (rc != REGIONE_OK) return rc;
        LatentMove lm;
        lm.x = (const uint4*)x_t; lm.v = (const uint4*)v; lm.slot = p->slot; lm.n_edit = p->n_edit;
        lm.x_e = (uint4*)p->x_e; lm.v_e = (uint4*)p->v_e; lm.v_avd = (uint4*)p->v_avd; lm.x_out = (uint4*)p->x_out;
        lm.N = N; lm.Ne_cap = p->ne_cap; lm.cpr = C / 8;
        // rows taken along: the attention reads K and V themselves, only the queries are gathered (see the kernel)
        RowCopyPairs rows = {};
        rows.p[0] = RowCopyPair{(const uint4*)q_full, (uint4*)p->q_e};
        rows.p[1] = RowCopyPair{(const uint4*)k_full, (uint4*)p->k_fresh};
        rows.p[2] = RowCopyPair{(const uint4*)v_full, (uint4*)p->v_fresh};
        const int n_pairs = q_cap == 0 ? 0 : along ? 1 : 3;
        RowCopyPairs kept = {};
        kept.p[0] = RowCopyPair{(const uint4*)k_full, (uint4*)p->k_cache};
        kept.p[1] = RowCopyPair{(const uint4*)v_full, (uint4*)p->v_cache};
        const int kept_blocks = (int)((n_full * row_cpr + per_block - 1) / per_block);
        const int lat_blocks = (int)((lat_chunks + kCopyThreads - 1) / kCopyThreads);
        const int row_blocks = (int)((q_cap * row_cpr + per_block - 1) / per_block);
        const int tail_blocks = !store_cache ? 0 : !along ? 2 * kept_blocks : kApartBlocks;
        cudaError_t e = cudaSuccess;
        for (int b0 = 0; b0 < B && e == cudaSuccess; b0 += kReqChunk) {
            const int nb = B - b0 < kReqChunk ? B - b0 : kReqChunk;
            PerRequestF a, u;
            for (int i = 0; i < nb; ++i) {
                a.v[i] = -(dt[b0 + i] * scale[b0 + i]);      // x - (dt * scale) * v, the product formed in fp32 first
                u.v[i] = -dt_unedited[b0 + i];
            }
            e = launch_overlapped(region_step_move_kernel, dim3(lat_blocks + n_pairs * row_blocks + tail_blocks, nb),
                                  dim3(kCopyThreads), 0,
                                  st, lm, a, u, b0, lat_blocks, rows, n_pairs, row_blocks > 0 ? row_blocks : 1, p->query_rows,
                                  p->n_q, n_full, q_cap, (int)row_cpr, kept, kept_blocks, along, tail_blocks, p->cache_rows,
                                  p->n_cache, p->dev_status);
        }
        if (e != cudaSuccess) return REGIONE_CUDA_ERROR;
    }
    if (parts & REGIONE_STEP_ATTENTION) {
        if (q_cap == 0) return REGIONE_OK;                    // no query can exist
        const size_t need = regione_region_step_workspace(p);
        if (need > 0 && (!p->workspace || (reinterpret_cast<uintptr_t>(p->workspace) & 255u))) return REGIONE_INVALID_ARG;
        if (p->workspace_bytes < need) return REGIONE_WORKSPACE_TOO_SMALL;
        const float sm = 1.0f / sqrtf((float)D);
        if (along) {
            CacheStore cs = {};
            cs.keep_rows = p->cache_rows; cs.n_keep = p->n_cache; cs.cap = n_full;
            cs.k_cache = p->k_cache; cs.v_cache = p->v_cache;
            cs.all_rows = n_full; cs.k_apart = p->k_fresh; cs.v_apart = p->v_fresh;
            return launch_region_attention_tc(p->q_e, k_full, v_full, nullptr, nullptr, p->n_q, p->n_q, p->n_cache, B, q_cap,
                                              n_full, 0, H, D, sm, p->o_full, p->query_rows, n_full, p->workspace,
                                              p->workspace_bytes, p->dev_status, st, &cs);
        }
        return launch_region_attention_tc(p->q_e, p->k_fresh, p->v_fresh, p->k_cache, p->v_cache, p->n_q, p->n_q, p->n_cache,
                                          B, q_cap, q_cap, n_full, H, D, sm, p->o_full, p->query_rows, n_full, p->workspace,
                                          p->workspace_bytes, p->dev_status, st, nullptr);
    }
    return REGIONE_OK;
}
