// Elementwise latent updates of the region steps: decayed cached velocity with
// the Euler update of the edited tokens (Sec. 4, case equation of the AVDCache;
// Sec. 3, Euler sampler equation) and the merge with one-step-predicted
// unedited tokens (one-step estimation equation; Algorithm 1).
//
// Both are HBM-bound: one thread owns 8 channels (one 128-bit access per
// tensor), fp32 math, bf16 round-to-nearest-even on the way out.
#include "common.cuh"

namespace regione {

constexpr int kLatThreads = 256;

// x_e <- x_e - dt * (scale * v_in), n_steps times with the steps' own dt and scale and the rounding to bf16
// between them; optionally v_cache_out <- v_in.  One thread = 8 channels.  A launch of 1 to 2 us bounds the small
// latents of a sampler loop, so the steps that reuse a velocity ride with the step that computed it.
__global__ void __launch_bounds__(kLatThreads)
velocity_decay_kernel(const uint4* __restrict__ v_in, const __grid_constant__ PerRequestF neg_dt_scale, int n_steps, int b0,
                      uint4* __restrict__ x_e, uint4* __restrict__ v_cache_out,
                      const int32_t* __restrict__ n_edit, int Ne_cap, int cpr, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = b0 + blockIdx.y;                       // requests b0 .. b0 + gridDim.y of the batch
    const float* a = neg_dt_scale.v + blockIdx.y * n_steps;
    if (a[0] != a[0]) return;                            // NaN: this request sits the call out
    int ne = n_edit[b];
    if (ne < 0 || ne > Ne_cap) {
        if (threadIdx.x == 0 && blockIdx.x == 0) record_status(dev_status, REGIONE_DEV_BOUNDS);
        ne = max(0, min(ne, Ne_cap));
    }
    const unsigned live = (unsigned)ne * (unsigned)cpr;
    const unsigned e = blockIdx.x * (unsigned)kLatThreads + threadIdx.x;
    if (e >= live) return;
    const size_t off = (size_t)b * Ne_cap * cpr + e;
    const uint4 v = ld_stream128(v_in + off);
    uint4 x = x_e[off];
    for (int i = 0; i < n_steps; ++i) x = axpy8(x, v, a[i]);
    x_e[off] = x;
    if (v_cache_out != nullptr) v_cache_out[off] = v;
}

// x_out[n] = slot[n] >= 0 ? x_e[slot[n]] : x_full[n] - dt * v_last[n].  One thread = kMergeUnroll
// chunks of 8 channels, blockDim apart; all slots are read first, then every data load is issued
// before the first store, so several independent loads per thread are in flight.
constexpr int kMergeUnroll = 4;

__global__ void __launch_bounds__(kLatThreads)
merge_kernel(const uint4* x_full, const uint4* __restrict__ v_last,
             const uint4* __restrict__ x_e, const int32_t* __restrict__ slot,
             const PerRequestF neg_dt_v, int b0, int N, int Ne_cap, int cpr, uint4* x_out,
             int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = b0 + blockIdx.y;
    const float neg_dt = neg_dt_v.v[blockIdx.y];
    if (neg_dt != neg_dt) return;                        // NaN: this request sits the call out
    const unsigned total = (unsigned)N * (unsigned)cpr;
    const unsigned base = blockIdx.x * (unsigned)(kLatThreads * kMergeUnroll) + threadIdx.x;
    const size_t req = (size_t)b * N * cpr;
    int s[kMergeUnroll];
    unsigned c[kMergeUnroll];
#pragma unroll
    for (int u = 0; u < kMergeUnroll; ++u) {
        const unsigned e = base + (unsigned)u * kLatThreads;
        s[u] = -2;                                   // -2: past the end, nothing to do
        if (e < total) {
            const unsigned n = e / (unsigned)cpr;
            c[u] = e - n * (unsigned)cpr;
            const int sv = slot[(size_t)b * N + n];
            s[u] = sv < 0 ? -1 : sv;                 // any negative slot means "unedited"
            if (s[u] >= Ne_cap) {
                record_status(dev_status, REGIONE_DEV_BOUNDS);
                s[u] = -2;
            }
        }
    }
    uint4 x[kMergeUnroll], v[kMergeUnroll];
#pragma unroll
    for (int u = 0; u < kMergeUnroll; ++u) {
        const size_t off = req + base + (size_t)u * kLatThreads;
        if (s[u] >= 0) {
            x[u] = ldg128(x_e + ((size_t)b * Ne_cap + s[u]) * cpr + c[u]);
        } else if (s[u] == -1) {
            x[u] = x_full[off];
            v[u] = ld_stream128(v_last + off);
        }
    }
#pragma unroll
    for (int u = 0; u < kMergeUnroll; ++u) {
        const size_t off = req + base + (size_t)u * kLatThreads;
        if (s[u] >= 0) x_out[off] = x[u];
        else if (s[u] == -1) x_out[off] = axpy8(x[u], v[u], neg_dt);
    }
}

// The sampler loop's updates of all tokens, each with what the loop does next to the same rows: a launch of these sizes is
// 1 to 3 us of memory round trips and 6 us of host time (28 steps of 4096 tokens: 29 launches -> 22, 237 -> 203 us with the host
// side).  The velocity may lie in the rows that the first half writes, not in those of the second: see loop.py.
//
// x <- x - dt * v and v_last <- v; where a run of region steps begins (slot != nullptr), the edited tokens to X^E as well.
__global__ void __launch_bounds__(kLatThreads)
loop_full_kernel(const uint4* __restrict__ v_in, const __grid_constant__ PerRequestF neg_dt_v, int b0, uint4* __restrict__ x,
                 uint4* __restrict__ v_last, const int32_t* __restrict__ slot, uint4* __restrict__ x_e, int N, int cpr,
                 int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = b0 + blockIdx.y;
    const float neg_dt = neg_dt_v.v[blockIdx.y];
    const unsigned e = blockIdx.x * (unsigned)kLatThreads + threadIdx.x;
    if (neg_dt != neg_dt || e >= (unsigned)N * (unsigned)cpr) return;    // NaN: this request sits the call out
    const size_t req = (size_t)b * N * cpr;
    const unsigned n = e / (unsigned)cpr;
    const int s = slot != nullptr ? slot[(size_t)b * N + n] : -1;
    const uint4 v = ld_stream128(v_in + req + e);
    const uint4 y = axpy8(x[req + e], v, neg_dt);
    x[req + e] = y;
    v_last[req + e] = v;
    if (s >= N) record_status(dev_status, REGIONE_DEV_BOUNDS);
    else if (s >= 0) x_e[req + (size_t)s * cpr + (e - n * (unsigned)cpr)] = y;
}

// The last update of a run of region steps and the merge behind it: velocity_decay_kernel on the edited tokens, whose
// new rows go to their places in x, and one step of v_last for the others.
__global__ void __launch_bounds__(kLatThreads)
loop_region_end_kernel(const uint4* v_in, const __grid_constant__ PerRequestF neg_dt_scale, int n_steps,
                       const __grid_constant__ PerRequestF neg_dt_u, int b0, uint4* __restrict__ x_e, uint4* v_cache_out,
                       const int32_t* __restrict__ n_edit, const int32_t* __restrict__ slot, const uint4* __restrict__ v_last,
                       uint4* __restrict__ x, int N, int cpr, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    const int b = b0 + blockIdx.y;
    const unsigned e = blockIdx.x * (unsigned)kLatThreads + threadIdx.x;
    if (e >= (unsigned)N * (unsigned)cpr) return;
    const float* a = neg_dt_scale.v + blockIdx.y * n_steps;
    const float u = neg_dt_u.v[blockIdx.y];
    int ne = n_edit[b];
    if (ne < 0 || ne > N) {
        if (e == 0) record_status(dev_status, REGIONE_DEV_BOUNDS);
        ne = max(0, min(ne, N));
    }
    const size_t req = (size_t)b * N * cpr;
    const unsigned n = e / (unsigned)cpr;
    const int s = slot[(size_t)b * N + n];
    if (s < 0) {
        if (u == u) x[req + e] = axpy8(x[req + e], ld_stream128(v_last + req + e), u);      // NaN: no merge
        return;
    }
    if (s >= N) {
        record_status(dev_status, REGIONE_DEV_BOUNDS);
        return;
    }
    const size_t at = req + (size_t)s * cpr + (e - n * (unsigned)cpr);
    uint4 y = x_e[at];
    if (s < ne && a[0] == a[0]) {                            // (NaN: no update)
        const uint4 v = v_in[at];
        for (int i = 0; i < n_steps; ++i) y = axpy8(y, v, a[i]);
        x_e[at] = y;
        if (v_cache_out != nullptr) v_cache_out[at] = v;
    }
    if (u == u) x[req + e] = y;
}

static bool loop_plan_ok(const regione_loop_plan* p, int* rc) {
    *rc = REGIONE_INVALID_ARG;
    if (!p || !p->x || !p->x_e || !p->v_last || !p->v_cache || !p->slot || !p->n_edit || p->B < 0 || p->N < 1 || p->C < 1) return false;
    if (!aligned16(p->x) || !aligned16(p->x_e) || !aligned16(p->v_last) || !aligned16(p->v_cache)) return false;
    *rc = REGIONE_UNSUPPORTED;
    if ((p->C & 7) != 0 || p->B > 65535 || (long long)p->N * (p->C / 8) + kLatThreads >= 0x7fffffffLL) return false;
    *rc = REGIONE_OK;
    return true;
}

}  // namespace regione

using namespace regione;

extern "C" int regione_loop_full_step(const regione_loop_plan* p, const regione_bf16* v, const float* dt, int starts_run,
                                      void* stream) {
    int rc;
    if (!loop_plan_ok(p, &rc)) return rc;
    if (!v || !dt || !aligned16(v)) return REGIONE_INVALID_ARG;
    const int cpr = p->C / 8;
    const unsigned blocks = ((unsigned)p->N * cpr + kLatThreads - 1) / kLatThreads;
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < p->B && e == cudaSuccess; b0 += kReqChunk) {
        const int nb = p->B - b0 < kReqChunk ? p->B - b0 : kReqChunk;
        PerRequestF a;
        for (int i = 0; i < nb; ++i) a.v[i] = -dt[b0 + i];
        e = launch_overlapped(loop_full_kernel, dim3(blocks, nb), dim3(kLatThreads), 0, (cudaStream_t)stream, (const uint4*)v, a, b0,
                              (uint4*)p->x, (uint4*)p->v_last, starts_run ? p->slot : nullptr, (uint4*)p->x_e, p->N, cpr,
                              p->dev_status);
    }
    return launch_status(e);
}

extern "C" int regione_loop_region_steps(const regione_loop_plan* p, const regione_bf16* v_e, const float* scale, const float* dt,
                                         int n_steps, const float* dt_unedited, void* stream) {
    int rc;
    if (!loop_plan_ok(p, &rc)) return rc;
    if (!scale || !dt || n_steps < 1 || n_steps > kReqChunk || !aligned16(v_e)) return REGIONE_INVALID_ARG;
    // (no velocity: the kept one)
    uint16_t* const keep = v_e != nullptr ? p->v_cache : nullptr;
    const uint16_t* const v = v_e != nullptr ? v_e : p->v_cache;
    if (dt_unedited == nullptr)
        return regione_velocity_decay_run(v, scale, dt, n_steps, p->x_e, keep, p->n_edit, p->B, p->N, p->C, p->dev_status, stream);
    const int cpr = p->C / 8;
    const unsigned blocks = ((unsigned)p->N * cpr + kLatThreads - 1) / kLatThreads;
    const int chunk = kReqChunk / n_steps;   // a launch carries kReqChunk scalars
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < p->B && e == cudaSuccess; b0 += chunk) {
        const int nb = p->B - b0 < chunk ? p->B - b0 : chunk;
        PerRequestF a, u;                    // x - (dt * scale) * v, the product formed in fp32 first
        for (int i = 0; i < nb; ++i) {
            u.v[i] = -dt_unedited[b0 + i];
            for (int k = 0; k < n_steps; ++k) {
                const size_t at = (size_t)k * p->B + b0 + i;
                a.v[i * n_steps + k] = -(dt[at] * scale[at]);
            }
        }
        e = launch_overlapped(loop_region_end_kernel, dim3(blocks, nb), dim3(kLatThreads), 0, (cudaStream_t)stream, (const uint4*)v, a,
                              n_steps, u, b0, (uint4*)p->x_e, (uint4*)keep, p->n_edit, p->slot, (const uint4*)p->v_last,
                              (uint4*)p->x, p->N, cpr, p->dev_status);
    }
    return launch_status(e);
}

extern "C" int regione_velocity_decay(const regione_bf16* v_in, const float* scale, const float* dt,
                                      regione_bf16* x_e, regione_bf16* v_cache_out,
                                      const int32_t* n_edit, int B, int Ne_cap, int C,
                                      int32_t* dev_status, void* stream) {
    return regione_velocity_decay_run(v_in, scale, dt, 1, x_e, v_cache_out, n_edit, B, Ne_cap, C, dev_status, stream);
}

extern "C" int regione_velocity_decay_run(const regione_bf16* v_in, const float* scale, const float* dt, int n_steps,
                                          regione_bf16* x_e, regione_bf16* v_cache_out, const int32_t* n_edit, int B,
                                          int Ne_cap, int C, int32_t* dev_status, void* stream) {
    if (!v_in || !x_e || !n_edit || !scale || !dt) return REGIONE_INVALID_ARG;
    if (B < 0 || Ne_cap < 0 || C < 1 || n_steps < 1 || n_steps > kReqChunk) return REGIONE_INVALID_ARG;
    if (!aligned16(v_in) || !aligned16(x_e) || !aligned16(v_cache_out)) return REGIONE_INVALID_ARG;
    if ((C & 7) != 0 || B > 65535) return REGIONE_UNSUPPORTED;
    const long long cpr = C / 8, total = (long long)Ne_cap * cpr;
    if (total + kLatThreads >= 0x7fffffffLL) return REGIONE_UNSUPPORTED;
    if (B == 0 || Ne_cap == 0) return REGIONE_OK;
    cudaError_t e = cudaSuccess;
    const int chunk = kReqChunk / n_steps;   // a launch carries kReqChunk scalars
    for (int b0 = 0; b0 < B && e == cudaSuccess; b0 += chunk) {
        const int nb = B - b0 < chunk ? B - b0 : chunk;
        PerRequestF a;                       // x - (dt * scale) * v, the product formed in fp32 first
        for (int i = 0; i < nb; ++i)
            for (int k = 0; k < n_steps; ++k) {
                const size_t at = (size_t)k * B + b0 + i;
                a.v[i * n_steps + k] = -(dt[at] * scale[at]);
            }
        dim3 grid((unsigned)((total + kLatThreads - 1) / kLatThreads), nb);
        e = launch_overlapped(velocity_decay_kernel, grid, dim3(kLatThreads), 0, (cudaStream_t)stream,
                              (const uint4*)v_in, a, n_steps, b0, (uint4*)x_e, (uint4*)v_cache_out, n_edit,
                              Ne_cap, (int)cpr, dev_status);
    }
    return launch_status(e);
}

extern "C" int regione_merge(const regione_bf16* x_full, const regione_bf16* v_last_full,
                             const regione_bf16* x_e, const int32_t* slot, const float* dt_unedited, int B,
                             int N, int Ne_cap, int C, regione_bf16* x_out, int32_t* dev_status,
                             void* stream) {
    if (!x_full || !v_last_full || !slot || !x_out || !dt_unedited) return REGIONE_INVALID_ARG;
    if (B < 0 || N < 1 || Ne_cap < 0 || C < 1) return REGIONE_INVALID_ARG;
    if (Ne_cap > 0 && !x_e) return REGIONE_INVALID_ARG;
    if (!aligned16(x_full) || !aligned16(v_last_full) || !aligned16(x_e) || !aligned16(x_out))
        return REGIONE_INVALID_ARG;
    if ((C & 7) != 0 || B > 65535) return REGIONE_UNSUPPORTED;
    const long long cpr = C / 8, total = (long long)N * cpr;
    if (total + kLatThreads >= 0x7fffffffLL) return REGIONE_UNSUPPORTED;
    if (B == 0) return REGIONE_OK;
    const long long per_block = (long long)kLatThreads * kMergeUnroll;
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < B && e == cudaSuccess; b0 += kReqChunk) {
        const int nb = B - b0 < kReqChunk ? B - b0 : kReqChunk;
        PerRequestF a;
        for (int i = 0; i < nb; ++i) a.v[i] = -dt_unedited[b0 + i];
        dim3 grid((unsigned)((total + per_block - 1) / per_block), nb);
        e = launch_overlapped(merge_kernel, grid, dim3(kLatThreads), 0, (cudaStream_t)stream,
                              (const uint4*)x_full, (const uint4*)v_last_full, (const uint4*)x_e, slot, a,
                              b0, N, Ne_cap, (int)cpr, (uint4*)x_out, dev_status);
    }
    return launch_status(e);
}
