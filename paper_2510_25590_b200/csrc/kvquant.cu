// 8-bit variant of the Region-Instruction KV cache (Sec. 4 "Stabilization Stage": K and V of every
// attention layer are kept from the last full step until the next forced one, i.e. the cache is
// resident for many steps and layers).  The paper keeps the cache in the model's own precision;
// this variant stores it as 8-bit floating point E4M3 (1 sign, 4 exponent, 3 mantissa bits, bias 7,
// largest finite value 448, no infinities) with one power-of-two scale per (row, head), which halves
// the bytes a cached layer occupies.  Before a region step's attention the cache is widened back to
// bf16 by a second kernel; because the scale is a power of two and E4M3 has 3 mantissa bits, the
// widened values are exactly the quantised ones (no second rounding), so the attention sees a cache
// whose every element is  round_to_E4M3(x / s) * s.
//
//   s = 2^k, k the smallest integer with amax / 2^k <= 448 (amax = largest magnitude of the D
//   elements of that row and head); written with frexp(amax) = m * 2^e, m in [0.5, 1):
//   k = e - 9 + (m > 0.875); k = 0 for amax = 0; k is kept >= -100.
//
// All kernels are HBM-bound row passes.
// Store: a block per row reads its count, its index and its data one after the other, and an SM has few reads in flight
// meanwhile unless the rows are long; in rings of bulk copies, one per warp, the chain is off the path.  See takes_rows for
// which of the two takes a call.
// Load: one block per kept row covers K and V of that row, a lane owns 8 consecutive elements (8 bytes of codes, 16 bytes of
// bf16); the codes of kQuantUnroll pieces are on their way before the first is widened, and are the first to leave L2.  7885
// rows of 24 x 128 and the attention behind them, one piece at a time -> three: 128.8 -> 128.0 us.
#include "common.cuh"
#include "sm100_ptx.cuh"

#include <algorithm>

namespace regione {

constexpr int kQuantThreads = 256;
constexpr int kQuantUnroll = 3;
constexpr int kRowBlocks = 8;                        // store, a block per row: blocks an SM

// Two fp32 -> two E4M3 codes (round to nearest even, saturating); `lo` lands in bits [7:0].
__device__ __forceinline__ uint32_t pack_e4m3x2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

// Two E4M3 codes -> their two values (exact: every E4M3 value is a half-precision value); the code
// in bits [7:0] comes back in `.x`.  (0x7f / 0xff, the NaN codes, are never produced by the
// saturating conversion above.)
__device__ __forceinline__ float2 unpack_e4m3x2(uint32_t codes) {
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)codes));
    float2 r;
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %2; cvt.f32.f16 %0, l; cvt.f32.f16 %1, h;}"
        : "=f"(r.x), "=f"(r.y) : "r"(h2));
    return r;
}

// k of the scale 2^k for a row-and-head maximum given as bf16 bits without their sign.  With exponent field E and seven
// mantissa bits M, frexp gives e = E - 126 and m > 0.875 where M > 96.  (A subnormal maximum ends at the floor of k as well;
// an infinite one saturates like the largest finite one, whose M is above 96.)
__device__ __forceinline__ int scale_exponent(uint32_t amax) {
    if (amax == 0) return 0;
    amax = min(amax, 0x7f7fu);
    return max((int)(amax >> 7) - 135 + ((amax & 127) > 96 ? 1 : 0), -100);
}

// n_keep[b] clamped to the capacity; an out-of-range count is recorded once per request.
__device__ __forceinline__ int live_rows(const int32_t* n_keep, int b, int Nc_cap, bool report, int32_t* dev_status) {
    const int live = n_keep[b];
    if (live >= 0 && live <= Nc_cap) return live;
    if (report) record_status(dev_status, REGIONE_DEV_BOUNDS);
    return live < 0 ? 0 : Nc_cap;
}

// ---- store, a block per row ------------------------------------------------------------------------
// A block covers K and V of its row, a lane owns 8 consecutive elements (16 bytes), the D / 8 lanes of one head sit side
// by side in a warp; whole warps walk the pieces so that every shuffle has its 32 lanes, kQuantUnroll loads are issued
// before the first is used.
template <int D>
__global__ void __launch_bounds__(kQuantThreads, kRowBlocks)
rikv_store_e4m3_rows_kernel(const uint16_t* __restrict__ k_full, const uint16_t* __restrict__ v_full,
                            const int32_t* __restrict__ keep_rows, const int32_t* __restrict__ n_keep, int N_full, int Nc_cap,
                            int H, uint8_t* __restrict__ k_q, uint8_t* __restrict__ v_q, float* __restrict__ k_scale,
                            float* __restrict__ v_scale, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    constexpr int kLanesPerHead = D / 8;                // 16 or 8: divides the warp
    const int b = blockIdx.y, j = blockIdx.x;
    if (j >= live_rows(n_keep, b, Nc_cap, threadIdx.x == 0 && j == 0, dev_status)) return;
    const int row = keep_rows[(size_t)b * Nc_cap + j];
    if (row < 0 || row >= N_full) {
        if (threadIdx.x == 0) record_status(dev_status, REGIONE_DEV_BOUNDS);
        return;
    }
    const size_t src_off = ((size_t)b * N_full + row) * H * D, dst_row = (size_t)b * Nc_cap + j;
    const int per_tensor = H * kLanesPerHead, total = 2 * per_tensor;     // 16-byte pieces of K, then of V
    for (int c0 = (threadIdx.x & ~31); c0 < total; c0 += kQuantUnroll * kQuantThreads) {
        uint4 w[kQuantUnroll];
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) {
            const int c = c0 + u * kQuantThreads + (threadIdx.x & 31);
            w[u] = make_uint4(0u, 0u, 0u, 0u);
            if (c < total)
                w[u] = ld_stream128((c >= per_tensor ? v_full : k_full) + src_off +
                                    (size_t)(c >= per_tensor ? c - per_tensor : c) * 8);
        }
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) {
            const int c = c0 + u * kQuantThreads + (threadIdx.x & 31);
            const bool live = c < total;
            const int is_v = live && c >= per_tensor, piece = c - (is_v ? per_tensor : 0);
            const float x[8] = {bf16_lo(w[u].x), bf16_hi(w[u].x), bf16_lo(w[u].y), bf16_hi(w[u].y),
                                bf16_lo(w[u].z), bf16_hi(w[u].z), bf16_lo(w[u].w), bf16_hi(w[u].w)};
            float amax = 0.f;                           // (as floats: as packed bf16 the row takes 4 % longer)
#pragma unroll
            for (int e = 0; e < 8; ++e) amax = fmaxf(amax, fabsf(x[e]));   // (a NaN element is ignored here)
#pragma unroll
            for (int d = kLanesPerHead / 2; d > 0; d >>= 1)
                amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
            const int k = scale_exponent(__float_as_uint(amax) >> 16);
            const float inv = __uint_as_float((uint32_t)(127 - k) << 23);  // 2^-k, exact
            if (!live) continue;
            uint2 q;
            q.x = pack_e4m3x2(x[0] * inv, x[1] * inv) | (pack_e4m3x2(x[2] * inv, x[3] * inv) << 16);
            q.y = pack_e4m3x2(x[4] * inv, x[5] * inv) | (pack_e4m3x2(x[6] * inv, x[7] * inv) << 16);
            __stcs(reinterpret_cast<uint2*>((is_v ? v_q : k_q) + dst_row * H * D + (size_t)piece * 8), q);
            if (piece % kLanesPerHead == 0)
                (is_v ? v_scale : k_scale)[dst_row * H + piece / kLanesPerHead] = __uint_as_float((uint32_t)(127 + k) << 23);
        }
    }
}

// ---- store, rings ----------------------------------------------------------------------------------
// Every warp works for itself: it takes pieces of rows (one tensor, as many heads as make at most 4.5 KB), each fetched by
// one bulk copy into a ring of its own of up to eight pieces, so that the chain of count, index and data is off the path of
// the arithmetic.  An SM has three blocks of four such rings: up to 216 KB of reads in flight, less where eight pieces do not
// fill a ring (48 KB with 4 heads of 64).  16 elements to a lane, three shuffles for a maximum.  Pieces of 24 heads of 128, three
// to a ring -> of 12, six to a ring: 40000 rows 140 -> 120 us, four requests of 17562 241 -> 218.
constexpr int kRingWarps = 4;
constexpr int kRingStages = 8;                       // at most
constexpr int kRingBytes = 72 * 1024;                // per block; three blocks an SM
constexpr int kRingBlocks = 3;
constexpr int kPieceBytes = 4608;
constexpr long long kRingWait = 4000000000LL;        // cycles (~2 s)

struct RingPiece {                                   // what a stage holds
    long long dst_row;
    int part;                                        // tensor * groups + group
};

__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(bar, parity))
        if (clock64() - t0 > kRingWait) return false;
    return true;
}

// Largest magnitude of the elements of two 16-byte pieces, as bf16 bits.  (A NaN element is ignored.)
__device__ __forceinline__ uint32_t max_bits(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t max_magnitude(const uint4& a, const uint4& b) {
    constexpr uint32_t kAbs = 0x7fff7fffu;
    const uint32_t m0 = max_bits(max_bits(0u, a.x & kAbs), a.y & kAbs), m1 = max_bits(max_bits(0u, a.z & kAbs), a.w & kAbs);
    const uint32_t m2 = max_bits(max_bits(0u, b.x & kAbs), b.y & kAbs), m3 = max_bits(max_bits(0u, b.z & kAbs), b.w & kAbs);
    return max_bits(max_bits(m0, m1), max_bits(m2, m3));
}

__device__ __forceinline__ uint32_t encode4(uint32_t a, uint32_t b, float inv) {
    return pack_e4m3x2(bf16_lo(a) * inv, bf16_hi(a) * inv) | (pack_e4m3x2(bf16_lo(b) * inv, bf16_hi(b) * inv) << 16);
}

// `heads` of a row to a piece, `groups` pieces to a row of one tensor, `stages` of `heads` * D elements to a warp's ring.
template <int D>
__global__ void __launch_bounds__(kRingWarps * 32, kRingBlocks)
rikv_store_e4m3_kernel(const uint16_t* __restrict__ k_full, const uint16_t* __restrict__ v_full,
                       const int32_t* __restrict__ keep_rows, const int32_t* __restrict__ n_keep, int B,
                       int N_full, int Nc_cap, int H, int heads, int groups, int stages, uint8_t* __restrict__ k_q,
                       uint8_t* __restrict__ v_q, float* __restrict__ k_scale, float* __restrict__ v_scale,
                       int32_t* dev_status) {
    extern __shared__ __align__(128) uint8_t ring_smem[];
    __shared__ uint64_t bars[kRingWarps][kRingStages];
    __shared__ RingPiece pieces[kRingWarps][kRingStages];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int stage_bytes = heads * D * 2;
    const uint8_t* ring = ring_smem + (size_t)warp * stages * stage_bytes;
    if (lane == 0) {
        for (int s = 0; s < stages; ++s) ptx::mbar_init(ptx::smem_addr(&bars[warp][s]), 1);
        ptx::fence_barrier_init();
    }
    __syncwarp();
    grid_dependency_wait();
    grid_launch_dependents();

    const long long per_request = (long long)Nc_cap * 2 * groups, total = (long long)B * per_request;
    const long long stride = (long long)gridDim.x * kRingWarps;
    long long at = (long long)blockIdx.x * kRingWarps + warp;         // first piece of the next batch of 32
    // one batch: a lane holds what it takes to fetch one piece
    uint32_t pending = 0;
    long long src = 0, dst_row = 0;
    int part = 0;
    int filled = 0, to_fill = 0;                     // pieces fetched, stage of the next one
    auto fetch_next = [&]() {
        while (pending == 0) {
            if (at >= total) return;
            const long long u = at + lane * stride;
            at += 32 * stride;
            bool live = false;
            if (u < total) {
                const int b = (int)(u / per_request);
                const long long in = u - b * per_request;
                const int j = (int)(in / (2 * groups));
                part = (int)(in - (long long)j * 2 * groups);
                const int row = keep_rows[(size_t)b * Nc_cap + j];
                if (j < live_rows(n_keep, b, Nc_cap, part == 0 && j == 0, dev_status)) {
                    live = row >= 0 && row < N_full;
                    if (!live) record_status(dev_status, REGIONE_DEV_BOUNDS);
                    src = ((long long)b * N_full + row) * H * D;
                    dst_row = (long long)b * Nc_cap + j;
                }
            }
            pending = __ballot_sync(0xffffffffu, live);
        }
        const int from = __ffs(pending) - 1;
        pending &= pending - 1;
        const long long f_src = __shfl_sync(0xffffffffu, src, from), f_dst = __shfl_sync(0xffffffffu, dst_row, from);
        const int f_part = __shfl_sync(0xffffffffu, part, from);
        if (lane == 0) {
            const int group = f_part >= groups ? f_part - groups : f_part, h0 = group * heads;
            const uint32_t bytes = (uint32_t)min(heads, H - h0) * D * 2, bar = ptx::smem_addr(&bars[warp][to_fill]);
            pieces[warp][to_fill] = {f_dst, f_part};
            ptx::mbar_arrive_expect_tx(bar, bytes);
            ptx::bulk_load(ptx::smem_addr(ring + (size_t)to_fill * stage_bytes), (f_part >= groups ? v_full : k_full) + f_src + (size_t)h0 * D,
                      bytes, bar);
        }
        ++filled;
        if (++to_fill == stages) to_fill = 0;
    };
    for (int s = 0; s < stages; ++s) fetch_next();
    __syncwarp();

    constexpr int kLanesPerHead = D / 16;            // 8 or 4, 16 elements each
    int stage = 0;
    uint32_t parity = 0;
    for (int done = 0; done < filled; ++done) {
        if (!__all_sync(0xffffffffu, ring_wait(ptx::smem_addr(&bars[warp][stage]), parity))) {
            // (the copies that are still on their way get as long again before their shared memory is given up)
            if (lane == 0) record_status(dev_status, REGIONE_DEV_TIMEOUT);
            for (; done < filled; ++done) {
                ring_wait(ptx::smem_addr(&bars[warp][stage]), parity);
                if (++stage == stages) { stage = 0; parity ^= 1; }
            }
            return;
        }
        const RingPiece piece = pieces[warp][stage];
        const int is_v = piece.part >= groups, h0 = (is_v ? piece.part - groups : piece.part) * heads;
        const int n = min(heads, H - h0) * kLanesPerHead;
        const uint4* in = reinterpret_cast<const uint4*>(ring + (size_t)stage * stage_bytes);
        uint8_t* codes = (is_v ? v_q : k_q) + ((size_t)piece.dst_row * H + h0) * D;
        float* scales = (is_v ? v_scale : k_scale) + (size_t)piece.dst_row * H + h0;
#pragma unroll 3
        for (int c0 = 0; c0 < n; c0 += 32) {
            const int c = c0 + lane;
            const bool live = c < n;
            uint4 x = make_uint4(0u, 0u, 0u, 0u), y = x;
            if (live) { x = in[2 * c]; y = in[2 * c + 1]; }
            uint32_t amax = max_magnitude(x, y);
#pragma unroll
            for (int d = kLanesPerHead / 2; d > 0; d >>= 1)
                amax = max_bits(amax, __shfl_xor_sync(0xffffffffu, amax, d));
            const int k = scale_exponent(max(amax & 0xffffu, amax >> 16));
            const float inv = __uint_as_float((uint32_t)(127 - k) << 23);  // 2^-k, exact
            if (!live) continue;
            uint4 q;
            q.x = encode4(x.x, x.y, inv); q.y = encode4(x.z, x.w, inv);
            q.z = encode4(y.x, y.y, inv); q.w = encode4(y.z, y.w, inv);
            __stcs(reinterpret_cast<uint4*>(codes) + c, q);
            if (c % kLanesPerHead == 0) scales[c / kLanesPerHead] = __uint_as_float((uint32_t)(127 + k) << 23);
        }
        __syncwarp();                                // the stage has been read
        fetch_next();
        __syncwarp();
        if (++stage == stages) { stage = 0; parity ^= 1; }
    }
}

template <int D>
__global__ void __launch_bounds__(kQuantThreads)
rikv_load_e4m3_kernel(const uint8_t* __restrict__ k_q, const uint8_t* __restrict__ v_q,
                      const float* __restrict__ k_scale, const float* __restrict__ v_scale,
                      const int32_t* __restrict__ n_keep, int Nc_cap, int H, uint16_t* __restrict__ k_cache,
                      uint16_t* __restrict__ v_cache, int32_t* dev_status) {
    grid_dependency_wait();
    grid_launch_dependents();
    constexpr int kLanesPerHead = D / 8;
    const int b = blockIdx.y, j = blockIdx.x;
    if (j >= live_rows(n_keep, b, Nc_cap, threadIdx.x == 0 && j == 0, dev_status)) return;
    const size_t dst_row = (size_t)b * Nc_cap + j;
    const int per_tensor = H * kLanesPerHead, total = 2 * per_tensor;
    for (int c0 = threadIdx.x; c0 < total; c0 += kQuantUnroll * kQuantThreads) {
        uint2 q[kQuantUnroll];
        float s[kQuantUnroll];
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) {
            const int c = c0 + u * kQuantThreads;
            if (c >= total) break;
            const int is_v = c >= per_tensor, piece = c - (is_v ? per_tensor : 0);
            q[u] = __ldcs(reinterpret_cast<const uint2*>((is_v ? v_q : k_q) + dst_row * H * D + (size_t)piece * 8));
            s[u] = (is_v ? v_scale : k_scale)[dst_row * H + piece / kLanesPerHead];
        }
#pragma unroll
        for (int u = 0; u < kQuantUnroll; ++u) {
            const int c = c0 + u * kQuantThreads;
            if (c >= total) break;
            const int is_v = c >= per_tensor, piece = c - (is_v ? per_tensor : 0);
            // (code value) * 2^k is exact in bf16: 4 significant bits, exponent well inside the range
            const float2 a = unpack_e4m3x2(q[u].x), c2 = unpack_e4m3x2(q[u].x >> 16);
            const float2 e = unpack_e4m3x2(q[u].y), g = unpack_e4m3x2(q[u].y >> 16);
            uint4 w;
            w.x = pack_bf16x2(a.x * s[u], a.y * s[u]); w.y = pack_bf16x2(c2.x * s[u], c2.y * s[u]);
            w.z = pack_bf16x2(e.x * s[u], e.y * s[u]); w.w = pack_bf16x2(g.x * s[u], g.y * s[u]);
            *reinterpret_cast<uint4*>((is_v ? v_cache : k_cache) + dst_row * H * D + (size_t)piece * 8) = w;
        }
    }
}

}  // namespace regione

using namespace regione;

static int check_quant_args(const void* a, const void* b, const void* c, const void* d, const void* e,
                            const void* f, int B, int Nc_cap, int H, int D) {
    if (!a || !b || !c || !d || !e || !f) return REGIONE_INVALID_ARG;
    if (B < 0 || Nc_cap < 0 || H < 1) return REGIONE_INVALID_ARG;
    if (D != 64 && D != 128) return REGIONE_UNSUPPORTED;
    if (B > 65535 || Nc_cap > 0x7fffffff / 2) return REGIONE_UNSUPPORTED;
    return REGIONE_OK;
}

// A block per row, or rings.  The block's passes of 768 pieces of 16 bytes have to be filled for it to keep up, and rings take
// longer to start and to drain.  Measured, block per row / rings, us:
//   passes full (24, 40, 48 heads of 128): 7885 rows 27.3 / 29.4, 44.4 / 47.0, 49.2 / 54.4
//   filled to two thirds or three quarters (16, 18, 33, 36 heads of 128): 22.3 / 20.5, 23.6 / 23.5 (14000 rows 40.0 / 36.7),
//   41.1 / 39.5, 42.2 / 40.0; 24 heads of 64 19.8 / 17.3
//   one full pass, many rows (24 heads of 128): 12000 rows 40.1 / 41.2, 16000 52.6 / 52.3, 20000 64.9 / 63.8, 40000 127.4 / 119.6;
//   two (48 heads): 20000 rows 119.7 / 132.8
//   all rows in two rounds of resident blocks: 1000 rows of 16 x 128 7.6 / 7.9, behind a flushed L2 10.2 / 12.3; 2000 rows 7.4 / 7.7,
//   12.3 / 14.4; 4000 rows 12.3 / 10.6, 18.5 / 18.4
static bool takes_rows(int B, int Nc_cap, int H, int D, int sms) {
    const long long rows = (long long)B * Nc_cap;
    if (rows <= 2LL * kRowBlocks * sms) return true;
    const long long pieces = 2LL * H * (D / 8), pass = kQuantUnroll * kQuantThreads, passes = (pieces + pass - 1) / pass;
    return 5 * pieces > 4 * pass * passes && (passes > 1 || rows < 18000);
}

template <int D>
static int launch_store(const uint16_t* k_full, const uint16_t* v_full, const int32_t* keep_rows, const int32_t* n_keep, int B,
                        int N_full, int Nc_cap, int H, uint8_t* k_q, uint8_t* v_q, float* k_scale, float* v_scale,
                        int32_t* dev_status, cudaStream_t st) {
    const int sms = sm_count();
    if (takes_rows(B, Nc_cap, H, D, sms))
        return launch_status(launch_overlapped(rikv_store_e4m3_rows_kernel<D>, dim3(Nc_cap, B), dim3(kQuantThreads), 0, st, k_full,
                                               v_full, keep_rows, n_keep, N_full, Nc_cap, H, k_q, v_q, k_scale, v_scale, dev_status));
    static int configured[kMaxDevices] = {};
    const int dev = current_device();
    if (dev < 0) return REGIONE_CUDA_ERROR;
    if (!__atomic_load_n(&configured[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(rikv_store_e4m3_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes) != cudaSuccess)
            return REGIONE_CUDA_ERROR;
        __atomic_store_n(&configured[dev], 1, __ATOMIC_RELEASE);
    }
    const int most = kPieceBytes / (2 * D), groups = (H + most - 1) / most, heads = (H + groups - 1) / groups;
    const int stage_bytes = heads * D * 2, stages = std::min(kRingStages, kRingBytes / (kRingWarps * stage_bytes));
    const long long blocks = ((long long)B * Nc_cap * 2 * groups + kRingWarps - 1) / kRingWarps;
    const cudaError_t e = launch_overlapped(
        rikv_store_e4m3_kernel<D>, dim3((unsigned)std::min<long long>(blocks, (long long)kRingBlocks * sms)),
        dim3(kRingWarps * 32), (size_t)kRingWarps * stages * stage_bytes, st, k_full, v_full, keep_rows, n_keep, B, N_full, Nc_cap,
        H, heads, groups, stages, k_q, v_q, k_scale, v_scale, dev_status);
    return launch_status(e);
}

extern "C" int regione_rikv_store_e4m3(const regione_bf16* k_full, const regione_bf16* v_full,
                                       const int32_t* keep_rows, const int32_t* n_keep, int B, int N_full,
                                       int Nc_cap, int H, int D, uint8_t* k_q, uint8_t* v_q, float* k_scale,
                                       float* v_scale, int32_t* dev_status, void* stream) {
    int rc = check_quant_args(k_full, v_full, k_q, v_q, k_scale, v_scale, B, Nc_cap, H, D);
    if (rc != REGIONE_OK) return rc;
    if (!keep_rows || !n_keep || N_full < 0) return REGIONE_INVALID_ARG;
    if (!aligned16(k_full) || !aligned16(v_full) || !aligned16(k_q) || !aligned16(v_q)) return REGIONE_INVALID_ARG;
    if (B == 0 || Nc_cap == 0) return REGIONE_OK;
    return D == 128 ? launch_store<128>(k_full, v_full, keep_rows, n_keep, B, N_full, Nc_cap, H, k_q, v_q, k_scale, v_scale,
                                        dev_status, (cudaStream_t)stream)
                    : launch_store<64>(k_full, v_full, keep_rows, n_keep, B, N_full, Nc_cap, H, k_q, v_q, k_scale, v_scale,
                                       dev_status, (cudaStream_t)stream);
}

extern "C" int regione_rikv_load_e4m3(const uint8_t* k_q, const uint8_t* v_q, const float* k_scale,
                                      const float* v_scale, const int32_t* n_keep, int B, int Nc_cap, int H,
                                      int D, regione_bf16* k_cache, regione_bf16* v_cache,
                                      int32_t* dev_status, void* stream) {
    int rc = check_quant_args(k_q, v_q, k_scale, v_scale, k_cache, v_cache, B, Nc_cap, H, D);
    if (rc != REGIONE_OK) return rc;
    if (!n_keep) return REGIONE_INVALID_ARG;
    if (!aligned16(k_q) || !aligned16(v_q) || !aligned16(k_cache) || !aligned16(v_cache)) return REGIONE_INVALID_ARG;
    if (B == 0 || Nc_cap == 0) return REGIONE_OK;
    const dim3 grid(Nc_cap, B);
    cudaError_t e = D == 128
        ? launch_overlapped(rikv_load_e4m3_kernel<128>, grid, dim3(kQuantThreads), 0, (cudaStream_t)stream,
                            k_q, v_q, k_scale, v_scale, n_keep, Nc_cap, H, k_cache, v_cache, dev_status)
        : launch_overlapped(rikv_load_e4m3_kernel<64>, grid, dim3(kQuantThreads), 0, (cudaStream_t)stream,
                            k_q, v_q, k_scale, v_scale, n_keep, Nc_cap, H, k_cache, v_cache, dev_status);
    return launch_status(e);
}
