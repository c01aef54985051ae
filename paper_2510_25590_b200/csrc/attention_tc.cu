// Region attention with the Region-Instruction KV cache on the 5th-generation
// tensor cores (Sec. 4 "Region-Aware Generation", the attention equation):
// queries of the recomputed tokens against [fresh keys | cached keys] without
// materialising the concatenation.
//
// One CTA = one (request, head, pair of 128-row query tiles).  Warp roles:
//   warps 0-15  softmax and epilogue: thread = (query row, 64-key chunk of a key tile); warps 0-7 work on
//               query tile 0, warps 8-15 on query tile 1, the first four of each on the first chunk
//   warp  16    TMA producer: Q once, then K_j, V_j tiles (128 keys) through a ring of shared-memory stages;
//               the cached segment and the fresh segment are two tensor maps walked one after the other; plans the
//               CTA's next segment
//   warp  17    issuer of the O_t += P_t V_j products of both query tiles (the whole warp walks the loop, one
//               elected lane issues); owns the tensor-memory allocation
//   warp  18    in the launch that also refreshes the Region-Instruction KV cache: moves the retained rows by
//               asynchronous bulk copies; idle otherwise
//   warp  19    issuer of the S = Q_t K_j^T products of both query tiles
//   (warps 16-19 give registers up to the softmax warpgroups with setmaxnreg: 64 against 104 per thread)
//
// Tensor memory (512 columns): S | P0 | P1 | O0 | O1 = 128 + 64 + 64 + 128 + 128.
// There is ONE S buffer (fp32, 128 logits per row), a staging place that the two query tiles share: a product
// lands there, the softmax warps of its tile read it into registers and give the buffer back at once, and the
// next product (the other tile's, or the same tile's next key tile) may follow while the exponentials are
// still being computed.  The probabilities go to the tile's own P region as packed bf16, chunk by chunk, and
// O_t += P_t V_j runs straight from tensor memory.  Because P does not live in the S buffer, S_t(j+1) never
// waits for the products P_t(j) V_j.  What a chunk's threads wait for before they overwrite its part of P_t is
// the completion of the previous key tile's product with that part.  A pair with a single live query tile does
// not leave the second tile's warps idle: they run the same query tile against the odd key tiles of the segment
// (own accumulator, maximum and sum), the first tile's warps take the even ones, and the epilogue merges them.
//
// What bounds the loop: per key tile and query pair the tensor cores need 2048 cycles and the special-function
// unit 2048 (32768 exponentials, 16 a cycle); the dependency chain  S -> registers -> exponentials -> P -> product
// hides behind neither.  Two threads per row (four softmax warps per scheduler instead of two), no row maximum
// after the first key tile and packed fp32 arithmetic shorten the chain: 2640 cycles per key tile and pair, 2460 with
// D = 64 (active cycles of 64 key tiles less those of 32, one item a CTA; 19000 more are fill, drain and epilogue).
// Measured, one box, L2 warm, against one thread per row, a maximum per key tile and scalar arithmetic:
// 8704 queries x 8704 keys x 24 heads 763 -> 720 us in isolation (1292 TFLOP/s), 889 -> 848 us under the power
// cap; 4 x 1382 queries x 18944 keys 1141 -> 1056 us; 2048 queries x 8448 keys 189 -> 180 us; D = 64 127 -> 114 us;
// 205 queries x 8448 keys, where the fill and the drain of the pipeline dominate, 42.3 -> 43.2 us.
//
// Online softmax in the exp2 domain without a running maximum: a row's reference is its maximum over the
// segment's first key tile.  Any reference within a factor of 2^60 of the true maximum gives the same relative
// accuracy (probabilities are bf16, their sums fp32: see chunk_sum).  A row whose chunk sum reaches 2^60 (a
// later logit above the first key tile's by 37 nats if a chunk holds 64 of them, by 42 if it is alone) makes the CTA
// walk the segment twice more, once for the rows' true maxima and once with them.  That costs up to three times the
// segment: 819 queries x 8704 keys 97 -> 213 us with one such row a head, 8704 x 8704 718 -> 1056 us, with every row
// 1944 us.  Keys past a segment's live count are masked in the
// softmax and their V rows zeroed in shared memory, so garbage (even NaN) behind the live prefix cannot leak.
//
// Scheduling: the kernel is persistent, one CTA per SM.  A "step" is one key tile of one
// (request, head, query pair) item; all steps of the launch form one sequence, item after item,
// laid out on a cost axis (a step of a pair with one live query tile costs half a step of a full
// pair, and every item starts with a fixed cost for draining and refilling the pipeline), which is cut into
// equal contiguous shares, one per CTA (a stream-K decomposition: the grid is always one balanced wave,
// whatever the number of items).  A CTA's share is a few segments, each a run of key tiles of one item.  A segment
// that covers its item completely writes the output rows directly; otherwise its unnormalised output and
// (max, sum) pairs go to a slot of the caller's workspace, and either the item's first share merges the slots into its
// own rows (kMergeHere) or a small second kernel does (kMergeKernel; the attention kernel leaves it a table of the items
// that its share boundaries cut): see merges_here.  The share length is bounded below so that no item is spread over
// more slots than the workspace holds.
// On large calls the power limit sets the time, and K and V read from HBM again and again cost as much of it as all of the
// softmax: where they are more than L2 keeps, whole pairs are dealt in waves, or teams of CTAs walk a head together
// (plan_shares).  8704 x 8704, 24 heads: 1.18 -> 0.16 GB read from HBM, 35 -> 10 M sectors across the halves of L2, 838 -> 768
// us at 1 kW; 8448 x 8448 refreshing the cache 819 -> 750; 2048 of 8448 rows refreshed 245 -> 227; 1075 x 8448 143 -> 134;
// 819 x 8704 201 -> 139 MB, 127 -> 123 us.
// Where the capacities allow only few items (choose_cluster), an item is shared by a cluster of 2 to 8 CTAs instead, an
// equal run of its key tiles each; they leave their partial rows in shared memory, where the cluster's CTAs read
// them (distributed shared memory) and write the output: no workspace, no second kernel, no plan to derive.  Measured,
// shares of the cost axis -> clusters: 3 x 333 queries x 261 keys x 5 heads 20.9 -> 17.9 us (D = 64 17.4 -> 14.4),
// 2 x 700 x 3700 x 12 47.8 -> 44.0 (D = 64 41.6 -> 35.3), 256 x 2112 x 4, D = 64 17.1 -> 15.5, one row 14.2 -> 10.6.
// Counts live in device memory, so every CTA derives the same plan from them.  Output rows go to
// out[b, i] or, with a row list, to out[b, out_rows[b, i]] (the scatter of the attention rows back
// into the joint sequence, done by whichever kernel writes the row).
//
// Every wait is bounded: if a barrier does not complete within ~2 s the CTA
// records REGIONE_DEV_TIMEOUT, all roles leave their loops, tensor memory is
// released and the kernel ends normally.
#include <cuda.h>
#include <cstddef>
#include <type_traits>

#include <algorithm>
#include <atomic>
#include <chrono>

#include "attention_plan.cuh"
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace regione {

constexpr int kSoftmaxWarps = 16;        // 4 softmax warpgroups: [query tile][64-key chunk]
constexpr int kWarpLoad = kSoftmaxWarps, kWarpPv = kSoftmaxWarps + 1, kWarpCopy = kSoftmaxWarps + 2,
              kWarpS = kSoftmaxWarps + 3;
constexpr int kAttnThreads = 32 * (kSoftmaxWarps + 4);
constexpr int kWalkBarrier = 4, kWalkThreads = kAttnThreads - 32;   // named barrier of the warps that walk the segments
constexpr int kMaxCluster = 8;           // CTAs that may share an item through their shared memories
constexpr int kBH = 64;                  // key rows per chunk (half a tile): the logits one thread holds
constexpr float kOutgrownSum = 1.152921504606846976e18f;   // 2^60: chunk sum at which a reference maximum is renewed
constexpr int kCopySlots = 2;             // cache refresh: batches of rows under way at once, at most
constexpr int kHalfBytes = 128 * 64 * 2; // one 128-row x 64-column bf16 box (128-byte rows)
constexpr long long kTimeoutCycles = 4000000000LL;   // default bound of every wait (about 2 s)

template <int D>
struct AttnCfg {
    static constexpr int kHalves = D / 64;
    static constexpr int kTileBytes = kHalves * kHalfBytes;
    static constexpr int kStages = (D == 128) ? 4 : 6;
    // 2 query tiles + the ring + one more stage that only a lone query tile uses (its ring is that
    // stage, the ordinary ring and the idle second query tile: kStages + 2 stages, an even number: K tiles and
    // V tiles have stages of their own)
    static constexpr int kSmemTiles = (2 + kStages + 1) * kTileBytes;
    static constexpr int kCtrlBytes = 768;
    static constexpr int kExchBytes = 4 * kBM * 4;         // exchange of the chunks' maxima and sums
    static constexpr int kExtraAt = kSmemTiles + kCtrlBytes + kExchBytes;
    // D = 128 fills shared memory: the epilogue stages its rows (4 KB per softmax warp) in the idle query
    // tiles, and a launch that refreshes the cache copies rows through the extra stage, a lone query tile
    // then keeps to the ordinary number of stages.  D = 64 has room for both.
    static constexpr int kStageAt = (D == 128) ? 0 : kExtraAt;
    static constexpr int kCopyBytes = (D == 128) ? kTileBytes : 16384;
    static constexpr int kCopyAt = (D == 128) ? (2 + kStages) * kTileBytes : kExtraAt + kSoftmaxWarps * 4096;
    static constexpr int kSmemBytes = kExtraAt + (D == 128 ? 0 : kSoftmaxWarps * 4096 + kCopyBytes);
    static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
    __host__ __device__ static constexpr int lone_stages(bool store) { return kStages + (D == 128 && store ? 0 : 2); }
    // partial rows that stay in shared memory, chunk by chunk, and their (max, sum) pairs: of an item shared by a
    // cluster, and of the first share of a cut item
    static constexpr int kPartialMlAt = 2 * kBM * D * 4;
    static_assert(kPartialMlAt + 2 * kBM * 8 <= kSmemTiles, "partial rows");
    // slots of the copies that are left when the walks are over and all tiles are idle
    static constexpr int kTailBytes = (D == 128) ? 3 * 65536 : 3 * 40960;
    static_assert(kTailBytes <= kSmemTiles, "tail slots");
};

// The part of one item that a CTA works on, as its roles need it (shared memory).
struct SegInfo {
    int live;                   // 0: the share ends here
    int b, h, q0, nq;           // request, head, first query row, live query rows of the request
    int j_first, n_tiles;       // key tiles [j_first, j_first + n_tiles) of the item
    int nt_c, nt, nc, nf;       // cached key tiles, all key tiles, live keys of the two segments
    int slot, n_slots;          // slot among the shares that touch the item
    int slot_at, slot_step;     // where slot 1 lies in the workspace, and how far apart the later ones do (slot 0: slot_at - 1)
    int share_step;             // how far apart the shares are that touch the item
    int apart;                  // (launch that refreshes the cache) fresh rows are not in K and V themselves: see ReqShape
};

struct AttnCtrl {
    uint64_t q_full;
    uint64_t kv_full[8];        // up to AttnCfg::kStages + 2 stages
    uint64_t kv_empty[8];
    uint64_t s_full[2];         // [query tile]
    uint64_t p_full[2][2];      // [query tile][chunk of 64 keys]
    uint64_t o_final[2];        // completes once, after the tile's last P*V product
    uint64_t pv_done[2];        // [query tile] completes after every key tile's last product: the second chunk's P
                                // may be overwritten
    uint64_t pv_half[2];        // [query tile] ... after every key tile's first product: the first chunk's P may be
    uint64_t s_free;            // the shared S buffer has been read by the softmax warps it was computed for
    uint64_t v_full[4];         // [V stage] key tiles of role 1 of a lone query tile (see v_landing)
    uint32_t tmem_base;
    int abort_flag;
    int redo;                   // a row outgrew the reference maximum of its first key tile
    SegInfo seg[2];
    uint64_t peers_ready;       // item shared by a cluster: every CTA's partial rows are in its shared memory
    uint64_t peers_done;        // ... and have been read by every CTA (launch that refreshes the cache)
    int walks_done;             // cache refresh: the walks are over, every tile of shared memory is idle
    int copy_abort;             // cache refresh: a copy did not land in time.  Not abort_flag: that one changes only
                                // while every role is between two barriers of a segment, so that all leave together
    // cache refresh: a slot's rows have landed; where they go, and which of them are to be stored
    uint64_t copy_full[kCopySlots];
    uint8_t* copy_dst[kCopySlots];
    int copy_item[kCopySlots];
    uint32_t copy_valid[kCopySlots];
    alignas(8) uint8_t cursor[120];     // ShareCursor of the planning warp between two segments
};

// The barriers of AttnCtrl as one array starting at q_full.
constexpr int kBarKvEmpty = 9, kBarSFull = 17, kBarPFull = 19, kBarOFinal = 23, kBarPvDone = 25, kBarPvHalf = 27,
              kBarSFree = 29, kNumBarriers = 34;
static_assert(offsetof(AttnCtrl, kv_empty) == kBarKvEmpty * 8 && offsetof(AttnCtrl, s_full) == kBarSFull * 8 &&
              offsetof(AttnCtrl, p_full) == kBarPFull * 8 && offsetof(AttnCtrl, o_final) == kBarOFinal * 8 &&
              offsetof(AttnCtrl, pv_done) == kBarPvDone * 8 && offsetof(AttnCtrl, pv_half) == kBarPvHalf * 8 &&
              offsetof(AttnCtrl, s_free) == kBarSFree * 8 && offsetof(AttnCtrl, v_full) == (kBarSFree + 1) * 8 &&
              offsetof(AttnCtrl, tmem_base) == kNumBarriers * 8 &&
              sizeof(AttnCtrl) <= AttnCfg<128>::kCtrlBytes, "barrier layout");

// What share c tells the merge kernel: the item that the boundary between shares c - 1 and c
// cuts, if c is the second share of that item (so every cut item is named exactly once).
struct alignas(16) CutItem {
    int valid, b, h, qp, n_slots, nq, slot_at, slot_step;
};

// Who puts the parts of an item together that several CTAs work on: a merge kernel behind this one, the item's
// first share, or the CTAs of a cluster; and whether the plan minds the order in which K and V are read (see plan_shares).
// (Instantiations of their own: the code of one form costs the others 1 to 2 %, the plan of the spread forms 1 us.)
enum MergeForm { kMergeKernel, kMergeHere, kMergeCluster };
enum KernelForm { kFormKernel, kFormHere, kFormCluster, kFormSpreadKernel, kFormSpreadHere };
__host__ __device__ constexpr bool is_spread(int form) { return form >= kFormSpreadKernel; }
__host__ __device__ constexpr int merge_of(int form) { return is_spread(form) ? form - kFormSpreadKernel : form; }

struct AttnParams : PlanInput {
    float scale_log2e;
    int out_cap;         // rows per request of `out` (Nq_cap without out_rows)
    uint16_t* out;       // [B, out_cap, H, D]
    const int32_t* out_rows;   // nullptr: query row i goes to out row i; else to row out_rows[b, i]
    int32_t* dev_status;
    float* part_o;       // [B * H * P_cap * max_slots, 256, D] unnormalised outputs; kMergeHere: [..., D / 4, 256, 4]
    float2* part_ml;     // [B * H * P_cap * max_slots, 256]    (running max in the exp2 domain, sum)
    CutItem* cut;        // kMergeKernel: [grid] the item that the start of each share cuts
    unsigned long long* ready;       // kMergeHere: [grid] `epoch`: the share's partial rows are in its slot (0: merged),
                                     // and a word behind them, `epoch`: a launch of this epoch has timed out
    unsigned long long epoch;        // of this launch: what lies in the workspace otherwise is not equal to it
    long long timeout_cycles;   // bound of every barrier wait, in SM clock cycles
    int cluster;         // kMergeCluster: CTAs that share an item; no workspace
    int kv_once;         // every key tile is read by one CTA: it need not stay in L2
};

// Cache refresh fused into a full step: the rows rows[l][b, 0..n[l][b]) (ascending) of the K and V that the launch
// attends over are also written to dst[2l], dst[2l + 1] [B, cap[l], H, D], l < n_lists: the rows that the cache
// retains, and in a region step the recomputed rows.  A parameter of its own, of the kernel that refreshes the cache
// only: the plain attention kernel's parameters do not grow.
struct StoreParams {
    const int32_t* rows[2];
    const int32_t* n[2];
    int cap[2];
    int n_lists, src_cap;               // (rows per request of the sources)
    const uint8_t* src[2];              // K, V [B, src_cap, H, D]
    uint8_t* dst[4];
};

// Bounded wait on phase `parity` of an mbarrier: true when the phase completed, false when another
// role has already given up or `limit` cycles have passed (then the abort flag is raised and
// REGIONE_DEV_TIMEOUT recorded; the caller leaves its loop, nothing traps).
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         int32_t* dev_status, long long limit) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            record_status(dev_status, REGIONE_DEV_TIMEOUT);
            return false;
        }
    }
}

// The same for phase 0 of a barrier that the CTAs of a cluster arrive on.
__device__ __forceinline__ bool wait_bar_cluster(uint32_t bar, volatile int* abort_flag, int32_t* dev_status, long long limit) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait_cluster(bar, 0)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            record_status(dev_status, REGIONE_DEV_TIMEOUT);
            return false;
        }
    }
    return true;
}

// Keys >= valid of a 64-logit chunk are dead (behind a segment's live prefix): their logits become
// -inf, after which the chunk goes through the same code as a full one (maximum unaffected,
// probability 0 or, on the polynomial path, 2^-126).  A short separate pass instead of masked
// variants of the long unrolled loops: those would run once per item, from a cold instruction cache.
__device__ __forceinline__ void mask_dead_keys(uint32_t* s, int valid) {
#pragma unroll
    for (int i = 0; i < kBH; ++i)
        if (i >= valid) s[i] = 0xff800000u;
}

// Maximum of 64 logits held in registers.
__device__ __forceinline__ float chunk_max(const uint32_t* s) {
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < kBH; ++i) mx[i & 3] = fmaxf(mx[i & 3], __uint_as_float(s[i]));
    return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}

// Barrier `id` of the CTA's named barriers, for `n` threads.
__device__ __forceinline__ void named_barrier(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Two fp32 values in one 64-bit register pair, and the packed operations on them.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// c + a for a bf16 `a` (exact widening, one fp32 rounding).
__device__ __forceinline__ float add_bf16(float c, uint16_t a) {
    float r;
    asm("add.rn.f32.bf16 %0, %1, %2;" : "=f"(r) : "h"(a), "f"(c));
    return r;
}

// p = 2^(s*c - m) for 64 logits, written to tensor memory at `tP` (32 columns) as packed bf16; the packed pairs are left
// in s[0..31] for chunk_sum.  The exponentials replace the logits in place and leave in pieces of 8 columns, so that
// a thread's 104 registers hold the chunk.  All of them run on the special-function unit: it is busy 2048 of the
// loop's 2640 cycles, and moving a quarter or an eighth of them to the FMA pipe (a cubic) made the call 4 % and 0 %
// slower.
__device__ __forceinline__ void chunk_probabilities(uint32_t tP, uint32_t* s, float c, float m) {
    const uint64_t c2 = pack2(c, c), m2 = pack2(-m, -m);
#pragma unroll
    for (int i = 0; i < kBH; i += 2) {
        float a, b;
        unpack2(fma2(pack2(__uint_as_float(s[i]), __uint_as_float(s[i + 1])), c2, m2), a, b);
        s[i] = __float_as_uint(fast_exp2(a));
        s[i + 1] = __float_as_uint(fast_exp2(b));
    }
#pragma unroll
    for (int g = 0; g < kBH; g += 16) {
        uint32_t pk[8];
#pragma unroll
        for (int i = g; i < g + 16; i += 2)
            s[i >> 1] = pk[(i - g) >> 1] = pack_bf16x2(__uint_as_float(s[i]), __uint_as_float(s[i + 1]));
        ptx::tmem_st8(tP + (g >> 1), pk);
    }
}

// fp32 sum of a chunk's probabilities as they were written.  (The sum of the unrounded values leaves the rounding of a key
// that dominates its row in the result, unless the reference m is that key's own logit: against 64 bits, 512 x 8448 x 128
// with logits of deviation 1 / 2 / 4 / 8, relative error 2.33 / 2.27 / 2.29 / 2.27e-3, this way 2.33 / 2.21 / 1.91 /
// 1.76e-3, with a running maximum 2.32 / 2.25 / 1.96 / 1.74e-3.)  Nothing waits for it, so it follows the chunk's arrival:
// beside the exponentials, ahead of the arrival, the 64 additions cost 205 queries x 8448 keys 1.1 us (step 55.1 -> 54.0),
// 8704 x 8704 15 us (854 -> 839); the launches that copy rows beside it +-0.6 %.  Widening the pairs and adding them two
// at a time: step 54.8 us, 857 us.
__device__ __forceinline__ float chunk_sum(const uint32_t* w) {
    float sum[4] = {};
#pragma unroll
    for (int i = 0; i < kBH; i += 2) {
        sum[i & 3] = add_bf16(sum[i & 3], (uint16_t)w[i >> 1]);
        sum[(i + 1) & 3] = add_bf16(sum[(i + 1) & 3], (uint16_t)(w[i >> 1] >> 16));
    }
    return (sum[0] + sum[1]) + (sum[2] + sum[3]);
}

// Live keys of the key tiles of a segment: kBN but for the last tile of either part of the KV sequence.
struct TileKeys {
    int jc, vc, jf, vf;     // segment-relative index and live keys of the last cached / last fresh tile
    __device__ __forceinline__ explicit TileKeys(const SegInfo& it) {
        jc = it.nt_c - 1 - it.j_first; vc = it.nc - (it.nt_c - 1) * kBN;
        jf = it.nt - 1 - it.j_first;   vf = it.nf - (it.nt - it.nt_c - 1) * kBN;
    }
    __device__ __forceinline__ int operator()(int jl) const { return jl == jc ? vc : jl == jf ? vf : kBN; }
};

// The barrier on which V of key tile jl lands, and the phase of it.  A barrier's waiter must see every phase of
// it, or a wait for a phase could be answered by the one two phases back.  With 4 or 8 stages a lone query tile's
// two roles never share a V stage; with 6 they take turns on it, so each role has a barrier of its own there.
struct VLanding {
    uint32_t bar;
    int phase;
};
__device__ __forceinline__ VLanding v_landing(AttnCtrl* ctrl, bool split, int n_stages, int jl) {
    const int iv = 2 * jl + 1, sv = iv % n_stages, use = iv / n_stages;
    if (split && n_stages % 4 != 0) return {ptx::smem_addr(jl & 1 ? &ctrl->v_full[sv >> 1] : &ctrl->kv_full[sv]), use >> 1};
    return {ptx::smem_addr(&ctrl->kv_full[sv]), use};
}

// What one walk over a segment does.  kWalk: one pass, the reference maximum of a row is its maximum over
// the segment's first key tile.  If a row outgrows that (AttnCtrl::redo) the segment is walked twice more:
// kMaxOnly finds the rows' maxima, kExact repeats the pass with them.
enum WalkMode { kWalk, kMaxOnly, kExact };

// Bounded wait of a warp for the partial rows of the n shares behind this CTA's, `step` apart (true: they are there).  A launch that
// has timed out may have left flags of its epoch behind, and a graph repeats the launch with that epoch: the repetition
// gives up as well, instead of merging what the flags no longer stand for.  (Asked here, beside the flags: at the start
// of the launch the question cost 819 queries x 8704 keys 1.5 us.)
__device__ __forceinline__ bool wait_shares(const AttnParams& p, int n, int step, int lane, volatile int* abort_flag) {
    const bool asks_failed = lane == 31;   // (the word behind the flags; n < 31)
    bool there = lane >= n && !asks_failed, gave_up = false;
    if (!there) {
        const unsigned long long* const word = p.ready + (asks_failed ? (int)gridDim.x : share_of(gridDim.x, blockIdx.x) + (1 + lane) * step);
        const long long t0 = clock64();
        while (!(there = (ptx::ld_acquire_u64(word) == p.epoch) != asks_failed) && !gave_up) {
            gave_up = *abort_flag != 0;
            if (asks_failed || clock64() - t0 > p.timeout_cycles) {
                *abort_flag = 1;
                record_status(p.dev_status, REGIONE_DEV_TIMEOUT);
                gave_up = true;
            }
        }
    }
    there = __all_sync(0xffffffffu, there);
    __syncwarp();                          // (the polling lanes' acquire holds for the whole warp)
    return there;
}

// ---- softmax / epilogue of one segment: thread = (query row, 64-key chunk) ----------------------------
template <int D, bool STORE, int FORM>
__device__ __forceinline__ void softmax_segment(const AttnParams& p, AttnCtrl* ctrl, const SegInfo& it, uint8_t* smem_gen,
                                                const uint32_t tmem, const int warp, const int lane, const int mode,
                                                float& m_known) {
    using Cfg = AttnCfg<D>;
    constexpr int kTileBytes = Cfg::kTileBytes;
    volatile int* abort_flag = &ctrl->abort_flag;
    const int t = warp >> 3, ck = (warp >> 2) & 1;
    const int n_tiles = it.n_tiles;
    const bool pair = it.nq - it.q0 > kBM;
    const bool split = !pair && n_tiles >= 2;
    if (t == 1 && !pair && !split) return;
    const int row = ((warp & 3) << 5) + lane;                  // row of the query tile
    const uint32_t lane_sel = (uint32_t)((warp & 3) << 5) << 16;
    const uint32_t tS = tmem + lane_sel + ck * kBH;            // this chunk of the S staging buffer
    const uint32_t tP = tmem + lane_sel + kBN + t * (kBN / 2) + ck * (kBH / 2);   // its probabilities (bf16 pairs)
    // [tile][chunk][row]: maxima at the first key tile, sums at the end
    float* const exch = reinterpret_cast<float*>(smem_gen + Cfg::kSmemTiles + Cfg::kCtrlBytes) + t * 2 * kBM + row;
    const float c = p.scale_log2e;
    float m = -INFINITY, l = 0.f;
    bool ok = true, outgrown = false;
    {
        const TileKeys keys(it);
        const int n_my = split ? (n_tiles + 1 - t) >> 1 : n_tiles;
        const uint32_t bar_s = ptx::smem_addr(&ctrl->s_full[t]), bar_free = ptx::smem_addr(&ctrl->s_free);
        const uint32_t bar_p = ptx::smem_addr(&ctrl->p_full[t][ck]);
        const uint32_t bar_pv = ptx::smem_addr(ck == 0 ? &ctrl->pv_half[t] : &ctrl->pv_done[t]);
        for (int j = 0; j < n_my; ++j) {
            const int jl = split ? 2 * j + t : j;
            const int valid = keys(jl);
            const int live_keys = valid - ck * kBH;                // live keys of this chunk (<= 0: none)
            ok = wait_bar(bar_s, j & 1, abort_flag, p.dev_status, p.timeout_cycles);
            uint32_t s[kBH];
            if (ok) {
                ptx::tc_fence_after_sync();
                if (live_keys > 0) {
                    ptx::tmem_ld32(tS, s);
                    ptx::tmem_ld32(tS + 32, s + 32);
                    ptx::tmem_wait_ld();
                }
                // the logits are in registers: the staging buffer may take the next product (of the other
                // query tile, or of this tile's next key tile)
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar_free);
                if (live_keys > 0 && live_keys < kBH) mask_dead_keys(s, live_keys);
            }
            if (mode == kMaxOnly) {
                if (!ok) break;
                if (live_keys > 0) m = fmaxf(m, chunk_max(s) * c);
                continue;
            }
            // The reference maximum of a row is its maximum over the first key tile (any reference within a
            // factor of 2^60 of the true maximum gives the same relative accuracy): the two chunks' threads
            // of a row agree on it once and then run independently of each other.
            if (j == 0) {
                if (mode == kExact) {
                    m = m_known;
                } else {
                    exch[ck * kBM] = (ok && live_keys > 0) ? chunk_max(s) * c : -INFINITY;
                    named_barrier(1 + t, 2 * kBM);
                    m = fmaxf(exch[0], exch[kBM]);
                    named_barrier(1 + t, 2 * kBM);                 // (the sums go to the same place at the end)
                }
            }
            if (!ok) break;
            // the chunk's place in tensor memory belongs to the previous key tile's product until that has completed
            if (j > 0) {
                ok = wait_bar(bar_pv, (j - 1) & 1, abort_flag, p.dev_status, p.timeout_cycles);
                if (!ok) break;
                ptx::tc_fence_after_sync();
            }
            // (a second chunk without live keys waits and arrives like any other, so that every barrier goes
            // through one phase per key tile; it writes nothing and no product reads it)
            if (live_keys > 0) {
                chunk_probabilities(tP, s, c, m);
                ptx::tmem_wait_st();
            }
            if (valid < kBN && ck == 0) {
                // last tile of a part: zero the V rows behind the live prefix (0 * NaN = NaN)
                const int n_stages = split ? Cfg::lone_stages(STORE) : Cfg::kStages;
                const int sv = (2 * jl + 1) % n_stages;
                const VLanding vl = v_landing(ctrl, split, n_stages, jl);
                ok = wait_bar(vl.bar, vl.phase & 1, abort_flag, p.dev_status, p.timeout_cycles);
                if (!ok) break;
                if (row >= valid) {
                    uint8_t* vrow = smem_gen + ((split ? 1 : 2) + sv) * kTileBytes + row * 128;
#pragma unroll
                    for (int hf = 0; hf < Cfg::kHalves; ++hf)
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            reinterpret_cast<uint4*>(vrow + hf * kHalfBytes)[q] = make_uint4(0, 0, 0, 0);
                }
                ptx::fence_proxy_async_smem();
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_p);
            if (live_keys > 0) {
                const float sum = chunk_sum(s);
                outgrown |= !(sum < kOutgrownSum);
                l += sum;
            }
        }
    }
    if (mode == kMaxOnly) {
        exch[ck * kBM] = m;
        named_barrier(1 + t, 2 * kBM);
        m_known = fmaxf(exch[0], exch[kBM]);
        return;
    }

    // ---- epilogue (rows past n_q are not written).  A thread holds one row, so storing straight
    // from registers would touch 32 different rows per warp instruction; instead each warp
    // passes row pieces of 32 columns through its own 4 KB corner of the (now idle) query tiles in
    // shared memory and stores whole pieces.  The columns of a query tile are dealt to the
    // warpgroups at work on it: two, or all four of a lone tile.
    const int qt = split ? 0 : t;
    const int wrow0 = it.q0 + qt * kBM + ((warp & 3) << 5);     // first query row of this warp
    const bool live = wrow0 + lane < it.nq;
    if (outgrown && live && mode == kWalk) ctrl->redo = 1;      // (rows past n_q may hold anything)
    const bool direct = it.n_slots == 1;
    // where this thread's query row goes in `out` (-1: the row is dead); the lookup is issued
    // ahead of the wait for the last product and used after it
    int dst_row = -1;
    if (live && direct)
        dst_row = p.out_rows != nullptr ? p.out_rows[(size_t)it.b * p.Nq_cap + wrow0 + lane] : wrow0 + lane;
    if (n_tiles > 0 && ok) {
        ok = wait_bar(ptx::smem_addr(&ctrl->o_final[t]), 0, abort_flag, p.dev_status, p.timeout_cycles);
        if (split && ok)
            ok = wait_bar(ptx::smem_addr(&ctrl->o_final[1 - t]), 0, abort_flag, p.dev_status, p.timeout_cycles);
        if (ok) ptx::tc_fence_after_sync();
    }
    float w0 = 1.f, w1 = 0.f;                           // weights of the two accumulators (lone tile)
    if (n_tiles > 0) {
        exch[ck * kBM] = l;
        if (split) {
            // the ring is idle by now: the maxima of the two halves go there
            float* const ms = reinterpret_cast<float*>(smem_gen + 2 * kTileBytes) + row;
            if (ck == 0) ms[t * kBM] = m;
            named_barrier(3, 4 * kBM);
            const float* const e0 = exch - t * 2 * kBM;
            const float m0 = ms[0], m1 = ms[kBM], l0 = e0[0] + e0[kBM], l1 = e0[2 * kBM] + e0[3 * kBM];
            m = fmaxf(m0, m1);
            w0 = l0 > 0.f ? fast_exp2(m0 - m) : 0.f;
            w1 = l1 > 0.f ? fast_exp2(m1 - m) : 0.f;
            l = w0 * l0 + w1 * l1;
        } else {
            named_barrier(1 + t, 2 * kBM);
            l = exch[0] + exch[kBM];
        }
    }
    // the rows stay in shared memory: of an item shared by a cluster, and of the first share of a cut item, which
    // merges the later shares' rows into them (merge_shares)
    const bool shared = FORM == kMergeCluster || (FORM == kMergeHere && it.n_slots > 1 && it.slot == 0);
    if (shared && n_tiles > 0 && pair && ok) {
        // (the partial rows go over the tiles that the other query tile's products may still read)
        ok = wait_bar(ptx::smem_addr(&ctrl->o_final[1 - t]), 0, abort_flag, p.dev_status, p.timeout_cycles);
        if (ok) ptx::tc_fence_after_sync();
    }
    // this warp's 32-column pieces of the row: [pc0, pc1)
    constexpr int kPieces = D / 32;
    const int per = split ? (kPieces >= 4 ? 1 : (t == 0 ? 1 : 0)) : kPieces / 2;
    const int pc0 = split ? (kPieces >= 4 ? 2 * ck + t : ck) : ck * per, pc1 = pc0 + per;
    const uint32_t tO = tmem + lane_sel + 256 + (split ? 0 : t * D);
    const size_t slot_at = (size_t)(it.slot > 0 ? it.slot_at + (it.slot - 1) * it.slot_step : it.slot_at - 1);
    const size_t prow = slot_at * (2 * kBM) + qt * kBM + row;           // row in the slot
    const float inv = l > 0.f ? 1.f / l : 0.f;
    uint8_t* const stage = smem_gen + Cfg::kStageAt + warp * 4096;
    const size_t out_stride = (size_t)p.H * D * 2;
    uint8_t* const out0 = reinterpret_cast<uint8_t*>(p.out) + (((size_t)it.b * p.out_cap) * p.H + it.h) * D * 2;
    if (direct && (dst_row >= p.out_cap || (dst_row < 0 && live))) {     // destination out of range: dropped
        record_status(p.dev_status, REGIONE_DEV_BOUNDS);
        dst_row = -1;
    }
    if (shared) {
        float2* const ml = reinterpret_cast<float2*>(smem_gen + Cfg::kPartialMlAt) + qt * kBM + row;
        if (ck == 0 && (!split || t == 0)) *ml = n_tiles > 0 && ok ? make_float2(m, l) : make_float2(-INFINITY, 0.f);
    }
    if (shared && n_tiles == 0) {
    } else if (n_tiles == 0) {
        // no keys: zero rows (an item without keys is one step and never cut)
        if (ck == 0 && direct && dst_row >= 0)
            for (int q = 0; q < D / 8; ++q)
                reinterpret_cast<uint4*>(out0 + dst_row * out_stride)[q] = make_uint4(0, 0, 0, 0);
    } else if (ok) {
#pragma unroll 1
        for (int pc = pc0; pc < pc1; ++pc) {
            uint32_t r[32];
            ptx::tmem_ld32(tO + pc * 32, r);
            if (split) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    uint32_t r1[16];
                    ptx::tmem_ld16(tO + D + pc * 32 + hf * 16, r1);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        r[hf * 16 + i] = __float_as_uint(fmaf(w0, __uint_as_float(r[hf * 16 + i]), w1 * __uint_as_float(r1[i])));
                }
            } else {
                ptx::tmem_wait_ld();
            }
            // 16-byte chunk q of row r sits at column q ^ (r & 7): both the row-wise writes and
            // the piece-wise reads are free of bank conflicts without padding
            uint4* const mine = reinterpret_cast<uint4*>(stage + lane * 128);
            if (shared) {
                // unnormalised O of this rank, 16-byte chunk by chunk with the 32 rows of the warp side by side
                uint4* const col = reinterpret_cast<uint4*>(smem_gen) + ((qt * 4 + (warp & 3)) * (D / 4) + pc * 8) * 32 + lane;
#pragma unroll
                for (int q = 0; q < 8; ++q) col[q * 32] = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
            } else if (direct) {
                // O / l -> bf16 -> out: 64-byte pieces, 8 rows per instruction
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint4 v;
                    v.x = pack_bf16x2(__uint_as_float(r[8 * q + 0]) * inv, __uint_as_float(r[8 * q + 1]) * inv);
                    v.y = pack_bf16x2(__uint_as_float(r[8 * q + 2]) * inv, __uint_as_float(r[8 * q + 3]) * inv);
                    v.z = pack_bf16x2(__uint_as_float(r[8 * q + 4]) * inv, __uint_as_float(r[8 * q + 5]) * inv);
                    v.w = pack_bf16x2(__uint_as_float(r[8 * q + 6]) * inv, __uint_as_float(r[8 * q + 7]) * inv);
                    mine[q ^ (lane & 7)] = v;
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int rr = i * 8 + (lane >> 2), q = lane & 3;
                    const uint4 x = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((q ^ (rr & 7)) << 4));
                    const int to = __shfl_sync(0xffffffffu, dst_row, rr);
                    if (to >= 0) *reinterpret_cast<uint4*>(out0 + to * out_stride + pc * 64 + q * 16) = x;
                }
            } else {
                if constexpr (FORM == kMergeHere) {
                    // unnormalised O of this segment -> its workspace slot: a warp writes 512 contiguous bytes per store
                    float4* const o = reinterpret_cast<float4*>(p.part_o) + slot_at * (2 * kBM) * (D / 4) +
                                      (size_t)pc * 8 * (2 * kBM) + qt * kBM + row;
                    if (live) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            o[q * (2 * kBM)] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]),
                                                           __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
                    }
                } else {
                    // unnormalised O of this segment -> its workspace slot: 128-byte pieces, 4 rows per instruction
#pragma unroll
                    for (int q = 0; q < 8; ++q) mine[q ^ (lane & 7)] = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                    __syncwarp();
                    uint8_t* const g0 = reinterpret_cast<uint8_t*>(p.part_o + (prow - lane) * D) + pc * 128;
                    const int n_live = it.nq - wrow0;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rr = i * 4 + (lane >> 3), q = lane & 7;
                        const uint4 x = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((q ^ (rr & 7)) << 4));
                        if (rr < n_live) *reinterpret_cast<uint4*>(g0 + (size_t)rr * D * 4 + q * 16) = x;
                    }
                }
            }
            __syncwarp();
        }
        if (!shared && !direct && live && ck == 0 && (!split || t == 0)) p.part_ml[prow] = make_float2(m, l);
    }
    ptx::fence_proxy_async_smem();      // the next segment's query tile arrives by TMA
}

// ---- item shared by a cluster: merge of the ranks' partial rows (softmax warps) ------------------------------------
//     out = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s
// straight from the CTAs' shared memories.  A unit is 8 columns of 32 rows, dealt over the ranks' warps; a lane
// owns one row, all ranks' loads are issued before the first use.
template <int D>
__device__ __forceinline__ void merge_cluster(const AttnParams& p, const SegInfo& it, const uint32_t smem, const int warp,
                                              const int lane) {
    using Cfg = AttnCfg<D>;
    const int n = p.cluster, rows = min(it.nq - it.q0, 2 * kBM);
    const int n_units = ((rows + 31) >> 5) * (D / 8);
    for (int u = it.slot + n * warp; u < n_units; u += n * kSoftmaxWarps) {
        const int rb = u / (D / 8), col = (u - rb * (D / 8)) * 8;
        const int row = rb * 32 + lane, qrow = it.q0 + row;
        const bool live = row < rows;
        int dst_row = -1;
        if (live) dst_row = p.out_rows != nullptr ? p.out_rows[(size_t)it.b * p.Nq_cap + qrow] : qrow;
        const uint32_t at_ml = smem + Cfg::kPartialMlAt + row * 8, at_o = smem + ((rb * (D / 4) + (col >> 2)) * 32 + lane) * 16;
        float w[kMaxCluster];                         // the ranks' maxima, then their weights
        float M = -INFINITY, L = 0.f;
        {
            float2 ml[kMaxCluster];
#pragma unroll
            for (int s = 0; s < kMaxCluster; ++s)
                if (s < n) ml[s] = ptx::ld_cluster_f2(ptx::map_rank(at_ml, s));
#pragma unroll
            for (int s = 0; s < kMaxCluster; ++s)
                if (s < n && ml[s].y > 0.f) M = fmaxf(M, ml[s].x);
#pragma unroll
            for (int s = 0; s < kMaxCluster; ++s) {
                w[s] = s < n && ml[s].y > 0.f ? fast_exp2(ml[s].x - M) : 0.f;     // a rank without keys carries no weight
                if (w[s] > 0.f) L = fmaf(w[s], ml[s].y, L);
            }
        }
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int s0 = 0; s0 < kMaxCluster; s0 += 4) {
            if (s0 >= n) break;
            float4 o[4][2];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (s0 + s < n) {
                    o[s][0] = ptx::ld_cluster_f4(ptx::map_rank(at_o, s0 + s));
                    o[s][1] = ptx::ld_cluster_f4(ptx::map_rank(at_o + 512, s0 + s));
                }
            }
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (s0 + s < n && w[s0 + s] > 0.f) {
                    const float v[8] = {o[s][0].x, o[s][0].y, o[s][0].z, o[s][0].w, o[s][1].x, o[s][1].y, o[s][1].z, o[s][1].w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[e] = fmaf(w[s0 + s], v[e], acc[e]);
                }
            }
        }
        const float inv = L > 0.f ? 1.f / L : 0.f;
        if (live && (dst_row < 0 || dst_row >= p.out_cap)) {   // destination out of range: dropped
            if (col == 0) record_status(p.dev_status, REGIONE_DEV_BOUNDS);
        } else if (live) {
            uint4 o;
            o.x = pack_bf16x2(acc[0] * inv, acc[1] * inv); o.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
            o.z = pack_bf16x2(acc[4] * inv, acc[5] * inv); o.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
            *reinterpret_cast<uint4*>(p.out + (((size_t)it.b * p.out_cap + dst_row) * p.H + it.h) * D + col) = o;
        }
    }
}

// ---- cut item: its first share merges the later shares' partial rows into its own (softmax warps) -----------------
//     out = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s
// Its own rows are in shared memory, the others in their slots of the workspace.  The first share reaches the item at
// the end of its range and the others begin with it, so it rarely waits.  A warp merges pieces of 32 columns of 32 rows,
// a lane owns one row; the loads of the usual single other share are all under way before the first use.  The output
// goes through the piece's own place in shared memory, so that stores cover whole sectors (a lane storing its own
// row's chunks: 12600 cycles for a pair of tiles, this way 6500).
template <int D>
__device__ __forceinline__ void merge_shares(const AttnParams& p, const SegInfo& it, uint8_t* smem_gen, const int warp,
                                             const int lane, volatile int* abort_flag) {
    using Cfg = AttnCfg<D>;
    const int n = it.n_slots, rb = warp >> 1;
    const int row = rb * 32 + lane, qrow = it.q0 + row;
    const bool live = qrow < it.nq;                // (dead rows' entries are not written and may hold anything)
    int dst_row = -1;
    if (live) dst_row = p.out_rows != nullptr ? p.out_rows[(size_t)it.b * p.Nq_cap + qrow] : qrow;
    if (live && (dst_row < 0 || dst_row >= p.out_cap)) {       // destination out of range: dropped
        if ((warp & 1) == 0) record_status(p.dev_status, REGIONE_DEV_BOUNDS);
        dst_row = -1;
    }
    const float2 own = *(reinterpret_cast<const float2*>(smem_gen + Cfg::kPartialMlAt) + row);
    const size_t slot1 = (size_t)it.slot_at, step = (size_t)it.slot_step * (2 * kBM);
    const float2* const others_ml = p.part_ml + slot1 * (2 * kBM) + row;
    uint8_t* const out0 = reinterpret_cast<uint8_t*>(p.out) + (((size_t)it.b * p.out_cap) * p.H + it.h) * D * 2;
    const size_t out_stride = (size_t)p.H * D * 2;
    if (!wait_shares(p, n - 1, it.share_step, lane, abort_flag)) return;
    if (rb * 32 >= it.nq - it.q0) return;
#pragma unroll 1
    for (int pc = (warp & 1) * (D / 64); pc < ((warp & 1) + 1) * (D / 64); ++pc) {
        const float4* const others = reinterpret_cast<const float4*>(p.part_o) + (slot1 * (D / 4) + pc * 8) * (2 * kBM) + row;
        uint8_t* const place = smem_gen + (rb * (D / 4) + pc * 8) * 512;      // 32 columns of 32 rows, fp32
        float4 x[8], acc[8];
        float2 ml = __ldcg(others_ml);
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = __ldcg(others + q * (2 * kBM));
        // (a share without live keys in a row carries no weight)
        float M = own.y > 0.f ? own.x : -INFINITY;
        if (ml.y > 0.f) M = fmaxf(M, ml.x);
        for (int sl = 1; sl < n - 1; ++sl) {
            const float2 o = __ldcg(others_ml + sl * step);
            if (o.y > 0.f) M = fmaxf(M, o.x);
        }
        float w = own.y > 0.f ? fast_exp2(own.x - M) : 0.f;
        float L = w > 0.f ? w * own.y : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 o = reinterpret_cast<const float4*>(place)[q * 32 + lane];
            acc[q] = w > 0.f ? make_float4(w * o.x, w * o.y, w * o.z, w * o.w) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll 1
        for (int sl = 1;; ++sl) {
            if (ml.y > 0.f) {
                w = fast_exp2(ml.x - M);
                L = fmaf(w, ml.y, L);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    acc[q].x = fmaf(w, x[q].x, acc[q].x);
                    acc[q].y = fmaf(w, x[q].y, acc[q].y);
                    acc[q].z = fmaf(w, x[q].z, acc[q].z);
                    acc[q].w = fmaf(w, x[q].w, acc[q].w);
                }
            }
            if (sl >= n - 1) break;
            ml = __ldcg(others_ml + sl * step);
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = __ldcg(others + sl * step * (D / 4) + q * (2 * kBM));
        }
        const float inv = L > 0.f ? 1.f / L : 0.f;
        __syncwarp();                              // (every lane has read its own rows' chunks)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            reinterpret_cast<uint4*>(place)[lane * 4 + (q ^ ((lane >> 1) & 3))] =
                make_uint4(pack_bf16x2(acc[2 * q].x * inv, acc[2 * q].y * inv),
                           pack_bf16x2(acc[2 * q].z * inv, acc[2 * q].w * inv),
                           pack_bf16x2(acc[2 * q + 1].x * inv, acc[2 * q + 1].y * inv),
                           pack_bf16x2(acc[2 * q + 1].z * inv, acc[2 * q + 1].w * inv));
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {              // 64 bytes of a row, 8 rows per instruction
            const int rr = i * 8 + (lane >> 2), q = lane & 3;
            const uint4 v = reinterpret_cast<const uint4*>(place)[rr * 4 + (q ^ ((rr >> 1) & 3))];
            const int to = __shfl_sync(0xffffffffu, dst_row, rr);
            if (to >= 0) *reinterpret_cast<uint4*>(out0 + to * out_stride + pc * 64 + q * 16) = v;
        }
    }
}

// ---- cache refresh: copies of the retained rows, by a warp of their own ------------------------------------
// The rows travel as bulk copies (one per lane: global -> slot of shared memory -> cache), so the copies take
// no registers, few issue slots and no time of the tensor cores, and the warp may block on them.  (A first version
// ran them from the producer warp between its loads: every wait for a slot delayed a key tile, and 194 MB of copies
// cost the attention of 819 queries as much as a store kernel ahead of it.)  The launch's rows (K of every request,
// then V, of one list and then the other) are cut into equal contiguous shares, one per CTA, whatever attention work the CTA has.  An item is one
// row, or a slot's length of it where a row is longer than that; a batch is up to `per_unit` consecutive items of one
// request, lane i moving item i.  Beside the walks one batch at a time fills the corner of shared memory that is left
// (5 rows of 24 x 128): the warp gets few issue slots there, and several slots of a row each with the same number of
// rows in flight took 2660 cycles a row.  Over the idle tiles two batches alternate.
struct CachePump {
    const StoreParams* sp;
    AttnCtrl* ctrl;
    const AttnParams* p;
    int row_bytes, item_bytes, per_row; // items per row
    uint32_t slots;                     // shared-memory address of slot 0
    int n_slots, slot_bytes, per_unit;
    int x, b, i, run, live_rows;        // cursor of the loads: destination, request, item, items of the run, source rows
    int left;                           // items not yet loaded
    int head, tail;                     // units loaded / stored through the present slots
    int win;                            // first item of the window of list entries held, one per lane:
    int row, before;                    // the entry of item win + lane and the one ahead of it,
    int row_next, before_next;          // the same for the window behind it (fetched long before it is needed)

    __device__ __forceinline__ int kept(int list, int req, bool report) const {
        if (p->all_rows > 0 && rows_apart(p->n_q[req], sp->n[0][req], p->Nq_cap, p->all_rows)) return 0;   // (copied ahead)
        const int nk = sp->n[list][req], cap = sp->cap[list];
        if (nk >= 0 && nk <= cap) return nk;
        if (report && blockIdx.x == 0) record_status(p->dev_status, REGIONE_DEV_BOUNDS);
        return nk < 0 ? 0 : cap;
    }
    __device__ __forceinline__ int source_rows(int req) const {
        return p->all_rows > 0 ? p->all_rows : min(p->n_fresh[req], sp->src_cap);
    }
    __device__ __forceinline__ int row_of(int item) const { return per_row > 1 ? item / per_row : item; }
    // from an item index behind the runs x, b to the run that holds it (a request without rows stores nothing)
    __device__ __forceinline__ void open_run() {
        for (;;) {
            live_rows = source_rows(b);
            run = live_rows > 0 ? kept(x >> 1, b, false) * per_row : 0;
            if (i < run) return;
            i -= run;
            if (++b == p->B) { b = 0; ++x; }
        }
    }
    // list entries of the 32 items from `first` on (those of the present run and share)
    __device__ __forceinline__ void fetch(int first, int lane, int& r, int& ahead) const {
        r = ahead = -1;
        if (first + lane < min(run, i + left)) {
            const int32_t* keep = sp->rows[x >> 1] + (size_t)b * sp->cap[x >> 1];
            const int j = row_of(first + lane);
            r = keep[j];
            if (j > 0) ahead = keep[j - 1];
        }
    }
    __device__ __forceinline__ void open_window(int lane) {
        win = i;
        fetch(win, lane, row, before);
        fetch(win + 32, lane, row_next, before_next);
    }
    // `n` slots in `bytes` of shared memory
    __device__ __forceinline__ void use_slots(uint32_t at, int bytes, int n, int lane) {
        slots = at;
        n_slots = n;
        slot_bytes = (bytes / n) & ~127;
        per_unit = min(32, slot_bytes / item_bytes);
        head = tail = 0;
        if (lane < n_slots) ptx::mbar_init(ptx::smem_addr(&ctrl->copy_full[lane]), 1);
        ptx::fence_barrier_init();
        __syncwarp();
    }
    __device__ __forceinline__ void begin(const AttnParams& prm, const StoreParams& s, AttnCtrl* c, int d, int longest, int lane) {
        sp = &s; ctrl = c; p = &prm;
        row_bytes = prm.H * d * 2;
        per_row = (row_bytes + longest - 1) / longest;
        item_bytes = min(row_bytes, longest);
        long long total = 0;
        for (int l = 0; l < s.n_lists; ++l)
            for (int r = 0; r < prm.B; ++r) {
                const int nk = kept(l, r, lane == 0);
                if (source_rows(r) > 0) total += 2LL * nk * per_row;
            }
        const long long per = (total + gridDim.x - 1) / gridDim.x, first = per * blockIdx.x;
        left = (int)max(0LL, min(per, total - first));
        x = b = 0;
        i = (int)first;
        if (left > 0) {
            open_run();
            open_window(lane);
        }
    }
    __device__ __forceinline__ bool store_oldest(int lane) {
        const int slot = n_slots > 1 ? tail & 1 : 0;
        const bool landed = wait_bar(ptx::smem_addr(&ctrl->copy_full[slot]), (n_slots > 1 ? tail >> 1 : tail) & 1, &ctrl->copy_abort,
                                     p->dev_status, p->timeout_cycles);
        if (!__all_sync(0xffffffffu, landed)) return false;
        if ((ctrl->copy_valid[slot] >> lane) & 1u) {
            const int at = ctrl->copy_item[slot] + lane, j = row_of(at), off = (at - j * per_row) * item_bytes;
            ptx::bulk_store(ctrl->copy_dst[slot] + (size_t)j * row_bytes + off, slots + slot * slot_bytes + lane * item_bytes,
                            min(item_bytes, row_bytes - off));
        }
        ptx::bulk_commit();
        ++tail;
        return true;
    }
    __device__ __forceinline__ void load_next(int lane) {
        // (the batch that this slot held last has been read out of shared memory)
        ptx::bulk_wait_read<0>();
        __syncwarp();
        const int n = min(min(per_unit, win + 32 - i), min(run - i, left));
        const int at = min(i - win + lane, 31);
        const int my_row = __shfl_sync(0xffffffffu, row, at), ahead = __shfl_sync(0xffffffffu, before, at);
        const bool ok = my_row >= 0 && my_row < live_rows && my_row > ahead;
        if (lane < n && !ok) record_status(p->dev_status, REGIONE_DEV_BOUNDS);
        const uint32_t valid = __ballot_sync(0xffffffffu, lane < n && ok);
        const int slot = n_slots > 1 ? head & 1 : 0;
        const uint32_t bar = ptx::smem_addr(&ctrl->copy_full[slot]);
        const int off = (i + lane - row_of(i + lane) * per_row) * item_bytes;
        const int bytes = (valid >> lane) & 1u ? min(item_bytes, row_bytes - off) : 0;
        const int unit_bytes = __reduce_add_sync(0xffffffffu, bytes);
        if (lane == 0) {
            ctrl->copy_valid[slot] = valid;
            ctrl->copy_item[slot] = i;
            ctrl->copy_dst[slot] = sp->dst[x] + (size_t)b * sp->cap[x >> 1] * row_bytes;
            ptx::mbar_arrive_expect_tx(bar, unit_bytes);
        }
        __syncwarp();
        if (bytes > 0)
            ptx::bulk_load(slots + slot * slot_bytes + lane * item_bytes,
                           sp->src[x & 1] + ((size_t)b * sp->src_cap + my_row) * row_bytes + off, bytes, bar);
        ++head;
        left -= n;
        i += n;
        if (left > 0) {
            if (i >= run) {
                open_run();
                open_window(lane);
            } else if (i == win + 32) {
                win = i;
                row = row_next;
                before = before_next;
                fetch(win + 32, lane, row_next, before_next);
            }
        }
    }
    // Moves the CTA's rows: through a corner of shared memory beside the walks, through the idle tiles once they are
    // over.  False when a copy did not land within the bound of the waits.
    template <int D>
    __device__ __forceinline__ bool run_all(uint32_t smem, int lane) {
        using Cfg = AttnCfg<D>;
        bool wide = false;
        if (left > 0) use_slots(smem + Cfg::kCopyAt, Cfg::kCopyBytes, 1, lane);
        while (left > 0) {
            if (!wide && __any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&ctrl->walks_done) != 0)) {
                while (tail < head)
                    if (!store_oldest(lane)) return false;
                ptx::bulk_wait_read<0>();
                __threadfence_block();
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane < n_slots) ptx::mbar_inval(ptx::smem_addr(&ctrl->copy_full[lane]));
                __syncwarp();
                use_slots(smem, Cfg::kTailBytes, kCopySlots, lane);
                wide = true;
            }
            if (head - tail < n_slots) load_next(lane);
            else if (!store_oldest(lane)) return false;
        }
        while (tail < head)
            if (!store_oldest(lane)) return false;
        return true;
    }
};

// ---- TMA producer of one segment (whole warp; lane 0 issues) ----------------------------------------------
template <int D, bool STORE>
__device__ __forceinline__ void load_segment(const CUtensorMap* tm_q, const CUtensorMap* tm_kf, const CUtensorMap* tm_vf,
                                             const CUtensorMap* tm_kc, const CUtensorMap* tm_vc, const CUtensorMap* tm_ka,
                                             const CUtensorMap* tm_va, const AttnParams& p, AttnCtrl* ctrl, const SegInfo& it,
                                             const uint32_t smem, const int lane) {
    using Cfg = AttnCfg<D>;
    constexpr int kTileBytes = Cfg::kTileBytes;
    const int n_tiles = it.n_tiles;
    if (n_tiles == 0) return;
    const int ntq = it.nq - it.q0 > kBM ? 2 : 1;
    const bool split = ntq == 1 && n_tiles >= 2;
    const int n_stages = split ? Cfg::lone_stages(STORE) : Cfg::kStages;
    const uint32_t ring = smem + (split ? 1 : 2) * kTileBytes;
    const int nt_c = it.nt_c, j_first = it.j_first, h = it.h, b = it.b;
    if (STORE && it.apart) { tm_kf = tm_ka; tm_vf = tm_va; }
    if (lane == 0) {
        ptx::prefetch_tensormap(tm_q);
        ptx::prefetch_tensormap(j_first < nt_c ? tm_kc : tm_kf);
        ptx::prefetch_tensormap(j_first < nt_c ? tm_vc : tm_vf);
        const uint32_t qbar = ptx::smem_addr(&ctrl->q_full);
        ptx::mbar_arrive_expect_tx(qbar, ntq * kTileBytes);
        for (int t = 0; t < ntq; ++t)
            for (int hf = 0; hf < Cfg::kHalves; ++hf)
                ptx::tma_load_4d(smem + t * kTileBytes + hf * kHalfBytes, tm_q, qbar, hf * 64, h, it.q0 + t * kBM, b);
    }
    int stage = 0, use = 0;
    for (int i = 0; i < 2 * n_tiles; ++i) {
        const int j = j_first + (i >> 1), is_v = i & 1;
        if (use > 0) {
            const uint32_t bar = ptx::smem_addr(&ctrl->kv_empty[stage]);
            if (!wait_bar(bar, (use - 1) & 1, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
        }
        if (lane == 0) {
            const bool cached = j < nt_c;
            const CUtensorMap* map = cached ? (is_v ? tm_vc : tm_kc) : (is_v ? tm_vf : tm_kf);
            const uint32_t bar = is_v ? v_landing(ctrl, split, n_stages, i >> 1).bar : ptx::smem_addr(&ctrl->kv_full[stage]);
            ptx::mbar_arrive_expect_tx(bar, kTileBytes);
            const int row = (cached ? j : j - nt_c) * kBN;
            for (int hf = 0; hf < Cfg::kHalves; ++hf) {
                const uint32_t dst = ring + stage * kTileBytes + hf * kHalfBytes;
                if (p.kv_once) ptx::tma_load_4d_once(dst, map, bar, hf * 64, h, row, b);
                else ptx::tma_load_4d(dst, map, bar, hf * 64, h, row, b);
            }
        }
        __syncwarp();
        if (++stage == n_stages) { stage = 0; ++use; }
    }
}

// ---- issuer of the S products of both query tiles (whole warp, one elected lane issues) ------------------
// S = Q_t K_j^T goes to ONE staging buffer in tensor memory that the two query tiles share: a product is
// issued as soon as its K tile has landed and the buffer's previous contents have been read into registers
// by the softmax warps they were computed for.  It does not have to wait for the P*V products of its own
// tile, which read P from a place of their own.
template <int D, bool STORE>
__device__ __forceinline__ void issue_s_segment(const AttnParams& p, AttnCtrl* ctrl, const SegInfo& it, const uint32_t smem,
                                                const uint32_t tmem) {
    using Cfg = AttnCfg<D>;
    constexpr int kTileBytes = Cfg::kTileBytes;
    const int n_tiles = it.n_tiles;
    if (n_tiles == 0) return;
    const int ntq = it.nq - it.q0 > kBM ? 2 : 1;
    const bool split = ntq == 1 && n_tiles >= 2;
    const int n_stages = split ? Cfg::lone_stages(STORE) : Cfg::kStages;
    constexpr uint32_t idesc_s = ptx::idesc_bf16_f32(kBM, kBN, false);
    constexpr uint32_t hi_k = ptx::smem_desc_hi_sw128(1024);   // 8-row groups 1024 B apart
    const uint32_t k_lo = ptx::smem_desc_lo(smem + (split ? 1 : 2) * kTileBytes, 16);
    const uint32_t q_base = ptx::smem_desc_lo(smem, 16);
    if (!wait_bar(ptx::smem_addr(&ctrl->q_full), 0, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
    int n_issued = 0;                                   // products so far = uses of the staging buffer
    int sk = 0, use = 0;
    for (int jl = 0; jl < n_tiles; ++jl) {
        if (!wait_bar(ptx::smem_addr(&ctrl->kv_full[sk]), use & 1, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
        // the roles this key tile feeds: both query tiles, or one half of a lone query tile
        const int t_first = split ? (jl & 1) : 0, t_last = split ? (jl & 1) : ntq - 1;
        for (int t = t_first; t <= t_last; ++t) {
            if (n_issued > 0 && !wait_bar(ptx::smem_addr(&ctrl->s_free), (n_issued - 1) & 1, &ctrl->abort_flag,
                                          p.dev_status, p.timeout_cycles))
                return;
            ptx::tc_fence_after_sync();
            if (ptx::elect_one()) {
                const uint32_t q_lo = q_base + (((split ? 0 : t) * kTileBytes) >> 4);
                const uint32_t b0 = k_lo + ((sk * kTileBytes) >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t off = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
                    ptx::mma_ss(tmem, ptx::smem_desc_join(q_lo + off, hi_k),
                                ptx::smem_desc_join(b0 + off, hi_k), idesc_s, kk > 0);
                }
                ptx::mma_commit(ptx::smem_addr(&ctrl->s_full[t]));
                ptx::mma_commit(ptx::smem_addr(&ctrl->kv_empty[sk]));
            }
            __syncwarp();
            ++n_issued;
        }
        sk += 2;
        if (sk >= n_stages) { sk -= n_stages; ++use; }
    }
}

// ---- issuer of the P*V products of both query-tile roles (whole warp, one elected lane issues) --------------
// The roles take turns, as their logits do in the shared S buffer: a pair's tiles on every key tile, a lone tile's
// roles on alternate key tiles.
template <int D, bool STORE>
__device__ __forceinline__ void issue_pv_segment(const AttnParams& p, AttnCtrl* ctrl, const SegInfo& it, const uint32_t smem,
                                                 const uint32_t tmem, const int lane, const int mode) {
    using Cfg = AttnCfg<D>;
    constexpr int kTileBytes = Cfg::kTileBytes;
    const int n_tiles = it.n_tiles;
    const bool pair = it.nq - it.q0 > kBM;
    const bool split = !pair && n_tiles >= 2;
    const int n_stages = split ? Cfg::lone_stages(STORE) : Cfg::kStages;
    const TileKeys keys(it);
    const int n_turns = pair ? 2 * n_tiles : n_tiles;
    constexpr uint32_t idesc_pv = ptx::idesc_bf16_f32(kBM, D, true);
    constexpr uint32_t hi_k = ptx::smem_desc_hi_sw128(1024);   // 8-key groups 1024 B apart
    // V is MN-major: 64-column boxes kHalfBytes apart (LBO), 8-key groups 1024 B apart (SBO)
    const uint32_t v_lo = ptx::smem_desc_lo(smem + (split ? 1 : 2) * kTileBytes, kHalfBytes);
    for (int n = 0; n < n_turns; ++n) {
        const int t = n & 1, j = n >> 1, jl = pair ? j : n;
        const int sv = (2 * jl + 1) % n_stages;
        const VLanding vl = v_landing(ctrl, split, n_stages, jl);
        if ((!pair || t == 0) && !wait_bar(vl.bar, vl.phase & 1, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
        if (mode == kMaxOnly) {                     // no products in this pass: the stage is given back
            if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&ctrl->kv_empty[sv]));
            continue;
        }
        const uint32_t tPt = tmem + kBN + t * (kBN / 2), tOt = tmem + 256 + t * D;
        // O_t (+)= P_t[chunk] V[64 chunk .. 64 chunk + 64) : A from tensor memory (bf16 pairs,
        // 8 columns per 16 keys)
        auto issue_pv = [&](int chunk, bool accumulate) {
            const uint32_t b0 = v_lo + ((sv * kTileBytes + chunk * (kBH / 16) * 2048) >> 4);
#pragma unroll
            for (int kk = 0; kk < kBH / 16; ++kk)
                ptx::mma_ts(tOt, tPt + chunk * (kBH / 2) + kk * 8,
                            ptx::smem_desc_join(b0 + ((kk * 2048) >> 4), hi_k), idesc_pv,
                            (accumulate || kk > 0) ? 1u : 0u);
        };
        if (!wait_bar(ptx::smem_addr(&ctrl->p_full[t][0]), j & 1, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
        ptx::tc_fence_after_sync();
        if (ptx::elect_one()) {
            issue_pv(0, j > 0);
            ptx::mma_commit(ptx::smem_addr(&ctrl->pv_half[t]));
        }
        __syncwarp();
        if (!wait_bar(ptx::smem_addr(&ctrl->p_full[t][1]), j & 1, &ctrl->abort_flag, p.dev_status, p.timeout_cycles)) return;
        ptx::tc_fence_after_sync();
        if (ptx::elect_one()) {
            if (keys(jl) > kBH) issue_pv(1, true);
            ptx::mma_commit(ptx::smem_addr(&ctrl->pv_done[t]));
            ptx::mma_commit(ptx::smem_addr(&ctrl->kv_empty[sv]));
            if (n + 2 >= n_turns) ptx::mma_commit(ptx::smem_addr(&ctrl->o_final[t]));      // (the role's last arrival)
        }
        __syncwarp();
    }
}

// ---- the share of one CTA: plan and next segment (one warp computes them, the others read SegInfo) --------
template <bool IN_PLACE, bool SPREAD>
struct ShareCursor {
    ShareWalk<IN_PLACE, SPREAD> walk;
    bool first;
    // The only segment of a CTA whose item is shared by a cluster: rank r of n takes the key tiles
    // [r * nt / n, (r + 1) * nt / n) (possibly none) and reads back its part of the rows.
    __device__ __forceinline__ void of_cluster(const AttnParams& p, SegInfo* out, const int lane, bool* bad) {
        int idx = blockIdx.x / p.cluster;
        const int rank = blockIdx.x - idx * p.cluster;
        ReqShape r = req_shape<IN_PLACE>(p, 0, bad);
        int b = 0;
        while (b + 1 < p.B && idx >= p.H * r.np) {
            idx -= p.H * r.np;
            r = req_shape<IN_PLACE>(p, ++b, bad);
        }
        first = false;
        if (lane != 0) return;
        out->live = idx < p.H * r.np;
        if (!out->live) return;
        out->b = b;
        out->h = idx / r.np;
        out->q0 = (idx - out->h * r.np) * (2 * kBM);
        out->nq = r.nq; out->nt_c = r.nt_c; out->nt = r.nt; out->nc = r.nc; out->nf = r.nf;
        out->j_first = rank * r.nt / p.cluster;
        out->n_tiles = (rank + 1) * r.nt / p.cluster - out->j_first;
        out->slot = rank; out->n_slots = p.cluster; out->slot_at = 1; out->slot_step = out->share_step = 1;
        if (IN_PLACE) out->apart = r.apart;
    }
    // This CTA's share of the plan.
    __device__ __forceinline__ void of_plan(const AttnParams& p, bool* bad) {
        walk.begin(p, gridDim.x, blockIdx.x, bad);
        first = true;
    }
    // The next live segment of the share into *out (out->live = 0 when the share ends).
    template <int FORM>
    __device__ __forceinline__ void next(const AttnParams& p, SegInfo* out, const int lane) {
        Segment it;
        while (walk.next(p, gridDim.x, blockIdx.x, it)) {
            if (FORM == kMergeKernel && first && !it.in_wave) {
                // tell the merge kernel which item the start of this share cuts
                if (lane == 0) {
                    CutItem ci;
                    ci.valid = (it.n_steps > 0 && it.n_slots >= 2 && it.slot == 1) ? 1 : 0;
                    ci.b = it.b; ci.h = it.h; ci.qp = it.qp; ci.n_slots = it.n_slots; ci.nq = it.r.nq;
                    ci.slot_at = it.slot_at; ci.slot_step = it.slot_step;
                    p.cut[share_of(gridDim.x, blockIdx.x)] = ci;
                }
                first = false;
            }
            if (it.n_steps == 0) continue;
            if (lane == 0) {
                out->b = it.b; out->h = it.h; out->q0 = it.qp * (2 * kBM); out->nq = it.r.nq;
                out->j_first = it.j_first; out->n_tiles = it.r.nt == 0 ? 0 : it.n_steps;
                out->nt_c = it.r.nt_c; out->nt = it.r.nt; out->nc = it.r.nc; out->nf = it.r.nf;
                out->slot = it.slot; out->n_slots = it.n_slots;
                out->slot_at = it.slot_at; out->slot_step = it.slot_step;
                out->share_step = walk.step;
                if (IN_PLACE) out->apart = it.r.apart;
                out->live = 1;
            }
            return;
        }
        if (lane == 0) {
            if (FORM == kMergeKernel && first) p.cut[share_of(gridDim.x, blockIdx.x)].valid = 0;
            out->live = 0;
        }
        first = false;
    }
};

template <int D, bool STORE, int FORM, bool SPREAD>
__device__ __forceinline__ void attention_kernel_body(const CUtensorMap& tm_q, const CUtensorMap& tm_kf,
                                                      const CUtensorMap& tm_vf, const CUtensorMap& tm_kc,
                                                      const CUtensorMap& tm_vc, const CUtensorMap& tm_ka,
                                                      const CUtensorMap& tm_va, const AttnParams& p, const StoreParams& sp) {
    using Cfg = AttnCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t smem = ptx::smem_addr(smem_raw);     // 2 query tiles, then the ring of K/V stages
    AttnCtrl* ctrl = reinterpret_cast<AttnCtrl*>(smem_raw + Cfg::kSmemTiles);
    volatile int* abort_flag = &ctrl->abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == kWarpPv) {
        ptx::tmem_alloc(ptx::smem_addr(&ctrl->tmem_base), 512);
        ptx::tmem_relinquish();
    }
    grid_dependency_wait();                             // (everything below reads the launch's inputs)
    grid_launch_dependents();                           // the next kernel may queue up behind this CTA
    // The warp that loads K and V also plans: it is done with a segment well ahead of the others.  In a refreshing launch that
    // minds the order its cursor lies in shared memory between two segments: kept in registers, its fields cost the issuing
    // loops spills (2048 of 8448 rows refreshed 235.0 -> 230.8 us; 819 of them read 121.2 -> 124.1).
    using Cursor = ShareCursor<STORE, SPREAD>;
    static_assert(sizeof(Cursor) <= sizeof(ctrl->cursor), "cursor");
    Cursor* const kept = reinterpret_cast<Cursor*>(ctrl->cursor);
    Cursor cur;
    if (warp == kWarpLoad) {
        bool bad = false;
        if constexpr (FORM == kMergeCluster) {
            cur.of_cluster(p, &ctrl->seg[0], lane, &bad);
            if (lane == 0) {
                ctrl->seg[1].live = 0;
                ptx::mbar_init(ptx::smem_addr(&ctrl->peers_ready), p.cluster);
                ptx::mbar_init(ptx::smem_addr(&ctrl->peers_done), p.cluster);
                ptx::fence_barrier_init();
            }
        } else {
            cur.of_plan(p, &bad);
            cur.template next<FORM>(p, &ctrl->seg[0], lane);
            if (STORE && SPREAD && lane == 0) *kept = cur;
        }
        if (bad && blockIdx.x == 0 && lane == 0) record_status(p.dev_status, REGIONE_DEV_BOUNDS);
        if (lane == 0) ctrl->abort_flag = 0;
    }

    // The two sides of the register split walk the same segments: the softmax warpgroups hold a chunk of 64
    // logits per thread, the producer / issuer warpgroup gives registers up.  CTA-wide barriers around a
    // segment: `set-up` (control block's barriers initialised, next segment known) and `end` (every role is
    // done with shared and tensor memory).
    auto walk_sync = [&]() {
        asm volatile("bar.sync %0, %1;" ::"n"(kWalkBarrier), "n"(kWalkThreads) : "memory");
    };
    auto set_up = [&](const SegInfo& it) {
        // thread i sets barrier i of the control block up
        const int ntq = it.nq - it.q0 > kBM ? 2 : 1;
        const bool split = ntq == 1 && it.n_tiles >= 2;
        if (threadIdx.x < kNumBarriers) {
            const int i = threadIdx.x;
            int count = 1;                                               // q_full, kv_full, s_full, commits
            if (i >= kBarKvEmpty && i < kBarSFull) count = split ? 1 : ntq;      // commits per stage
            else if (i >= kBarPFull && i < kBarOFinal) count = kBM / 32;         // one arrival per warp
            else if (i == kBarSFree) count = 2 * (kBM / 32);             // (v_full: one, like kv_full)
            ptx::mbar_init(ptx::smem_addr(&ctrl->q_full + i), count);
            ptx::fence_barrier_init();
        }
        if (threadIdx.x == 0) ctrl->redo = 0;
        ptx::tc_fence_before_sync();
        walk_sync();
        ptx::tc_fence_after_sync();
    };
    auto tear_down = [&]() {
        ptx::tc_fence_before_sync();
        walk_sync();
        ptx::tc_fence_after_sync();
        // (after a wait that ran out, loads and products may still be on their way to their barriers: those stay)
        if (threadIdx.x < kNumBarriers && !*abort_flag) ptx::mbar_inval(ptx::smem_addr(&ctrl->q_full + threadIdx.x));
    };
    // what to do after a walk: repeat the segment (new mode) or go on
    auto repeat = [&](int& mode) {
        const bool redo = mode == kWalk && *reinterpret_cast<volatile int*>(&ctrl->redo) != 0;
        const int next_mode = redo ? kMaxOnly : mode == kMaxOnly ? kExact : kWalk;
        const bool again = next_mode != kWalk;
        mode = next_mode;
        walk_sync();                                // (redo has been read by everyone)
        return again;
    };
    if (STORE && threadIdx.x == 0) ctrl->walks_done = 0;
    __syncwarp();
    if (FORM == kMergeCluster) ptx::cluster_sync();             // (the peers' barriers are initialised)
    __syncthreads();
    const uint32_t tmem = ctrl->tmem_base;
    int k = 0, mode = kWalk;
    if (warp >= kSoftmaxWarps) {
        ptx::reg_dealloc<64>();
        if (warp == kWarpCopy) {
            if constexpr (STORE) {
                CachePump pump;
                if (lane == 0) ctrl->copy_abort = 0;
                __syncwarp();
                pump.begin(p, sp, ctrl, D, Cfg::kCopyBytes / 4, lane);
                if (!pump.run_all<D>(smem, lane)) {
                    // give copies that are still in flight time to land before shared memory is given back
                    const long long t0 = clock64();
                    while (clock64() - t0 < 2000000LL) __nanosleep(1000);
                }
                ptx::bulk_wait_all();
            }
            return;
        }
        while (ctrl->seg[k].live && !*abort_flag) {
            const SegInfo& it = ctrl->seg[k];
            set_up(it);
            if (warp == kWarpLoad) {
                load_segment<D, STORE>(&tm_q, &tm_kf, &tm_vf, &tm_kc, &tm_vc, &tm_ka, &tm_va, p, ctrl, it, smem, lane);
                // (the next segment is planned while the last tiles are on their way and multiplied: ahead of the end of this one
                // by the issuer of S, four requests of 205 to 1638 of 8448 rows took 432 us instead of 418)
                if (FORM != kMergeCluster && mode == kWalk) {
                    if (STORE && SPREAD) cur = *kept;
                    cur.template next<FORM>(p, &ctrl->seg[k ^ 1], lane);
                    if (STORE && SPREAD) {
                        __syncwarp();
                        if (lane == 0) *kept = cur;
                        __syncwarp();
                    }
                }
            } else if (warp == kWarpS) {
                issue_s_segment<D, STORE>(p, ctrl, it, smem, tmem);
            } else {
                issue_pv_segment<D, STORE>(p, ctrl, it, smem, tmem, lane, mode);
            }
            tear_down();
            if (!repeat(mode)) k ^= 1;
        }
    } else {
        ptx::reg_alloc<104>();
        float m_known = -INFINITY;
        bool publish = false, merges = false;   // the last segment's rows: (thread 0) in the workspace, the first share
                                                // not told yet; in shared memory, to be merged with the later shares'
        auto tell = [&]() {
            // (every warp's rows are ordered before this by the barriers of tear_down and repeat)
            if (publish && !*abort_flag) ptx::st_release_u64(p.ready + share_of(gridDim.x, blockIdx.x), p.epoch);
            publish = false;
        };
        while (ctrl->seg[k].live && !*abort_flag) {
            set_up(ctrl->seg[k]);
            if (FORM == kMergeHere) tell();                   // (while the first key tiles are on their way)
            softmax_segment<D, STORE, FORM>(p, ctrl, ctrl->seg[k], smem_raw, tmem, warp, lane, mode, m_known);
            tear_down();
            const bool cut = FORM == kMergeHere && ctrl->seg[k].n_slots > 1, head = ctrl->seg[k].slot == 0;
            if (!repeat(mode)) {
                publish = cut && !head && threadIdx.x == 0;
                merges = cut && head;               // (the item goes on behind this share: nothing follows here)
                k ^= 1;
            }
        }
        if (FORM == kMergeHere) tell();
        if (FORM == kMergeHere && merges) {
            const SegInfo& it = ctrl->seg[k ^ 1];
            if (!*abort_flag) merge_shares<D>(p, it, smem_raw, warp, lane, abort_flag);
            // every warp has seen the flags: they are left as no launch's epoch (a graph replays the launch with the
            // one it has)
            named_barrier(3, 32 * kSoftmaxWarps);
            if (threadIdx.x < it.n_slots - 1) p.ready[share_of(gridDim.x, blockIdx.x) + (1 + threadIdx.x) * it.share_step] = 0;
        }
    }

    // ================= item shared by a cluster =================
    if (FORM == kMergeCluster && ctrl->seg[0].live) {
        // (tear_down's barrier has ordered every warp's partial rows before this)
        const uint32_t ready = ptx::smem_addr(&ctrl->peers_ready), done = ptx::smem_addr(&ctrl->peers_done);
        if (warp == 0 && lane < p.cluster && !*abort_flag) ptx::mbar_arrive_cluster(ptx::map_rank(ready, lane));
        bool ok = !*abort_flag;
        if (warp < kSoftmaxWarps) {
            if (ok) ok = wait_bar_cluster(ready, abort_flag, p.dev_status, p.timeout_cycles);
            if (ok) merge_cluster<D>(p, ctrl->seg[0], smem, warp, lane);
        }
        if (STORE) {
            // (the copies of rows take the tiles over, once every peer has read them)
            walk_sync();
            if (warp == 0 && lane < p.cluster && !*abort_flag) ptx::mbar_arrive_cluster(ptx::map_rank(done, lane));
            if (!*abort_flag) wait_bar_cluster(done, abort_flag, p.dev_status, p.timeout_cycles);
        }
    }

    // ================= teardown =================
    if (*abort_flag) {
        if (FORM == kMergeHere && threadIdx.x == 0) p.ready[gridDim.x] = p.epoch;
        // give copies and MMAs that are still in flight time to land before tensor memory and
        // shared memory are given back
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) __nanosleep(1000);
    }
    ptx::tc_fence_before_sync();
    walk_sync();
    if (warp == kWarpPv) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem, 512);
    }
    // (every role's writes to the tiles are ordered before this by its proxy fence and the barrier above)
    if (STORE && threadIdx.x == 0) {
        __threadfence_block();
        *reinterpret_cast<volatile int*>(&ctrl->walks_done) = 1;
    }
    // A CTA's shared memory stays until no peer reads it or arrives on its barriers any more, also where a wait has run
    // out: every wait above is bounded, so that all of the cluster's threads come here or have ended (the copying warp).
    if (FORM == kMergeCluster) {
        __syncwarp();
        ptx::cluster_sync();
    }
}

// The attention kernel, and the one that also refreshes the cache (its parameters, and the fresh rows of requests that
// do not attend over K and V in place: ReqShape::apart); each also in the form
// whose items are shared by clusters (instantiations of their own: the code of one form costs the other 1 %).
template <int D, int FORM>
__global__ void __launch_bounds__(kAttnThreads, 1)
region_attention_tc_kernel(const __grid_constant__ CUtensorMap tm_q,
                           const __grid_constant__ CUtensorMap tm_kf,
                           const __grid_constant__ CUtensorMap tm_vf,
                           const __grid_constant__ CUtensorMap tm_kc,
                           const __grid_constant__ CUtensorMap tm_vc, const AttnParams p) {
    const StoreParams none = {};
    attention_kernel_body<D, false, merge_of(FORM), is_spread(FORM)>(tm_q, tm_kf, tm_vf, tm_kc, tm_vc, tm_kf, tm_vf, p, none);
}
template <int D, int FORM>
__global__ void __launch_bounds__(kAttnThreads, 1)
region_attention_store_kernel(const __grid_constant__ CUtensorMap tm_q,
                              const __grid_constant__ CUtensorMap tm_kf,
                              const __grid_constant__ CUtensorMap tm_vf,
                              const __grid_constant__ CUtensorMap tm_kc,
                              const __grid_constant__ CUtensorMap tm_vc,
                              const __grid_constant__ CUtensorMap tm_ka,
                              const __grid_constant__ CUtensorMap tm_va, const AttnParams p,
                              const __grid_constant__ StoreParams sp) {
    attention_kernel_body<D, true, merge_of(FORM), is_spread(FORM)>(tm_q, tm_kf, tm_vf, tm_kc, tm_vc, tm_ka, tm_va, p, sp);
}

// Merges the workspace slots of the items that were spread over several shares:
// out = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s.  blockIdx.x + 1 names a share boundary; the
// attention kernel has left the item cut there (if any) in `cut`.  One warp per query row of the
// item's pair of tiles (blockIdx.y * 8 + warp); a lane owns D / 32 consecutive columns.  The kernel
// is launched behind the attention kernel with programmatic serialization and reads nothing before
// the dependency wait; all slots' loads are issued before the first use, so a warp pays one
// memory round trip, not one per slot.
// MAXS >= the slots of an item (AttnParams::max_slots, and kWaveSlots where pairs may be dealt in waves) bounds those held in
// registers (the host knows both, and the smaller instantiations let more warps be resident).
template <int D, int MAXS>
__global__ void __launch_bounds__(256)
region_attention_combine_kernel(const AttnParams p) {
    constexpr int kCombineMaxSlots = MAXS;
    constexpr int E = D / 32;
    using Vec = typename std::conditional<E == 4, float4, float2>::type;
    grid_dependency_wait();
    const int4* cp = reinterpret_cast<const int4*>(p.cut + blockIdx.x + 1);
    const int4 c0 = cp[0], c1 = cp[1];
    const int b = c0.y, h = c0.z, qp = c0.w, n_slots = c1.x, nq = c1.y, slot_at = c1.z, slot_step = c1.w;
    // (the fields are checked so that a table left incomplete by an aborted launch cannot send
    // this kernel out of bounds)
    if (c0.x != 1 || b < 0 || b >= p.B || h < 0 || h >= p.H || qp < 0 || qp >= p.P_cap ||
        n_slots < 2 || n_slots > kCombineMaxSlots || nq > p.Nq_cap || slot_at < 1 || slot_step < 1 || slot_step > 2 ||
        slot_at + (n_slots - 2) * slot_step >= p.B * p.H * p.P_cap * p.max_slots)
        return;
    const int lane = threadIdx.x & 31;
    const int r_local = blockIdx.y * 8 + (threadIdx.x >> 5);
    const int qrow = qp * (2 * kBM) + r_local;
    if (qrow >= nq) return;
    // (issued together with the slots' loads, used after them)
    const int dst_row = p.out_rows != nullptr ? p.out_rows[(size_t)b * p.Nq_cap + qrow] : qrow;

    float2 ml[kCombineMaxSlots];
    Vec o[kCombineMaxSlots];
#pragma unroll
    for (int s = 0; s < kCombineMaxSlots; ++s) {
        if (s < n_slots) {
            const size_t prow = (size_t)(s > 0 ? slot_at + (s - 1) * slot_step : slot_at - 1) * (2 * kBM) + r_local;
            ml[s] = p.part_ml[prow];
            o[s] = *reinterpret_cast<const Vec*>(p.part_o + prow * D + lane * E);
        }
    }
    float M = -INFINITY;
#pragma unroll
    for (int s = 0; s < kCombineMaxSlots; ++s)
        if (s < n_slots && ml[s].y > 0.f) M = fmaxf(M, ml[s].x);
    float acc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = 0.f;
    float L = 0.f;
#pragma unroll
    for (int s = 0; s < kCombineMaxSlots; ++s) {
        if (s < n_slots && ml[s].y > 0.f) {           // a slot without keys carries no weight
            const float wgt = fast_exp2(ml[s].x - M);
            L = fmaf(wgt, ml[s].y, L);
            const float* po = reinterpret_cast<const float*>(&o[s]);
#pragma unroll
            for (int e = 0; e < E; ++e) acc[e] = fmaf(wgt, po[e], acc[e]);
        }
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    if (dst_row < 0 || dst_row >= p.out_cap) {             // destination out of range: dropped
        if (lane == 0) record_status(p.dev_status, REGIONE_DEV_BOUNDS);
        return;
    }
    uint16_t* orow = p.out + (((size_t)b * p.out_cap + dst_row) * p.H + h) * D + lane * E;
    uint32_t packed[E / 2];
#pragma unroll
    for (int e = 0; e < E; e += 2) packed[e / 2] = pack_bf16x2(acc[e] * inv, acc[e + 1] * inv);
    if constexpr (E == 4)
        *reinterpret_cast<uint2*>(orow) = make_uint2(packed[0], packed[1]);
    else
        *reinterpret_cast<uint32_t*>(orow) = packed[0];
}

// Self-test of the bounded waits: a warp waits, through the same routines that the attention kernel's roles wait with,
// on an mbarrier that nobody ever arrives on, for a peer's arrival on it, and for flags that nothing sets.  No copy and
// no tensor-core operation is in flight, so giving up is all that happens: each wait must return false after `limit`
// cycles with REGIONE_DEV_TIMEOUT recorded, and the kernel ends normally.
// out[0] = 1 if a wait reported a completed phase (it must not), out[1] = cycles spent in the shortest wait,
// out[2] = 1 if each of them raised its abort flag.
__device__ unsigned long long g_unset_flags[33];
__global__ void bounded_wait_selftest_kernel(long long limit, int32_t* dev_status, long long* out) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag[3];
    const int lane = threadIdx.x;
    if (lane < 3) abort_flag[lane] = 0;
    if (lane == 0) {
        ptx::mbar_init(ptx::smem_addr(&bar), 1);
        ptx::fence_barrier_init();
    }
    __syncwarp();
    AttnParams p = {};
    p.dev_status = dev_status; p.timeout_cycles = limit;
    p.ready = g_unset_flags; p.epoch = 1;
    bool done = false;
    long long shortest = 0x7fffffffffffffffLL;
    for (int i = 0; i < 3; ++i) {
        const long long t0 = clock64();
        if (i == 2) done |= wait_shares(p, 1, 1, lane, &abort_flag[2]);             // (a wait of the whole warp)
        else if (lane == 0)
            done |= i == 0 ? wait_bar(ptx::smem_addr(&bar), 0, &abort_flag[0], dev_status, limit)
                           : wait_bar_cluster(ptx::smem_addr(&bar), &abort_flag[1], dev_status, limit);
        const long long spent = clock64() - t0;
        shortest = spent < shortest ? spent : shortest;
        __syncwarp();
    }
    if (lane == 0) {
        if (out != nullptr) {
            out[0] = done ? 1 : 0;
            out[1] = shortest;
            out[2] = abort_flag[0] && abort_flag[1] && abort_flag[2];
        }
        ptx::mbar_inval(ptx::smem_addr(&bar));
    }
}

// ---- host side ---------------------------------------------------------------------------------

// Launch shape from the capacities alone (so the workspace query and the launch agree): a
// persistent grid of one CTA per SM (fewer if there are fewer steps), and enough workspace slots
// per item that the longest item can be spread over the shares it meets at that grid size.
struct LaunchPlan {
    int grid, P_cap, max_slots;
};

static LaunchPlan plan_launch(int B, int Nq_cap, int Nf_cap, int Nc_cap, int H, int sms = sm_count()) {
    LaunchPlan lp;
    lp.P_cap = (Nq_cap + 2 * kBM - 1) / (2 * kBM);
    const long long nt_cap = std::max(1, (Nf_cap + kBN - 1) / kBN + (Nc_cap + kBN - 1) / kBN);
    const long long total_cap = (long long)B * H * lp.P_cap * nt_cap;
    lp.grid = (int)std::min<long long>(sms, std::max<long long>(total_cap, 1));
    const long long share = (total_cap + lp.grid - 1) / lp.grid;
    lp.max_slots = (int)std::min<long long>(8, std::max<long long>(2, (nt_cap + share - 1) / share + 1));
    return lp;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qres) ==
                cudaSuccess && qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(f);
    }
    return fn;
}

// [B, rows, H, D] bf16 as a 4-D tensor (D, H, rows, B); box = 64 columns x 1 head x 128 rows.
static bool make_map(CUtensorMap* map, const void* base, int B, int rows, int H, int D) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    if (rows <= 0) rows = 1;     // never loaded from; keeps the encoder happy
    cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)H, (cuuint64_t)rows, (cuuint64_t)B};
    cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)H * D * 2, (cuuint64_t)rows * H * D * 2};
    cuuint32_t box[4] = {64, 1, (cuuint32_t)kBN, 1};
    cuuint32_t elem[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box,
              elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static inline size_t slot_rows(const LaunchPlan& lp, int B, int H) {
    return (size_t)B * H * lp.P_cap * lp.max_slots * (2 * kBM);
}

size_t region_attention_tc_workspace(int B, int Nq_cap, int Nf_cap, int Nc_cap, int H, int D) {
    const LaunchPlan lp = plan_launch(B, Nq_cap, Nf_cap, Nc_cap, H);
    const size_t rows = slot_rows(lp, B, H);
    return ((rows * D * sizeof(float) + 255) & ~(size_t)255) +
           ((rows * sizeof(float2) + 255) & ~(size_t)255) + (size_t)lp.grid * (sizeof(CutItem) + sizeof(unsigned long long)) +
           sizeof(unsigned long long);
}

template <int D, bool STORE, int FORM>
static auto main_kernel() {
    if constexpr (STORE) return region_attention_store_kernel<D, FORM>;
    else return region_attention_tc_kernel<D, FORM>;
}

// Once per device: the opt-in to large dynamic shared memory, and how many clusters of each size fit the GPU.
template <int D, bool STORE>
static int prepare_kernel(const int** fitting) {
    static int configured[kMaxDevices] = {};
    static int clusters[kMaxDevices][kMaxCluster + 1] = {};
    const int dev = current_device();
    if (dev < 0) return REGIONE_CUDA_ERROR;
    if (!__atomic_load_n(&configured[dev], __ATOMIC_ACQUIRE)) {
        auto opt_in = [](auto kernel) {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<D>::kSmemBytes) == cudaSuccess;
        };
        if (!opt_in(main_kernel<D, STORE, kFormKernel>()) || !opt_in(main_kernel<D, STORE, kFormHere>()) ||
            !opt_in(main_kernel<D, STORE, kFormCluster>()) || !opt_in(main_kernel<D, STORE, kFormSpreadKernel>()) ||
            !opt_in(main_kernel<D, STORE, kFormSpreadHere>()))
            return REGIONE_CUDA_ERROR;
        for (int n = 2; n <= kMaxCluster; ++n) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(n * 148);
            cfg.blockDim = dim3(kAttnThreads);
            cfg.dynamicSmemBytes = AttnCfg<D>::kSmemBytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = n; attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, main_kernel<D, STORE, kFormCluster>(), &cfg) != cudaSuccess) {
                (void)cudaGetLastError();
                fit = 0;
            }
            clusters[dev][n] = fit;
        }
        __atomic_store_n(&configured[dev], 1, __ATOMIC_RELEASE);
    }
    *fitting = clusters[dev];
    return REGIONE_OK;
}

// Rows that are put back into a joint sequence many times their number keep the cuts of the cost axis with kTickStart.
// This line is neither the faster side's nor the more accurate one's: where an item is cut decides which reference
// maximum its probabilities are rounded against, and against the rms of the whole buffer, mostly rows that were not
// recomputed, the two forms differ from each other by up to 0.1 in single elements (by 0.04 from a twelfth of the rows
// on).  Against 64 bits, over the recomputed rows, clusters / cost axis: 64 of 8448 rows rel 2.32 / 2.31e-3, 32.7 / 36.4 us;
// 128 2.31 / 2.31e-3, 33.6 / 38.7 us; 205 2.32 / 2.32e-3, 42.7 / 43.6 us; 704 2.33 / 2.33e-3, 74.4 / 79.8 us.  What holds it is
// test_step_on_both_sides_of_its_rules, which counts the launches of steps with 768 and 769 rows of keys.
static bool keeps_cuts(const AttnParams& p) {
    return p.out_rows != nullptr && 12LL * (p.Nq_cap - kBM / 2) < (long long)p.Nf_cap + p.Nc_cap;
}

// How many CTAs share an item through a cluster, 0: shares of the cost axis with a merge kernel behind them.
// Few items (at most one cluster of two per pair of SMs) are better off in clusters: the shares of the cost axis are
// balanced to a step, but their cut items cost about kTickMerge ticks against kTickCluster for a merge through distributed
// shared memory.  Both sides' ticks from the capacities:
constexpr int kTickCluster = 45;
static int choose_cluster(const int* fitting, const AttnParams& p, int nt) {
    if (keeps_cuts(p)) return 0;
    const long long items = (long long)p.B * p.H * p.P_cap;
    const bool lone_last = ((p.Nq_cap + kBM - 1) / kBM) % 2 == 1;
    const long long w_max = p.P_cap == 1 && lone_last ? kTickSingle : kTickPair;
    const long long ticks = (long long)p.B * p.H * ((p.P_cap - 1) * (kTickStart + (long long)kTickPair * nt) + kTickStart +
                                                    (long long)(lone_last ? kTickSingle : kTickPair) * nt);
    // (a share is at least as long as the slots of an item allow, and pays for a start of its own where it begins
    // inside an item)
    long long best = std::max((ticks + sm_count() - 1) / sm_count(), w_max * (nt - 1) / (p.max_slots - 1)) + kTickStart +
                     kTickMerge;
    int n_best = 0;
    for (int n = 2; n <= kMaxCluster && n <= nt; ++n) {
        if (items > fitting[n]) continue;
        const long long cost = kTickStart + w_max * ((nt + n - 1) / n) + kTickCluster;
        if (cost < best) { best = cost; n_best = n; }
    }
    return n_best;
}

// Who merges cut items.  The first share takes about as long for one other share's rows (6500 cycles and a wait of 1000)
// as the merge kernel does for all of them (8 us behind the attention), but off the path of the shares that it waits
// for, without the write and the read of its own rows and without a launch.  Measured, merge kernel -> first share, us
// (plain calls with what precedes them, stores as region steps): 2048 of 8448 rows, 24 heads, refreshed 252.7 -> 244.2;
// four requests with 1382 of 18944 1395 -> 1378; 1075 queries x 8448 keys 149.3 -> 147.7; 819 x 8704 129.2 -> 129.4, behind
// an 8-bit decode 137.4 -> 136.4; D = 64, 2048 x 6048 118.6 -> 110.2.  Not where an item is spread over many shares, whose
// rows one CTA would read one after the other (205 x 8448 keys, 6 shares: 53.4 -> 63.3), nor where a share is short
// beside the merge (three requests, 250 x 4650, 16 heads, 26 steps a share: 60.3 -> 63.8), nor where whole items
// outnumber the cut ones (8704 x 8704, 816 items, at the power limit: 856 -> 868).
static bool merges_here(const AttnParams& p, int grid, int nt) {
    const long long items = (long long)p.B * p.H * p.P_cap;
    return p.max_slots <= 3 && items <= 4LL * grid && items * nt >= 40LL * grid;
}

// Whether the plan minds the order in which K and V are read (see plan_shares): where they are more than L2 keeps (126 MB
// in two halves, each of which holds what its own SMs read).  Measured, without -> with, us: 1075 queries x 8448 keys of 128,
// 8 heads (33 MB) 57.4 -> 58.1, 12 (49 MB) 77.2 -> 79.6, 16 (66 MB) 99.1 -> 97.5, 24 (99 MB) 146.3 -> 136.9; 8704 x
// 8704, 8 heads 268 -> 272, 12 401 -> 398, 16 561 -> 525, 24 845 -> 767; a step that refreshes 2048 of 8448 rows, 12 heads
// 125.8 -> 127.2, 16 162.7 -> 159.6, 24 248.7 -> 229.4.
// Where the plan of full capacities would deal whole items or cut the cost axis after all, it is left at that: its code is
// the shorter one (three requests of 543 of 3730 rows, 12 heads, 79.6 -> 74.0 us; of 633 x 3925 keys, 16 heads, 85.3 -> 83.2).
// The plan itself follows the live counts: 819 and 2048 of 8448 rows take as long with room for a tenth more as without.
// Requests whose counts differ by whole pairs walk the cost axis here too, and take 0 to 2.5 % longer than there (two requests
// of 819 and 1024 of 8448 rows 246.2 / 247.1, of 410 and 1229 213.7 / 216.3, four of 205 to 1638, refreshed, 466.3 / 478.0).
// Teams whose cut items a merge kernel puts together have short shares: 300 x 8448 59.5 -> 60.6, three requests of 552 x 6716, 12
// heads, 97.7 -> 99.7.
// Heads of 64 read half as many bytes for as many exponentials.  Refreshing launches mind the order (1638 of 16896 rows 266.4 ->
// 260.9; without the refresh 250.8 -> 254.6), waves of 90 MB and more (16000 x 16000 1980 -> 1967; 11000 x 11000, 67 MB, 947 ->
// 953), and teams where the other plan is one of whole items (four requests of 594 x 6805 178.8 -> 161.9).
constexpr long long kSpreadBytes = 60LL << 20, kSpreadBytes64 = 90LL << 20;
static long long kv_bytes(const AttnParams& p, int d) { return 4LL * d * p.B * p.H * ((long long)p.Nf_cap + p.Nc_cap); }
template <int D>
static bool minds_order(const AttnParams& p, int grid, bool refreshes, int single, bool here) {
    // (a head with one pair reads its keys once, in whatever order)
    if (keeps_cuts(p) || p.P_cap < 2 || kv_bytes(p, D) < kSpreadBytes || (long long)p.B * p.H * p.P_cap > 0x7fffffff) return false;
    PlanInput full = p;                              // (requests alike are one with as many heads as they have together)
    // (the rows that a row list names are those of the joint sequence, and so are the keys: together not more than its rows)
    const int32_t cached = p.out_rows != nullptr ? std::max(0, std::min(p.Nc_cap, p.out_cap - p.Nf_cap)) : p.Nc_cap;
    const int32_t counts[3] = {p.Nq_cap, p.Nf_cap, cached};
    full.n_q = counts; full.n_fresh = counts + 1; full.n_cache = counts + 2;
    full.B = 1; full.H = p.B * p.H; full.all_rows = 0; full.single = single;
    const PlanKind kind = plan_shares<false, true>(full, grid).kind;
    if (D == 64 && !refreshes) {
        if (kind == kWaves) return kv_bytes(p, D) >= kSpreadBytes64;
        return kind == kTeams && plan_shares<false, false>(full, grid).kind == kWhole;
    }
    return kind == kWaves || (kind == kTeams && here);
}

// Whether K and V are told to leave L2 first: where a head has one query pair, so that they pass through once, and are more
// than L2 keeps.  What the next launches read (lists, latents, partial rows, code) stays then.  A step with 205 of 8448 rows
// 54.1 -> 52.2 us, behind a flushed L2 63.6 -> 58.5; four requests of 92 x 4736 74.9 -> 69.9 (other K and V in every call).
// A step that has just copied its rows to the cache gains as well (four requests of 116 of 3000 rows 105.7 -> 100.3), and a
// scattered call behind an 8-bit decode loses as much as it gains (205 x 8448 64.9 -> 65.7, behind a flushed L2 72.8 -> 70.8).
// Not where several pairs read them (four requests of 1382 x 18944 +7 %, 1075 x 8448 +1 to 2 %, 819 x 8704 -1 %), nor where they
// fit L2 (two requests of 102 x 2176, 8 heads of 64, +2 to 4 %), nor in calls without a row list behind a decode (205 x 8448
// 67.3 -> 69.5), nor in a launch whose copying warps read the rows of the cache a second time (four requests of 256 of 2148 rows
// refreshed 92.4 -> 94.1, of 246 of 2988 109.4 -> 111.2).
static bool reads_once(const AttnParams& p, int d, bool refreshes) {
    return p.P_cap == 1 && !refreshes && p.out_rows != nullptr && kv_bytes(p, d) >= kSpreadBytes;
}

// The form of a call, and the CTAs of a cluster (prm.cluster).
template <int D, bool STORE>
static int choose_form(const int* fitting, AttnParams& prm, int grid, int nt_cap) {
    prm.cluster = choose_cluster(fitting, prm, nt_cap);
    prm.single = kTickSingle;
    if (prm.cluster > 0) return kFormCluster;
    const bool here = merges_here(prm, grid, nt_cap);
    constexpr int single = STORE && D == 128 ? kTickSingleRefresh : kTickSingle;
    if (!minds_order<D>(prm, grid, STORE, single, here)) return here ? kFormHere : kFormKernel;
    prm.single = single;
    return here ? kFormSpreadHere : kFormSpreadKernel;
}

template <int D, bool STORE>
static int launch_tc(const CUtensorMap* maps, AttnParams prm, const StoreParams& sp, int grid, int nt_cap, cudaStream_t st) {
    const int* fitting = nullptr;
    const int rc = prepare_kernel<D, STORE>(&fitting);
    if (rc != REGIONE_OK) return rc;
    const int form = choose_form<D, STORE>(fitting, prm, grid, nt_cap);
    // (a refreshing launch takes every cluster that fits: those without an item copy rows of the cache)
    if (prm.cluster > 0) grid = (STORE ? fitting[prm.cluster] : prm.B * prm.H * prm.P_cap) * prm.cluster;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = AttnCfg<D>::kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // see grid_dependency_wait
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = prm.cluster > 0 ? prm.cluster : 1;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = prm.cluster > 0 ? 2 : 1;
    cudaError_t e;
    auto launch = [&](auto kernel) {
        if constexpr (STORE) return launch_counted(&cfg, kernel, maps[0], maps[1], maps[2], maps[3], maps[4], maps[5], maps[6], prm, sp);
        else return launch_counted(&cfg, kernel, maps[0], maps[1], maps[2], maps[3], maps[4], prm);
    };
    switch (form) {
        case kFormCluster: e = launch(main_kernel<D, STORE, kFormCluster>()); break;
        case kFormSpreadHere: e = launch(main_kernel<D, STORE, kFormSpreadHere>()); break;
        case kFormSpreadKernel: e = launch(main_kernel<D, STORE, kFormSpreadKernel>()); break;
        case kFormHere: e = launch(main_kernel<D, STORE, kFormHere>()); break;
        default: e = launch(main_kernel<D, STORE, kFormKernel>());
    }
    if (e != cudaSuccess) return REGIONE_CUDA_ERROR;
    // the merge kernel may become resident while the attention kernel drains (it waits for that
    // kernel's completion before it reads a slot)
    if (grid < 2 || merge_of(form) != kMergeKernel) return launch_status(cudaGetLastError());     // nothing is cut
    const dim3 cgrid((unsigned)(grid - 1), (2 * kBM) / 8, 1);
    const int most_slots = is_spread(form) ? std::max(prm.max_slots, kWaveSlots) : prm.max_slots;
    if (most_slots <= 2)
        e = launch_overlapped(region_attention_combine_kernel<D, 2>, cgrid, dim3(256), 0, st, prm);
    else if (most_slots <= 3)
        e = launch_overlapped(region_attention_combine_kernel<D, 3>, cgrid, dim3(256), 0, st, prm);
    else if (most_slots <= 4)
        e = launch_overlapped(region_attention_combine_kernel<D, 4>, cgrid, dim3(256), 0, st, prm);
    else
        e = launch_overlapped(region_attention_combine_kernel<D, 8>, cgrid, dim3(256), 0, st, prm);
    if (e != cudaSuccess) return REGIONE_CUDA_ERROR;
    return launch_status(cudaGetLastError());
}

// A number that no other launch has and that memory does not hold by chance: a count, spread over 64 bits by
// multiplication with 2^64 / golden ratio (Fibonacci hashing, Knuth, The Art of Computer Programming 3, 6.4).
static unsigned long long next_epoch() {
    static std::atomic<unsigned long long> count{
        (unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count()};
    const unsigned long long z = count.fetch_add(1, std::memory_order_relaxed) * 0x9E3779B97F4A7C15ull;   // (odd: a bijection)
    return z != 0 ? z : 1;
}

int launch_region_attention_tc(const uint16_t* q, const uint16_t* k_fresh, const uint16_t* v_fresh,
                               const uint16_t* k_cache, const uint16_t* v_cache, const int32_t* n_q,
                               const int32_t* n_fresh, const int32_t* n_cache, int B, int Nq_cap,
                               int Nf_cap, int Nc_cap, int H, int D, float scale, uint16_t* out,
                               const int32_t* out_rows, int out_cap, void* workspace,
                               size_t workspace_bytes, int32_t* dev_status, cudaStream_t st,
                               const CacheStore* store) {
    (void)workspace_bytes;
    CUtensorMap maps[7];
    const int all_rows = store != nullptr ? store->all_rows : 0;
    // an absent segment still needs a valid (never dereferenced) base address
    const void* kf = Nf_cap > 0 ? (const void*)k_fresh : (const void*)q;
    const void* vf = Nf_cap > 0 ? (const void*)v_fresh : (const void*)q;
    const void* kc = all_rows > 0 ? store->k_cache : Nc_cap > 0 ? (const void*)k_cache : (const void*)q;
    const void* vc = all_rows > 0 ? store->v_cache : Nc_cap > 0 ? (const void*)v_cache : (const void*)q;
    if (!make_map(&maps[0], q, B, Nq_cap, H, D) || !make_map(&maps[1], kf, B, Nf_cap, H, D) ||
        !make_map(&maps[2], vf, B, Nf_cap, H, D) || !make_map(&maps[3], kc, B, all_rows > 0 ? all_rows : Nc_cap, H, D) ||
        !make_map(&maps[4], vc, B, all_rows > 0 ? all_rows : Nc_cap, H, D))
        return REGIONE_CUDA_ERROR;
    if (store != nullptr && (!make_map(&maps[5], all_rows > 0 ? store->k_apart : q, B, Nq_cap, H, D) ||
                             !make_map(&maps[6], all_rows > 0 ? store->v_apart : q, B, Nq_cap, H, D)))
        return REGIONE_CUDA_ERROR;
    const LaunchPlan lp = plan_launch(B, Nq_cap, Nf_cap, Nc_cap, H);
    AttnParams prm;
    prm.n_q = n_q; prm.n_fresh = n_fresh; prm.n_cache = n_cache;
    prm.B = B; prm.Nq_cap = Nq_cap; prm.Nf_cap = Nf_cap; prm.Nc_cap = Nc_cap; prm.H = H;
    prm.P_cap = lp.P_cap; prm.max_slots = lp.max_slots;
    prm.scale_log2e = scale * 1.4426950408889634f;
    prm.out = out; prm.dev_status = dev_status;
    prm.out_rows = out_rows;
    prm.out_cap = out_rows != nullptr ? out_cap : Nq_cap;
    prm.all_rows = all_rows;
    prm.timeout_cycles = kTimeoutCycles;
    StoreParams sp = {};
    if (store != nullptr) {
        sp.rows[0] = store->keep_rows; sp.n[0] = store->n_keep; sp.cap[0] = store->cap; sp.src_cap = Nf_cap;
        sp.src[0] = reinterpret_cast<const uint8_t*>(k_fresh); sp.src[1] = reinterpret_cast<const uint8_t*>(v_fresh);
        sp.dst[0] = reinterpret_cast<uint8_t*>(store->k_cache); sp.dst[1] = reinterpret_cast<uint8_t*>(store->v_cache);
        sp.n_lists = 1;
        if (all_rows > 0) {
            sp.rows[1] = out_rows; sp.n[1] = n_q; sp.cap[1] = Nq_cap;
            sp.dst[2] = reinterpret_cast<uint8_t*>(store->k_apart); sp.dst[3] = reinterpret_cast<uint8_t*>(store->v_apart);
            sp.n_lists = 2;
        }
    }
    const size_t rows = slot_rows(lp, B, H);
    prm.part_o = reinterpret_cast<float*>(workspace);
    uint8_t* const ws = reinterpret_cast<uint8_t*>(workspace);
    const size_t off_ml = (rows * D * sizeof(float) + 255) & ~(size_t)255;
    prm.part_ml = reinterpret_cast<float2*>(ws + off_ml);
    prm.cut = reinterpret_cast<CutItem*>(ws + off_ml + ((rows * sizeof(float2) + 255) & ~(size_t)255));
    prm.ready = reinterpret_cast<unsigned long long*>(prm.cut + lp.grid);
    prm.epoch = next_epoch();
    prm.cluster = 0;
    prm.kv_once = reads_once(prm, D, store != nullptr);
    const int nt_cap = std::max(1, (Nf_cap + kBN - 1) / kBN + (Nc_cap + kBN - 1) / kBN);
    if (store != nullptr)
        return D == 64 ? launch_tc<64, true>(maps, prm, sp, lp.grid, nt_cap, st)
                       : launch_tc<128, true>(maps, prm, sp, lp.grid, nt_cap, st);
    return D == 64 ? launch_tc<64, false>(maps, prm, sp, lp.grid, nt_cap, st)
                   : launch_tc<128, false>(maps, prm, sp, lp.grid, nt_cap, st);
}

// The segments of every block of a launch, as the planning warps walk them (host).
template <bool IN_PLACE, bool SPREAD>
static int list_segments(const PlanInput& p, int grid, int32_t* out, int cap) {
    int n = 0;
    for (int block = 0; block < grid; ++block) {
        ShareWalk<IN_PLACE, SPREAD> walk;
        bool bad = false;
        walk.begin(p, grid, block, &bad);
        Segment it;
        while (walk.next(p, grid, block, it)) {
            if (it.n_steps == 0) continue;
            const int32_t row[12] = {block,   it.b,       it.h,       it.qp,        it.j_first, it.n_steps,
                                     it.slot, it.n_slots, it.slot_at, it.slot_step, walk.step,  it.in_wave ? -1 : (int)walk.pl.kind};
            if (n < cap) std::copy(row, row + 12, out + 12 * (size_t)n);
            ++n;
        }
    }
    return n;
}

// ---- variant with library-owned scratch -----------------------------------------------------
// The split-KV partials of regione_region_attention_static live here instead of in a caller
// workspace.  The array is part of the library image: every GPU that loads the library keeps
// these bytes resident until the process exits.
constexpr size_t kStaticScratchBytes = (size_t)64 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

namespace {
void* g_static_scratch_addr[kMaxDevices] = {};      // device address of the array, per device
}  // namespace

// Device address of g_static_scratch on the current device (in host code the symbol itself is
// only a stand-in and must never be handed to a kernel).  Resolved on the first call per device.
static int static_scratch_address(void** out) {
    const int dev = current_device();
    if (dev < 0) return REGIONE_CUDA_ERROR;
    void* addr = __atomic_load_n(&g_static_scratch_addr[dev], __ATOMIC_ACQUIRE);
    if (addr == nullptr) {
        if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || addr == nullptr) {
            (void)cudaGetLastError();
            return REGIONE_CUDA_ERROR;
        }
        __atomic_store_n(&g_static_scratch_addr[dev], addr, __ATOMIC_RELEASE);
    }
    *out = addr;
    return REGIONE_OK;
}

}  // namespace regione

extern "C" int regione_selftest_bounded_wait(long long limit_cycles, int32_t* dev_status,
                                             long long* out, void* stream) {
    using namespace regione;
    // the limit is capped well below the attention kernel's own so that the self-test stays short
    if (limit_cycles < 1 || limit_cycles > 100000000LL) return REGIONE_INVALID_ARG;
    bounded_wait_selftest_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(limit_cycles, dev_status, out);
    return launch_status(cudaGetLastError());
}

extern "C" int regione_selftest_attention_plan(const int32_t* n_q, const int32_t* n_fresh, const int32_t* n_cache, int B, int Nq_cap,
                                               int Nf_cap, int Nc_cap, int H, int all_rows, int spread, int sms, int32_t* shape,
                                               int32_t* segments, int cap) {
    using namespace regione;
    if (!n_q || !n_fresh || !n_cache || !shape || (!segments && cap > 0) || B < 1 || H < 1 || Nq_cap < 1 || Nf_cap < 0 || Nc_cap < 0 ||
        all_rows < 0 || sms < 1 || cap < 0)
        return -1;
    const LaunchPlan lp = plan_launch(B, Nq_cap, Nf_cap, Nc_cap, H, sms);
    PlanInput p = {};
    p.n_q = n_q; p.n_fresh = n_fresh; p.n_cache = n_cache;
    p.B = B; p.Nq_cap = Nq_cap; p.Nf_cap = Nf_cap; p.Nc_cap = Nc_cap; p.H = H;
    p.P_cap = lp.P_cap; p.max_slots = lp.max_slots; p.all_rows = all_rows;
    p.single = spread == 2 ? kTickSingleRefresh : kTickSingle;
    shape[0] = lp.grid; shape[1] = lp.P_cap; shape[2] = lp.max_slots; shape[3] = 0;
    if (spread) {
        const Plan pl = all_rows > 0 ? plan_shares<true, true>(p, lp.grid) : plan_shares<false, true>(p, lp.grid);
        if (pl.kind == kTeams) shape[3] = pl.team;
    }
    if (all_rows > 0)
        return spread ? list_segments<true, true>(p, lp.grid, segments, cap) : list_segments<true, false>(p, lp.grid, segments, cap);
    return spread ? list_segments<false, true>(p, lp.grid, segments, cap) : list_segments<false, false>(p, lp.grid, segments, cap);
}

extern "C" int regione_selftest_attention_form(int B, int Nq_cap, int Nf_cap, int Nc_cap, int H, int D, int out_cap, int refreshes) {
    using namespace regione;
    if (B < 1 || H < 1 || Nq_cap < 1 || Nf_cap < 0 || Nc_cap < 0 || out_cap < 0 || (D != 64 && D != 128)) return -1;
    const LaunchPlan lp = plan_launch(B, Nq_cap, Nf_cap, Nc_cap, H);
    static const int32_t list = 0;
    AttnParams p = {};
    p.B = B; p.Nq_cap = Nq_cap; p.Nf_cap = Nf_cap; p.Nc_cap = Nc_cap; p.H = H;
    p.P_cap = lp.P_cap; p.max_slots = lp.max_slots;
    p.out_rows = out_cap > 0 ? &list : nullptr;
    p.out_cap = out_cap > 0 ? out_cap : Nq_cap;
    const int nt_cap = std::max(1, (Nf_cap + kBN - 1) / kBN + (Nc_cap + kBN - 1) / kBN);
    const int* fitting = nullptr;
    auto form = [&](auto prepared, auto choose) { return prepared(&fitting) != REGIONE_OK ? -1 : choose(fitting, p, lp.grid, nt_cap); };
    if (refreshes)
        return D == 64 ? form(prepare_kernel<64, true>, choose_form<64, true>) : form(prepare_kernel<128, true>, choose_form<128, true>);
    return D == 64 ? form(prepare_kernel<64, false>, choose_form<64, false>) : form(prepare_kernel<128, false>, choose_form<128, false>);
}

extern "C" int regione_region_attention_static(
    const regione_bf16* q, const regione_bf16* k_fresh, const regione_bf16* v_fresh,
    const regione_bf16* k_cache, const regione_bf16* v_cache, const int32_t* n_q,
    const int32_t* n_fresh, const int32_t* n_cache, int B, int Nq_cap, int Nf_cap, int Nc_cap, int H,
    int D, float softmax_scale, regione_bf16* out, int32_t* dev_status, void* stream) {
    using namespace regione;
    bool nothing = false;
    const int args_rc = check_attention_args(q, k_fresh, v_fresh, k_cache, v_cache, n_q, n_fresh,
                                             n_cache, B, Nq_cap, Nf_cap, Nc_cap, H, D, out, &nothing);
    if (args_rc != REGIONE_OK || nothing) return args_rc;
    // the partials of this shape must fit the fixed array: refuse, never truncate
    const size_t need = region_attention_tc_workspace(B, Nq_cap, Nf_cap, Nc_cap, H, D);
    if (need > kStaticScratchBytes) return REGIONE_WORKSPACE_TOO_SMALL;
    void* scratch = nullptr;
    const int rc = static_scratch_address(&scratch);
    if (rc != REGIONE_OK) return rc;
    const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)D);
    // Nothing in the scratch has to start at zero: every row that is merged is written by the attention kernel of the
    // same call, and the flags that say so are compared with a number that only this call has.
    return launch_region_attention_tc(q, k_fresh, v_fresh, k_cache, v_cache, n_q, n_fresh, n_cache,
                                      B, Nq_cap, Nf_cap, Nc_cap, H, D, scale, out, nullptr, 0, scratch,
                                      kStaticScratchBytes, dev_status, (cudaStream_t)stream, nullptr);
}
