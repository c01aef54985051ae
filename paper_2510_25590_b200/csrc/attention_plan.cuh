// How the work of one attention launch is cut into shares, one per CTA.  Every CTA derives the same plan from the
// request counts in device memory; the functions also run on the host, where a test checks that the shares cover
// every step once.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define REGIONE_HD __host__ __device__ __forceinline__

namespace regione {

constexpr int kBM = 128;                 // query rows per tile
constexpr int kBN = 128;                 // key rows per shared-memory tile

struct PlanInput {
    const int32_t* n_q;
    const int32_t* n_fresh;
    const int32_t* n_cache;
    int B, Nq_cap, Nf_cap, Nc_cap, H;
    int P_cap;           // query pairs per (request, head) at capacity
    int max_slots;       // workspace slots per item (>= 2)
    int all_rows;        // > 0: query and cached rows of a request are parts of its K and V of this many rows (see ReqShape)
    int single;          // ticks of a key tile of a pair with one live query tile (see kTickSingle)
};

// Shares are cut on a cost axis measured in ticks, not in steps, so that they take about the same
// time: a key tile of a full query pair costs kTickPair, a key tile of a pair with one live query
// tile kTickSingle (its even and odd key tiles run side by side on the two tile roles; measured per
// thread block against its share's composition: 0.55 to 0.56 of a pair's step, not half), and every
// item starts with kTickStart ticks that stand for the drain of the previous segment and the fill of
// the new one (measured the same way: 3.5 to 6 pair steps depending on the workload, 5 with 819 x 8704 and
// 1075 x 8448 keys, 24 heads of 128; 100, 120 and 140 ticks for items that a first share merges: 0 to +3 %).
constexpr int kTickPair = 16, kTickSingle = 9, kTickStart = 80;
// A launch that refreshes the cache with heads of 128 has no room for the wider ring of a lone tile, whose step takes 0.75 of
// a pair's (2320 of 3080 cycles).  It matters where lone tiles lie together, in the plans that mind the order of the keys (8211
// x 8211 refreshed, 24 heads, 786.3 -> 737.4 us, 750.0 on the cost axis; a step that refreshes 819 of 8448 rows 138.4 -> 126.6);
// the others deal them evenly among the pairs and keep the ticks above.
constexpr int kTickSingleRefresh = 12;
// What the merge of cut items costs a launch: every cut item's rows go through the workspace (7300 cycles per pair of
// tiles, all CTAs at once) and a second kernel (8 us behind the attention's last block).
constexpr int kTickMerge = 125;

struct ReqShape {
    int nq, nf, nc;      // clamped counts
    int np, full;        // live query pairs, those of them with two live query tiles (all, or all but the last)
    int nt_c, nt;        // cached key tiles, all key tiles
    long long items;     // H * np
    int steps;           // steps of an item: max(nt, 1) (an item without keys writes zeros in one step)
    bool apart;          // PlanInput::all_rows: the query and cached rows are not all rows (more tokens were edited than
                         // the capacity holds), so the request attends over [cached | fresh] as copied ahead of the launch
    int w_last;          // ticks per step of the last query pair
    long long ticks_full, ticks_last, head_ticks, ticks;   // per full-pair item, last item, head, request
};

// (IN_PLACE: the launch may read K and V in place, see ReqShape::apart; 0.5 us a call for the launches that never do)
template <bool IN_PLACE>
REGIONE_HD ReqShape req_shape(const PlanInput& p, int b, bool* bad = nullptr) {
    ReqShape r;
    int nq = p.n_q[b], nf = p.n_fresh[b], nc = p.n_cache == nullptr ? 0 : p.n_cache[b];      // (nullptr: no cached segment)
    const int all_rows = IN_PLACE ? p.all_rows : 0;
    const int c_cap = all_rows > 0 ? all_rows : p.Nc_cap;
    if (nq < 0 || nq > p.Nq_cap || nf < 0 || nf > p.Nf_cap || nc < 0 || nc > c_cap) {
        if (bad) *bad = true;
        nq = max(0, min(nq, p.Nq_cap));
        nf = max(0, min(nf, p.Nf_cap));
        nc = max(0, min(nc, c_cap));
    }
    r.apart = all_rows > 0 && nq + nc != all_rows;
    if (all_rows > 0) {
        nf = r.apart ? nq : all_rows;
        nc = r.apart ? nc : 0;
    }
    r.nq = nq; r.nf = nf; r.nc = nc;
    r.np = (nq + 2 * kBM - 1) / (2 * kBM);
    r.nt_c = (nc + kBN - 1) / kBN;
    r.nt = r.nt_c + (nf + kBN - 1) / kBN;
    r.items = (long long)p.H * r.np;
    r.steps = max(r.nt, 1);
    r.w_last = (nq - (r.np - 1) * 2 * kBM > kBM) ? kTickPair : p.single;
    r.full = r.w_last == kTickPair ? r.np : max(r.np - 1, 0);
    r.ticks_full = kTickStart + (long long)kTickPair * r.steps;
    r.ticks_last = kTickStart + (long long)r.w_last * r.steps;
    r.head_ticks = r.np > 0 ? (r.np - 1) * r.ticks_full + r.ticks_last : 0;
    r.ticks = p.H * r.head_ticks;
    return r;
}

// a / b for non-negative a and positive b; positions fit 32 bits in every realistic launch, and a
// 32-bit division is several times shorter than a 64-bit one (the lookups below sit between two
// segments, on every thread's path).
REGIONE_HD long long div_pos(long long a, long long b) {
    if (((a | b) >> 32) == 0) return (long long)((unsigned)a / (unsigned)b);
    return a / b;
}

// How the launch's work is cut into shares, one per CTA.
//  - kWhole: when handing out whole items wastes at most 6 % of the grid's last round, items are dealt
//    round-robin and never split (no workspace traffic, no merge): positions count items.
//  - kTicks: positions count ticks and CTA c owns the steps whose first tick lies in
//    [c * chunk, (c + 1) * chunk); shares may cut items.  The share length is bounded below so
//    that an item never meets more than max_slots shares.
// Those two leave the order in which K and V are read to chance: shares of the cost axis lie all over the heads, so that
// at any time the CTAs read every head's keys, each at a place of its own, and a key tile has left L2 by the time another
// query pair needs it.  Where the launch's K and V are more than L2 keeps (SPREAD):
//  - kWaves: full pairs are dealt whole, a round of the grid at a time, so that the CTAs walk a few heads from
//    their first key on together; what is left of the pairs, and then the pairs with one live query tile, are cut
//    into shares as above.
//  - kTeams: `team` CTAs walk the same keys of a head at the same time, each for a full pair of its own.  The axis counts the
//    ticks of one of them and is cut into one share per team; the pairs with one live query tile are an axis of their own,
//    shared by the CTAs that are in no team, as many as make the two kinds of share equally long.  The team is chosen from the
//    live counts, and taken where its longest share is within 4 % of the mean.
enum PlanKind { kWhole, kTicks, kWaves, kTeams };
struct Plan {
    PlanKind kind;
    long long total, chunk;      // kTeams: the pairs' axis and a team's share of it
    long long lone_chunk;        // kTeams: share of the pairs with one live query tile (their axis begins at `total`)
    long long lone_total;
    long long origin;            // kWaves: tick at which the cut part begins
    int waves;
    int team, n_teams;
};
// Items dealt round-robin are walked in step too.  Percent of the mean share up to which they are, where the grid's last round
// also is full by kWhole's rule: at the power limit CTAs that end early leave their power to the others, and nothing is
// merged.  Waves -> whole items, us: three requests of 4916 x 4916, 24 heads (4.8 % above the mean) 868 -> 841; four of 1382 x
// 18944 (10.6 %), with the line of keeps_cuts moved so that they came here, 1424 -> 1376.
constexpr int kWholeWaste = 112;
constexpr int kWaveSlots = 4;    // kWaves: shares that a cut item may meet

// A way to make teams: n_teams of `team` CTAs, the ticks of a member's axis, and the shares of it and of the pairs with one
// live query tile.
struct TeamCut {
    int team, n_teams;
    long long total, a, l;
    long long cost;              // longest share, weighted (0: not possible)
};

// One team for all full pairs of a head (i = 0, 1), or for half of them where the grid divides better by that (2, 3: the
// second reads K and V a second time, hence 1.5 %); as many teams as make their shares as long as those of the CTAs in
// no team, or one more (odd i).  most: full pairs of a head, at most.
REGIONE_HD TeamCut team_cut(const PlanInput& p, int grid, int i, int most, long long pair_ticks, long long lone_ticks) {
    TeamCut c;
    c.team = i < 2 ? most : (most + 1) >> 1;
    long long supers = 0;
    for (int b = 0; b < p.B; ++b) {
        const int full = ((max(0, min(p.n_q[b], p.Nq_cap)) + kBM - 1) / kBM) >> 1;
        supers += (long long)p.H * ((unsigned)(full + c.team - 1) / (unsigned)c.team);
    }
    c.total = supers * pair_ticks;
    const long long teams = div_pos(grid * c.total, lone_ticks + c.team * c.total);
    c.n_teams = (int)min(teams, (long long)((unsigned)grid / (unsigned)c.team)) + (i & 1);
    const int rest = grid - c.team * c.n_teams;
    c.a = c.l = c.cost = 0;
    if (c.n_teams < 1 || rest < 0 || (rest == 0 && lone_ticks > 0)) return c;
    c.a = div_pos(c.total + c.n_teams - 1, c.n_teams);
    if (rest > 0) c.l = div_pos(lone_ticks + rest - 1, rest);
    c.cost = max(c.a, c.l) * (i < 2 ? 1000 : 1015);
    return c;
}

// The shortest of the four; on the GPU by the lanes of the calling warp, which has to call this as a whole.
REGIONE_HD TeamCut best_team(const PlanInput& p, int grid, int most, long long pair_ticks, long long lone_ticks) {
#ifdef __CUDA_ARCH__
    const int i = threadIdx.x & 3;
    TeamCut c = team_cut(p, grid, i, most, pair_ticks, lone_ticks);
    int from = i;
    long long best = c.cost;
    for (int d = 1; d <= 2; d <<= 1) {
        const long long cost = __shfl_xor_sync(0xffffffffu, best, d);
        const int other = __shfl_xor_sync(0xffffffffu, from, d);
        if (cost > 0 && (best == 0 || cost < best || (cost == best && other < from))) { best = cost; from = other; }
    }
    c.team = __shfl_sync(0xffffffffu, c.team, from);
    c.n_teams = __shfl_sync(0xffffffffu, c.n_teams, from);
    c.total = __shfl_sync(0xffffffffu, c.total, from);
    c.a = __shfl_sync(0xffffffffu, c.a, from);
    c.l = __shfl_sync(0xffffffffu, c.l, from);
    c.cost = best;
    return c;
#else
    TeamCut best = team_cut(p, grid, 0, most, pair_ticks, lone_ticks);
    for (int i = 1; i < 4; ++i) {
        const TeamCut c = team_cut(p, grid, i, most, pair_ticks, lone_ticks);
        if (c.cost > 0 && (best.cost == 0 || c.cost < best.cost)) best = c;
    }
    return best;
#endif
}

template <bool IN_PLACE, bool SPREAD>
REGIONE_HD Plan plan_shares(const PlanInput& p, int grid, bool* bad = nullptr) {
    Plan pl;
    long long items = 0, ticks = 0, span = 0;      // span: first tick of an item's last step, at most
    long long pairs = 0, lone_ticks = 0;
    int steps = 0, most = 0;                       // steps of an item (-1: they differ), full pairs of a head at most
    for (int b = 0; b < p.B; ++b) {
        const ReqShape r = req_shape<IN_PLACE>(p, b, bad);
        items += r.items;
        ticks += r.ticks;
        if (r.np > 0) span = max(span, (long long)(r.np > 1 ? kTickPair : r.w_last) * (r.steps - 1));
        if (SPREAD && r.np > 0) {
            pairs += (long long)p.H * r.full;
            most = max(most, r.full);
            if (r.full < r.np) lone_ticks += p.H * r.ticks_last;
            steps = steps == 0 || steps == r.steps ? r.steps : -1;
        }
    }
    const long long per = div_pos(items + grid - 1, grid);
    const bool whole = per * grid * 100 <= items * 106;
    if (SPREAD) {
        pl.origin = 0;
        pl.waves = 0;
        pl.team = 1;
        const long long pair_ticks = kTickStart + (long long)kTickPair * steps, fair = div_pos(ticks + grid - 1, grid);
        // (whole items need no merge, and no second start)
        const bool spread = steps > 0 && per * pair_ticks > fair + kTickStart + kTickMerge;
        if (spread && pairs >= 2 * grid) {
            if (!(whole && per * pair_ticks * 100 <= fair * kWholeWaste)) {
                pl.kind = kWaves;
                pl.waves = (int)div_pos(pairs, grid);
                long long left = pairs - (long long)pl.waves * grid;
                if (left > 0 && left * kWaveSlots < grid) { --pl.waves; left += grid; }       // (an item would meet too many shares)
                pl.origin = (pairs - left) * pair_ticks;
                pl.total = pairs * pair_ticks + lone_ticks;
                pl.chunk = max(div_pos(pl.total - pl.origin + grid - 1, grid),
                               max((long long)kTickPair * (steps - 1) / (kWaveSlots - 1) + 1, (long long)kTickPair));
                return pl;
            }
        } else if (spread && pairs > 0) {
            const TeamCut c = best_team(p, grid, most, pair_ticks, lone_ticks);
            if (c.cost > 0 && max(c.a, c.l) * 100 <= fair * 104) {
                pl.kind = kTeams;
                pl.team = c.team;
                pl.n_teams = c.n_teams;
                pl.total = c.total;
                pl.lone_total = lone_ticks;
                const long long floor_len = max((long long)kTickPair * (steps - 1) / (p.max_slots - 1) + 1, (long long)kTickPair);
                pl.chunk = max(c.a, floor_len);
                pl.lone_chunk = max(c.l, floor_len);
                return pl;
            }
        }
    }
    if (whole) {
        pl.kind = kWhole;
        pl.total = items;
        pl.chunk = max(per, 1LL);
    } else {
        pl.kind = kTicks;
        pl.total = ticks;
        pl.chunk = (ticks + grid - 1) / grid;
        // an item meets at most span / chunk + 2 shares: keep that within max_slots; and a share is
        // at least one step long, so that every share between an item's first and last holds a
        // step of it (and writes its slot)
        const long long floor_len = max(span / (p.max_slots - 1) + 1, (long long)kTickPair);
        if (pl.chunk < floor_len) pl.chunk = floor_len;
    }
    return pl;
}

// The part of one item that a CTA works on.
struct Segment {
    int b, h, qp;
    ReqShape r;
    int j_first, n_steps;   // steps [j_first, j_first + n_steps) of the item; n_steps may be 0
    int slot, n_slots;      // this share's slot among the shares that hold steps of the item
    int slot_at, slot_step; // where slot 1 of the item lies in the workspace, and how far apart the later ones do
                            // (slot 0: slot_at - 1)
    bool in_wave;           // dealt whole, ahead of the share of the axis
    long long next;         // position behind the item
};

// Whole items: the item with index `idx`.
template <bool IN_PLACE>
REGIONE_HD Segment segment_whole(const PlanInput& p, long long idx) {
    Segment sg;
    long long base = 0;
    int b = 0;
    ReqShape r = req_shape<IN_PLACE>(p, 0);
    while (idx >= base + r.items && b + 1 < p.B) {
        base += r.items;
        ++b;
        r = req_shape<IN_PLACE>(p, b);
    }
    const long long item = idx - base;
    sg.b = b; sg.r = r;
    sg.h = r.np > 0 ? (int)div_pos(item, r.np) : 0;
    sg.qp = (int)(item - (long long)sg.h * r.np);
    sg.j_first = 0;
    sg.n_steps = r.np > 0 ? r.steps : 0;
    sg.slot = 0; sg.n_slots = 1;
    sg.next = idx + 1;
    return sg;
}

// The steps that share `c` owns of an item whose first step begins at tick `first_tick` (ticks behind the axis's origin),
// and the shares that the item meets.
REGIONE_HD void cut_item(Segment& sg, long long chunk, long long first_tick, int w, int c) {
    const long long lo = (long long)c * chunk, hi = lo + chunk;
    const int steps = sg.r.steps;
    long long s_lo = lo <= first_tick ? 0 : div_pos(lo - first_tick + w - 1, w);
    long long s_hi = hi <= first_tick ? 0 : div_pos(hi - first_tick + w - 1, w);
    s_lo = min(s_lo, (long long)steps);
    s_hi = min(s_hi, (long long)steps);
    sg.j_first = (int)s_lo;
    sg.n_steps = (int)(s_hi - s_lo);
    const int c_first = (int)div_pos(first_tick, chunk);
    sg.n_slots = (int)div_pos(first_tick + (long long)w * (steps - 1), chunk) - c_first + 1;
    sg.slot = c - c_first;
}

// Tick plan: the item that contains tick `pos`, and the steps of it that share `c` owns.
template <bool IN_PLACE>
REGIONE_HD Segment segment_ticks(const PlanInput& p, const Plan& pl, long long pos,
                                                 int c) {
    Segment sg;
    long long base = 0;
    int b = 0;
    ReqShape r = req_shape<IN_PLACE>(p, 0);
    while (pos >= base + r.ticks && b + 1 < p.B) {
        base += r.ticks;
        ++b;
        r = req_shape<IN_PLACE>(p, b);
    }
    sg.b = b; sg.r = r;
    if (r.np == 0) {                                  // nothing left behind the last live request
        sg.h = sg.qp = sg.j_first = sg.n_steps = sg.slot = 0;
        sg.n_slots = 1;
        sg.next = pl.total;
        return sg;
    }
    const long long rel = pos - base;
    sg.h = (int)div_pos(rel, r.head_ticks);
    const long long rem = rel - (long long)sg.h * r.head_ticks;
    sg.qp = (int)min(div_pos(rem, r.ticks_full), (long long)(r.np - 1));
    const long long t0 = base + (long long)sg.h * r.head_ticks + (long long)sg.qp * r.ticks_full;
    const bool last = sg.qp == r.np - 1;
    cut_item(sg, pl.chunk, t0 + kTickStart, last ? r.w_last : kTickPair, c);
    sg.next = t0 + (last ? r.ticks_last : r.ticks_full);
    return sg;
}

// Plans of the launches that mind the order of the keys (SPREAD), one function for all of them: the code of a plan is read
// once a launch, from memory, and what is not there is not waited for (three functions -> one: 2048 of 8448 rows with a
// capacity a tenth above 235.6 -> 221.5 us).  `by_head`: the axis holds the pairs of a head one after the other (kTicks, kWhole).
// Else it holds the full pairs of every head, `team` of them side by side, and behind them the pairs with one live query
// tile.  The item of the `member`th of a team that contains position `pos`, and the steps of it that share `c` of `chunk`
// ticks owns, the shares counted from tick `origin` on; whole: positions count items, and all steps are owned.
template <bool IN_PLACE>
REGIONE_HD Segment segment_spread(const PlanInput& p, long long pos, bool whole, bool by_head, long long origin, long long chunk,
                                  int c, int team, int member) {
    Segment sg;
    long long base = 0, col = 0, head = 0;
    int b = 0, cols = 0;
    bool lone = false;
    for (;;) {
        sg.r = req_shape<IN_PLACE>(p, b);
        const int sides = team == 1 ? sg.r.full : (int)((unsigned)(sg.r.full + team - 1) / (unsigned)team);
        cols = by_head ? sg.r.np : lone ? sg.r.np - sg.r.full : sides;
        col = whole ? 1 : lone ? sg.r.ticks_last : sg.r.ticks_full;
        head = by_head && !whole ? sg.r.head_ticks : cols * col;
        const long long len = p.H * head;
        if (pos < base + len || ((lone || by_head) && b + 1 == p.B)) break;
        base += len;
        if (++b == p.B) { b = 0; lone = true; }
    }
    sg.b = b;
    if (cols == 0) {                                  // nothing left behind the last live request
        sg.h = sg.qp = sg.j_first = sg.n_steps = sg.slot = 0;
        sg.n_slots = 1;
        sg.next = pos + 1;
        return sg;
    }
    sg.h = (int)div_pos(pos - base, head);
    const long long h0 = base + sg.h * head;
    const int s = (int)min(div_pos(pos - h0, col), (long long)(cols - 1));
    const long long t0 = h0 + s * col;
    lone |= by_head && s == cols - 1 && sg.r.full < sg.r.np;
    sg.qp = by_head ? s : lone ? sg.r.full : s * team + member;
    if (whole) {
        sg.j_first = 0;
        sg.n_steps = sg.r.steps;
        sg.slot = 0; sg.n_slots = 1;
    } else {
        cut_item(sg, chunk, t0 + kTickStart - origin, lone ? p.single : kTickPair, c);
    }
    if (sg.qp >= (lone ? sg.r.np : sg.r.full)) sg.n_steps = 0;        // (a team wider than what is left of the head)
    sg.next = t0 + (whole ? 1 : lone ? sg.r.ticks_last : col);
    return sg;
}

// Share of a CTA (block of a grid) on the cost axis.  The first share of an item waits for the later ones, so shares are dealt
// from the last block to the first: blocks become resident in the order of their indexes on this GPU, and a block
// waits only for blocks ahead of it, whatever else runs.  CUDA does not promise that order; were it another, a wait
// for a block that cannot start would end with its bound and REGIONE_DEV_TIMEOUT.
REGIONE_HD int share_of(int grid, int block) { return grid - 1 - block; }

// What one CTA works on, segment by segment.
template <bool IN_PLACE, bool SPREAD>
struct ShareWalk {
    Plan pl;
    long long pos, hi;
    int wave;                    // (kWaves) next wave
    int share, step, member;     // share of the axis, CTAs from it to the next share, member of its team

    REGIONE_HD void begin(const PlanInput& p, int grid, int block, bool* bad) {
        pl = plan_shares<IN_PLACE, SPREAD>(p, grid, bad);
        wave = member = 0;
        step = 1;
        share = share_of(grid, block);
        long long end = pl.total;
        if (pl.kind == kWhole) {
            // (dealt round-robin, so that the CTAs running at any one time work on neighbouring items, which share K/V
            // tiles in L2)
            pos = block;
            hi = end;
            return;
        }
        if (SPREAD && pl.kind == kTeams) {
            if (share < pl.team * pl.n_teams) {
                step = pl.team;
                member = share % step;
                share /= step;
            } else {
                share -= pl.team * pl.n_teams;
                pl.origin = pl.total;
                pl.chunk = pl.lone_chunk;
                end += pl.lone_total;
            }
        }
        pos = (SPREAD ? pl.origin : 0) + share * pl.chunk;         // (a share of steps is one contiguous range)
        hi = pos + pl.chunk < end ? pos + pl.chunk : end;
    }
    // The next segment, possibly without steps; false when the share ends.
    REGIONE_HD bool next(const PlanInput& p, int grid, int block, Segment& it) {
        const bool in_wave = SPREAD && pl.kind == kWaves && wave < pl.waves;
        if (!in_wave && pos >= hi) return false;
        const bool whole = pl.kind == kWhole || in_wave;
        if constexpr (SPREAD)
            it = segment_spread<IN_PLACE>(p, in_wave ? (long long)wave * grid + block : pos, whole,
                                          pl.kind == kTicks || pl.kind == kWhole, pl.origin, pl.chunk, share, pl.team, member);
        else
            it = whole ? segment_whole<IN_PLACE>(p, pos) : segment_ticks<IN_PLACE>(p, pl, pos, share);
        it.in_wave = in_wave;
        it.slot_at = ((it.b * p.H + it.h) * p.P_cap + it.qp) * p.max_slots + 1;
        it.slot_step = 1;
        if (SPREAD && pl.kind == kWaves) {          // (every share has room for two, in what the items have together)
            it.slot_at = 2 * (share - it.slot + 1);
            it.slot_step = 2;
        }
        if (in_wave) ++wave;
        else pos = whole ? pos + grid : it.next;
        return true;
    }
};

}  // namespace regione
