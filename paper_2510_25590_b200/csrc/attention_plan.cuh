// How the work of one attention launch is cut into shares, one per CTA.  Every CTA derives the same plan from the
// request counts in device memory; the functions also run on the host, where a test checks that the shares cover
// every step once.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

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
    int team;            // (SPREAD) 0: whole pairs in waves; else CTAs that walk a head's keys together (see plan_shares)
};

// Shares are cut on a cost axis measured in ticks, not in steps, so that they take about the same
// time: a key tile of a full query pair costs kTickPair, a key tile of a pair with one live query
// tile kTickSingle (its even and odd key tiles run side by side on the two tile roles; measured per
// thread block against its share's composition: 0.55 to 0.56 of a pair's step, not half), and every
// item starts with kTickStart ticks that stand for the drain of the previous segment and the fill of
// the new one (measured the same way: 3.5 to 6 pair steps depending on the workload, 5 with 819 x 8704 and
// 1075 x 8448 keys, 24 heads of 128; 100, 120 and 140 ticks for items that a first share merges: 0 to +3 %).
constexpr int kTickPair = 16, kTickSingle = 9, kTickStart = 80;
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
    r.w_last = (nq - (r.np - 1) * 2 * kBM > kBM) ? kTickPair : kTickSingle;
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
//    shared by the CTAs that are in no team, as many as make the two kinds of share equally long.
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

template <bool IN_PLACE, bool SPREAD>
REGIONE_HD Plan plan_shares(const PlanInput& p, int grid, bool* bad = nullptr) {
    Plan pl;
    long long items = 0, ticks = 0, span = 0;      // span: first tick of an item's last step, at most
    long long pairs = 0, supers = 0, lone_ticks = 0;
    int steps = 0;                                 // steps of an item (-1: they differ)
    for (int b = 0; b < p.B; ++b) {
        const ReqShape r = req_shape<IN_PLACE>(p, b, bad);
        items += r.items;
        ticks += r.ticks;
        if (r.np > 0) span = max(span, (long long)(r.np > 1 ? kTickPair : r.w_last) * (r.steps - 1));
        if (SPREAD && r.np > 0) {
            pairs += (long long)p.H * r.full;
            if (p.team > 0) supers += (long long)p.H * ((r.full + p.team - 1) / p.team);
            if (r.full < r.np) lone_ticks += p.H * r.ticks_last;
            steps = steps == 0 || steps == r.steps ? r.steps : -1;
        }
    }
    const long long per = div_pos(items + grid - 1, grid);
    const bool whole = per * grid * 100 <= items * 106;
    if (SPREAD) {
        pl.origin = 0;
        pl.waves = 0;
        const long long pair_ticks = kTickStart + (long long)kTickPair * steps, fair = div_pos(ticks + grid - 1, grid);
        // (whole items need no merge, and no second start)
        const bool spread = steps > 0 && per * pair_ticks > fair + kTickStart + kTickMerge;
        if (spread && p.team == 0 && pairs >= 2 * grid && !(whole && per * pair_ticks * 100 <= fair * kWholeWaste)) {
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
        if (spread && p.team > 0 && supers > 0) {
            // as many teams as make their shares as long as those of the CTAs in no team
            const long long total = supers * pair_ticks;
            int T = (int)min(div_pos(grid * total, lone_ticks + p.team * total), (long long)(grid / p.team));
            const int rest = grid - p.team * T;
            if (T > 0 && (rest > 0 || lone_ticks == 0)) {
                long long a = div_pos(total + T - 1, T), l = rest > 0 ? div_pos(lone_ticks + rest - 1, rest) : 0;
                if (a > l && rest > p.team) {
                    const long long a1 = div_pos(total + T, T + 1), l1 = div_pos(lone_ticks + rest - p.team - 1, rest - p.team);
                    if (max(a1, l1) < a) { ++T; a = a1; l = l1; }
                }
                if (max(a, l) * 100 <= fair * 104) {
                    pl.kind = kTeams;
                    pl.team = p.team;
                    pl.n_teams = T;
                    pl.total = total;
                    pl.lone_total = lone_ticks;
                    const long long floor_len = max((long long)kTickPair * (steps - 1) / (p.max_slots - 1) + 1, (long long)kTickPair);
                    pl.chunk = max(a, floor_len);
                    pl.lone_chunk = max(l, floor_len);
                    return pl;
                }
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

// Whole items: the item with index `idx`, of all of them or of those with two live query tiles.
template <bool IN_PLACE>
REGIONE_HD Segment segment_whole(const PlanInput& p, long long idx, bool full_only) {
    Segment sg;
    long long base = 0;
    int b = 0;
    ReqShape r = req_shape<IN_PLACE>(p, 0);
    int cols = full_only ? r.full : r.np;
    while (idx >= base + (long long)p.H * cols && b + 1 < p.B) {
        base += (long long)p.H * cols;
        ++b;
        r = req_shape<IN_PLACE>(p, b);
        cols = full_only ? r.full : r.np;
    }
    const long long item = idx - base;
    sg.b = b; sg.r = r;
    sg.h = cols > 0 ? (int)div_pos(item, cols) : 0;
    sg.qp = (int)(item - (long long)sg.h * cols);
    sg.j_first = 0;
    sg.n_steps = cols > 0 ? r.steps : 0;
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

// Waves and teams: the axis holds the full pairs of every head, `team` of them side by side, and behind them the pairs
// with one live query tile.  The item of the `member`th of a team that contains tick `pos`, and the steps of it that
// share `c` of `chunk` ticks owns, the shares counted from tick `origin` on.
template <bool IN_PLACE>
REGIONE_HD Segment segment_spread(const PlanInput& p, long long pos, long long origin, long long chunk, int c,
                                                  int team, int member) {
    Segment sg;
    long long base = 0, col = 0;
    int b = 0, cols = 0;
    bool lone = false;
    for (;;) {
        sg.r = req_shape<IN_PLACE>(p, b);
        cols = lone ? sg.r.np - sg.r.full : (sg.r.full + team - 1) / team;
        col = lone ? sg.r.ticks_last : sg.r.ticks_full;
        const long long len = p.H * cols * col;
        if (pos < base + len || (lone && b + 1 == p.B)) break;
        base += len;
        if (++b == p.B) { b = 0; lone = true; }
    }
    sg.b = b;
    const long long at = div_pos(pos - base, col);
    sg.h = cols > 0 ? (int)div_pos(at, cols) : 0;
    const int s = (int)(at - (long long)sg.h * cols);
    sg.qp = lone ? sg.r.full : s * team + member;
    const long long t0 = base + at * col;
    cut_item(sg, chunk, t0 + kTickStart - origin, lone ? kTickSingle : kTickPair, c);
    if (sg.qp >= (lone ? sg.r.np : sg.r.full)) sg.n_steps = 0;        // (a team wider than what is left of the head)
    sg.next = t0 + col;
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
        it = whole ? segment_whole<IN_PLACE>(p, in_wave ? (long long)wave * grid + block : pos, in_wave)
             : !SPREAD || pl.kind == kTicks
                 ? segment_ticks<IN_PLACE>(p, pl, pos, share)
                 : segment_spread<IN_PLACE>(p, pos, pl.origin, pl.chunk, share, pl.kind == kTeams ? pl.team : 1, member);
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

// ---- host side: what is decided from the capacities -------------------------------------------------------------

// CTAs of a team (0: waves).  One team for all pairs of a head, or for half of them where the grid divides better by that
// (the second reads K and V a second time).
inline int choose_team(const PlanInput& p, int grid, int nt) {
    const int tiles = (p.Nq_cap + kBM - 1) / kBM, full = tiles / 2;
    const long long heads = (long long)p.B * p.H;
    if (heads * full >= 2LL * grid) return 0;
    const double pair = kTickStart + (double)kTickPair * nt, lone = tiles % 2 ? heads * (kTickStart + (double)kTickSingle * nt) : 0;
    int team = 1;
    double best = 0;
    for (int k = 1; k <= 2 && full > 0; ++k) {
        const int g = (full + k - 1) / k;
        const int T0 = (int)std::min(grid * heads * k * pair / (lone + g * heads * k * pair), (double)(grid / g));
        for (int T = std::max(T0, 1); T <= T0 + 1 && g * T <= grid; ++T) {
            const int rest = grid - g * T;
            if (rest == 0 && lone > 0) continue;
            const double cost = std::max(heads * k * pair / T, lone > 0 ? lone / rest : 0.) * (k == 2 ? 1.015 : 1.);
            if (best == 0 || cost < best) { best = cost; team = g; }
        }
    }
    return team;
}

}  // namespace regione
