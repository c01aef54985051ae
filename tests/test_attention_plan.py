"""The shares that the attention kernel cuts a call into cover every key tile of every item once, and the shares that cut
an item can be put together again (host run of the functions that the kernel's planning warps run)."""
import ctypes
import random

import numpy as np
import pytest

from paper_2510_25590_b200 import binding

TILE, PAIR = 128, 256
WHOLE, TICKS, WAVES, TEAMS, IN_WAVE = 0, 1, 2, 3, -1


def plan(n_q, n_fresh, n_cache, caps, H, all_rows=0, spread=1, sms=148):
    B = len(n_q)
    i32 = lambda v: np.ascontiguousarray(v, dtype=np.int32)
    q, f, c, shape = i32(n_q), i32(n_fresh), i32(n_cache), np.zeros(4, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    call = lambda out, n: binding.load().regione_selftest_attention_plan(p(q), p(f), p(c), B, *caps, H, all_rows, spread, sms,
                                                                         p(shape), p(out), n)
    n = call(np.zeros(12, np.int32), 0)
    out = np.zeros((max(n, 1), 12), np.int32)
    assert n >= 0 and call(out, n) == n
    return out[:n], shape


def check(n_q, n_fresh, n_cache, caps, H, all_rows=0, spread=1, sms=148):
    segs, (grid, p_cap, max_slots, _) = plan(n_q, n_fresh, n_cache, caps, H, all_rows, spread, sms)
    tiles = lambda n: -(-n // TILE)
    items, order = {}, {}
    for at, (block, b, h, qp, j, n, slot, n_slots, slot_at, slot_step, share_step, kind) in enumerate(segs.tolist()):
        items.setdefault((b, h, qp), []).append((slot, j, n, block, n_slots, slot_at, slot_step, share_step, at))
        order.setdefault(block, []).append((at, kind))
    expected = set()
    used = set()
    for b, (q, f, c) in enumerate(zip(n_q, n_fresh, n_cache)):
        if all_rows and q + c == all_rows:
            steps = tiles(all_rows)
        elif all_rows:
            steps = tiles(c) + tiles(q)
        else:
            steps = tiles(c) + tiles(f)
        for h in range(H):
            for qp in range(-(-q // PAIR)):
                expected.add((b, h, qp))
                parts = sorted(items.get((b, h, qp), []))
                # slot s holds the s-th run of key tiles, and there are as many as every part says
                assert [p[0] for p in parts] == list(range(len(parts))) and all(p[4] == len(parts) for p in parts)
                at = 0
                for p in parts:
                    assert p[1] == at and p[2] > 0
                    at += p[2]
                assert at == max(steps, 1)
                if len(parts) == 1:
                    continue
                slot_at, slot_step, share_step = parts[0][5:8]
                assert all(p[5:8] == (slot_at, slot_step, share_step) for p in parts)
                assert len(parts) <= 8                              # what the merge kernel holds
                for p in parts:
                    where = slot_at - 1 if p[0] == 0 else slot_at + (p[0] - 1) * slot_step
                    assert 0 <= where < len(n_q) * H * p_cap * max_slots and where not in used
                    used.add(where)
                    # the shares of an item are share_step apart, later ones in blocks that start earlier
                    assert p[3] == parts[0][3] - p[0] * share_step
                    axis = [a for a, kind in order[p[3]] if kind != IN_WAVE]
                    if p[0] == 0:
                        assert p[8] == order[p[3]][-1][0]           # the first share reaches the item last
                    else:
                        assert p[8] == axis[0]                      # the others begin (the cut part of) their share with it
    assert set(items) == expected
    return segs, grid


@pytest.mark.parametrize("name,n_q,n_keys,caps,H,all_rows,kind", [
    ("8704 x 8704: waves, then the rest cut", [8704], 8704, (8704, 8704, 0), 24, 0, WAVES),
    ("8448 x 8448", [8448], 8448, (8448, 8448, 0), 24, 0, WAVES),
    ("819 of 8704: three pairs a team, lone tiles apart", [819], 8704, (896, 896, 8704), 24, 0, TEAMS),
    ("the same, K and V in place", [819], 8704, (896, 8704, 0), 24, 8704, TEAMS),
    ("2048 of 8448", [2048], 8448, (2048, 8448, 0), 24, 8448, TEAMS),
    ("1075 of 8448", [1075], 8448, (1075, 1075, 7373), 24, 0, TEAMS),
    ("eight pairs more than two waves: one wave", [256 * 38], 2048, (256 * 38, 2048, 0), 8, 0, WAVES),
    ("three of 4916 x 4916: whole items fill the rounds", [4916] * 3, 4916, (4916, 4916, 0), 24, 0, WHOLE),
    ("requests whose key tiles differ", [819, 600], 8704, (896, 896, 8704), 24, 0, TICKS),
])
def test_plans_of_known_shapes(name, n_q, n_keys, caps, H, all_rows, kind):
    if all_rows:
        f, c = [0] * len(n_q), [all_rows - q for q in n_q]
    elif caps[2] == 0:
        f, c = [n_keys] * len(n_q), [0] * len(n_q)
    else:
        f, c = list(n_q), [n_keys - q for q in n_q]
        c[1:] = [x - 2000 for x in c[1:]]
    segs, grid = check(n_q, f, c, caps, H, all_rows)
    assert kind in segs[:, 11]
    # whole pairs and shares together are balanced: no block has much more than the mean cost (whole items: by a merge and a second start)
    nq = np.array(n_q)[segs[:, 1]]
    cost = 80 + segs[:, 5] * np.where(nq - segs[:, 3] * PAIR > TILE, 16, 9)
    load = np.bincount(segs[:, 0], weights=cost, minlength=grid)
    assert load.max() <= 1.15 * load.mean() + 205


@pytest.mark.parametrize("seed", range(12))
def test_plans_cover_every_step_once(seed):
    rng = random.Random(seed)
    near = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))
    for _ in range(25):
        B, H, sms = rng.choice([1, 1, 2, 3, 5]), rng.choice([1, 3, 4, 8, 24]), rng.choice([148, 148, 132, 7, 1])
        q_cap = near(1, 9000 if H < 24 else 4000)
        same = rng.random() < 0.6
        n_q = [q_cap if same else rng.randint(0, q_cap) for _ in range(B)]
        mode = rng.choice(["cache", "full", "place"])
        if mode == "place":
            rows = q_cap + near(1, 9000)
            f, c, caps, all_rows = [0] * B, [rows - q - (rng.random() < 0.1) for q in n_q], (q_cap, rows, 0), rows
        elif mode == "full":
            f, c, caps, all_rows = n_q, [0] * B, (q_cap, q_cap, 0), 0
        else:
            c_cap = near(1, 9000)
            f, c = n_q, [c_cap if same else rng.randint(0, c_cap) for _ in range(B)]
            caps, all_rows = (q_cap, q_cap, c_cap), 0
        for spread in (0, 1, 2):
            check(n_q, f, c, caps, H, all_rows, spread, sms)


@pytest.mark.parametrize("rows", [819, 1075, 1229, 2048])
@pytest.mark.parametrize("room", [1.1, 1.25, 1.5, 2.0])
@pytest.mark.parametrize("refreshes", [False, True])
def test_capacities_above_the_counts_keep_the_teams(rows, room, refreshes):
    """The teams follow the live counts: a capacity above them changes nothing but the longest cut that its workspace holds."""
    def teams(cap):
        cap = -(-cap // TILE) * TILE
        if refreshes:
            segs, _ = check([rows], [0], [8448 - rows], (cap, 8448, 0), 24, 8448)
        else:
            segs, _ = check([rows], [rows], [8448 - rows], (cap, cap, 8448), 24)
        shape = plan([rows], [0 if refreshes else rows], [8448 - rows], (cap, 8448, 0) if refreshes else (cap, cap, 8448), 24,
                     8448 if refreshes else 0)[1]
        return segs, shape[2], shape[3]
    segs, slots, team = teams(rows)
    roomy, roomy_slots, roomy_team = teams(int(rows * room))
    assert team == roomy_team > 1 and set(roomy[:, 11]) == {TEAMS}
    if slots == roomy_slots:
        assert np.array_equal(segs[:, :8], roomy[:, :8])


@pytest.mark.parametrize("n_q,caps,all_rows", [
    ([8211], (8211, 8211, 0), 0),                    # waves, the lone tiles behind them
    ([6500], (6500, 6500, 0), 0),
    ([819], (896, 8448, 0), 8448),                   # teams, the lone tiles apart
    ([1075], (1152, 8448, 0), 8448),
    ([1638], (1664, 8448, 0), 8448),
])
def test_lone_tiles_of_a_refreshing_launch_weigh_three_quarters(n_q, caps, all_rows):
    f, c = ([0], [all_rows - n_q[0]]) if all_rows else (n_q, [0])
    segs, grid = check(n_q, f, c, caps, 24, all_rows, spread=2)
    assert set(segs[:, 11]) & {WAVES, TEAMS}
    cost = 80 + segs[:, 5] * np.where(n_q[0] - segs[:, 3] * PAIR > TILE, 16, 12)
    load = np.bincount(segs[:, 0], weights=cost, minlength=grid)
    assert load.max() <= 1.05 * load.mean() + 32     # (teams are taken within 4 % of the mean; a step each way)


@pytest.mark.parametrize("n_q,kind", [([1000, 1024], TEAMS), ([4096, 3900], WAVES), ([819, 1024], TICKS)])
def test_requests_of_other_counts(n_q, kind):
    """Counts of the same number of pairs walk in teams; where members would idle the cost axis is the shorter plan."""
    segs, _ = check(n_q, [0, 0], [8448 - n for n in n_q], (4096, 8448, 0), 24, 8448)
    assert kind in segs[:, 11]
