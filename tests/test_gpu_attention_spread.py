"""Attention whose K and V are more than L2 keeps: pairs of query tiles dealt in waves, or teams of thread blocks that walk a
head together.  Compared with the library's CUDA-core statement of the attention equation."""
import pytest

from gpu_util import assert_close, dev_i32, host_f64
from paper_2510_25590_b200 import binding
from test_attention_plan import IN_WAVE, TEAMS, TICKS, WAVES, plan
from test_gpu_attention_forms import _step

pytestmark = pytest.mark.gpu


def minds_order(B, caps, H, D, out_cap=0, refreshes=0):
    form = binding.load().regione_selftest_attention_form(B, *caps, H, D, out_cap, refreshes)
    assert form >= 0
    return form >= 3


def plan_of(n_q, n_f, n_c, caps, H):
    """Kind of the plan of these counts, and the waves ahead of its cut part."""
    import torch
    segs, _ = plan(n_q, n_f, n_c, caps, H, sms=torch.cuda.get_device_properties(0).multi_processor_count)
    return max(segs[:, 11]), (segs[segs[:, 0] == 0][:, 11] == IN_WAVE).sum()


# n_q ... : live counts; room: rows of capacity above the largest of them; kind: plan that the launch walks (None: launched in a
# form that does not mind the order), with the number of waves
@pytest.mark.parametrize("D,H,n_q,n_f,n_c,room,kind", [
    (64, 24, [13 * 256 + 100], [10291], [0], 0, None),               # (heads of 64 mind the order from 90 MB on)
    (64, 24, [25 * 256], [10300], [0], 0, None),
    (64, 24, [14 * 256 + 100], [16300], [0], 0, (WAVES, 2)),         # two waves, the rest of the pairs and then the lone tiles cut
    (128, 24, [13 * 256 + 1], [1], [5200], 0, (WAVES, 1)),           # a fresh key tile of one key, a lone tile of one row
    (128, 24, [14 * 256], [5200], [0], 0, (WAVES, 2)),
    (128, 24, [25 * 256], [5200], [0], 0, (WAVES, 3)),               # eight pairs behind four waves: three waves
    (128, 24, [819], [819], [7885], 0, (TEAMS, 0)),                  # teams of three, lone tiles apart
    (128, 24, [819], [819], [7885], 400, (TEAMS, 0)),                # ... chosen from the counts
    (128, 24, [2048], [2048], [6400], 0, (TEAMS, 0)),                # teams of half a head's pairs
    (64, 24, [2048], [2048], [8300], 0, None),
    (128, 8, [1100, 1090], [1100, 1090], [6700, 6700], 0, None),                     # (short shares, merged by a kernel)
    (128, 12, [1100, 1090], [1100, 1090], [6700, 6700], 0, (TEAMS, 0)),              # two requests with the same key tiles
    (128, 24, [1024, 1000], [1024, 1000], [5000, 5024], 0, (TEAMS, 0)),
    (128, 8, [1100, 700], [1100, 700], [6700, 7100], 0, None),
    (128, 12, [1100, 700], [1100, 700], [6700, 7100], 0, (TICKS, 0)),                # other queries: some members would idle
    (64, 24, [594] * 4, [594] * 4, [6211] * 4, 0, (TEAMS, 0)),                       # (as whole items far from balanced)
    (128, 8, [1100, 0, 300], [1100, 0, 300], [6700, 0, 2000], 0, (TICKS, 0)),        # key tiles that differ, a request without queries
    (128, 24, [3584, 256, 0], [3584, 256, 0], [2000, 5328, 5584], 0, None),          # (whole items of full capacities balance)
    (128, 24, [600], [600], [6000], 700, None),
    (64, 40, [100], [100], [6100], 0, None),                         # one pair a head
])
def test_spread_plans(D, H, n_q, n_f, n_c, room, kind):
    import torch
    caps = tuple(max(n) + room * (max(n) > 0) for n in (n_q, n_f, n_c))
    assert minds_order(len(n_q), caps, H, D) == (kind is not None)
    if kind is not None:
        assert plan_of(n_q, n_f, n_c, caps, H) == kind
    g = torch.Generator(device="cuda").manual_seed(D + H + n_q[0])
    r = lambda n: torch.randn((len(n_q), n, H, D), generator=g, device="cuda", dtype=torch.bfloat16)
    q, kf, vf, kc, vc = r(caps[0]), r(caps[1]), r(caps[1]), r(caps[2]), r(caps[2])
    assert 4 * D * H * len(n_q) * (max(n_f) + max(n_c)) >= 60 << 20
    counts = [dev_i32(n) for n in (n_q, n_f, n_c)]
    ws = torch.full((binding.region_attention_workspace(len(n_q), *caps, H, D),), 255, dtype=torch.uint8, device="cuda")
    status, out, want = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros_like(q), torch.zeros_like(q)
    binding.crosscheck_region_attention(q, kf, vf, kc, vc, *counts, want)
    graph = torch.cuda.CUDAGraph()
    binding.region_attention(q, kf, vf, kc, vc, *counts, out, workspace=ws, dev_status=status)
    torch.cuda.synchronize()
    first = out.clone()
    with torch.cuda.graph(graph):
        binding.region_attention(q, kf, vf, kc, vc, *counts, out, workspace=ws, dev_status=status)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert int(status[0]) == 0 and torch.equal(out, first)
    for b, n in enumerate(n_q):
        if n > 0:
            assert_close(host_f64(out[b, :n]), host_f64(want[b, :n]), f"request {b}")


def test_one_pair_a_head_behind_a_row_list():
    """K and V that pass through once (told to leave L2 first): rows of a ragged pair at their places."""
    import torch
    H, D, n_q, n_c = 24, 128, 205, 5400
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda n: torch.randn((1, n, H, D), generator=g, device="cuda", dtype=torch.bfloat16)
    q, kf, vf, kc, vc = r(n_q), r(n_q), r(n_q), r(n_c), r(n_c)
    rows = torch.randperm(n_q + n_c, device="cuda", generator=g)[:n_q].int()[None].contiguous()
    nq, nc = dev_i32([n_q]), dev_i32([n_c])
    assert 4 * D * H * (n_q + n_c) >= 60 << 20
    ws = torch.empty(binding.region_attention_workspace(1, n_q, n_q, n_c, H, D), dtype=torch.uint8, device="cuda")
    status, want = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros_like(q)
    full = torch.zeros((1, n_q + n_c, H, D), dtype=torch.bfloat16, device="cuda")
    binding.region_attention_scatter(q, kf, vf, kc, vc, nq, nq, nc, full, rows, workspace=ws, dev_status=status)
    binding.crosscheck_region_attention(q, kf, vf, kc, vc, nq, nq, nc, want)
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    assert_close(host_f64(full[0, rows[0].long()]), host_f64(want[0]), "rows")


@pytest.mark.parametrize("D,grid,ratio,ne_cap", [
    (64, (64, 80), 0.2, 1024),                       # teams, n_full = 10752
    (128, (64, 64), 0.2, 896),                       # the lone tiles apart
    (128, (65, 63), 0.26, 1152),
    (128, (64, 64), 0.2, 1024),                      # teams, more room than pairs
    (64, (64, 80), 0.8, 4096),                       # waves
])
def test_refreshing_steps(D, grid, ratio, ne_cap):
    """Steps that refresh the cache and mind the order of the keys: the planning warp's cursor lies in shared memory."""
    n_full = 512 + 2 * grid[0] * grid[1]
    assert minds_order(1, (ne_cap, n_full, 0), 24, D, n_full, 1)
    _step(D, grid, 512, 24, ratio, ne_cap)
