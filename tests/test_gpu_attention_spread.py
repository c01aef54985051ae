"""Attention whose K and V are more than L2 keeps: pairs of query tiles dealt in waves, or teams of thread blocks that walk a
head together.  Compared with the library's CUDA-core statement of the attention equation."""
import pytest

from gpu_util import assert_close, dev_i32, host_f64
from paper_2510_25590_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,n_q,n_f,n_c", [
    (64, 24, [13 * 256 + 100], [10291], [0]),         # two waves, the rest of the pairs and then the lone tiles cut
    (64, 24, [25 * 256], [10300], [0]),               # eight pairs behind four waves: three waves
    (128, 24, [13 * 256 + 1], [1], [5200]),          # a fresh key tile of one key, a lone tile of one row
    (128, 24, [819], [819], [7885]),                 # teams of three, lone tiles apart
    (64, 24, [2048], [2048], [8300]),                # teams of half a head's pairs
    (128, 8, [1100, 1090], [1100, 1090], [6700, 6700]),              # two requests with the same key tiles
    (128, 8, [1100, 700], [1100, 700], [6700, 7100]),                # other queries: teams of which some have no pair
    (128, 8, [1100, 0, 300], [1100, 0, 300], [6700, 0, 2000]),       # key tiles that differ, a request without queries
    (64, 40, [100], [100], [6100]),                  # lone tiles only
])
def test_spread_plans(D, H, n_q, n_f, n_c):
    import torch
    g = torch.Generator(device="cuda").manual_seed(D + H + n_q[0])
    r = lambda n: torch.randn((len(n_q), max(n), H, D), generator=g, device="cuda", dtype=torch.bfloat16)
    q, kf, vf, kc, vc = r(n_q), r(n_f), r(n_f), r(n_c), r(n_c)
    assert 4 * D * H * len(n_q) * (max(n_f) + max(n_c)) >= 60 << 20
    counts = [dev_i32(n) for n in (n_q, n_f, n_c)]
    ws = torch.full((binding.region_attention_workspace(len(n_q), max(n_q), max(n_f), max(n_c), H, D),), 255, dtype=torch.uint8,
                    device="cuda")
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
