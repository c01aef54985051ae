"""The forms of the attention at the sizes that take them, told by the number of kernels a call launches: one where the
first share of a cut item merges it (or a cluster shares it), two with a merge kernel behind.  Compared with the library's
CUDA-core statement of the attention equation, an arithmetic path of its own."""
import numpy as np
import pytest

from gpu_util import assert_close, dev_i32, host_f64
from paper_2510_25590_b200 import binding
from paper_2510_25590_b200.step import RegionStep, StepShapes
from test_gpu_region_step_call import _inputs

pytestmark = pytest.mark.gpu

H, NQ, NC = 24, 819, 7885        # three pairs of query tiles and a lone tile per head, 69 key tiles: cut, not clustered


def _launched(call):
    before = binding.kernel_launches()
    call()
    return binding.kernel_launches() - before


def _rand(seed, *shape, std=1.0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16) * std


def _want(q, k, v, softmax_scale=0.0):
    """Rows of q [1, n, H, D] against all rows of k, v."""
    import torch
    n = lambda t: dev_i32([t.shape[1]])
    out = torch.zeros_like(q)
    binding.crosscheck_region_attention(q, k, v, None, None, n(q), n(k), dev_i32([0]), out, softmax_scale=softmax_scale)
    return host_f64(out)[0]


def _case(D, kv=(NQ, NQ, NC, NC)):
    import torch
    q, kf, vf, kc, vc = (_rand(D + i, 1, n, H, D) for i, n in enumerate((NQ, *kv)))
    vf, vc = vf * 0.5, vc * 0.5
    ws = torch.empty(binding.region_attention_workspace(1, NQ, NQ, NC, H, D), dtype=torch.uint8, device="cuda")
    return q, kf, vf, kc, vc, dev_i32([NQ]), dev_i32([NC]), ws, torch.zeros(1, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("D", [64, 128])
def test_first_share_puts_rows_at_their_places_and_drops_bad_ones(D):
    import torch
    q, kf, vf, kc, vc, nq, nc, ws, status = _case(D)
    rows = torch.randperm(NQ + NC, generator=torch.Generator().manual_seed(D))[:NQ].int().cuda()[None].contiguous()
    bad = (5, 300, 818)                          # in a cut pair's two tiles and in the lone tile
    rows[0, bad[0]], rows[0, bad[1]], rows[0, bad[2]] = -1, NQ + NC, 2 ** 30
    full = torch.full((1, NQ + NC, H, D), -3.0, dtype=torch.bfloat16, device="cuda")
    assert _launched(lambda: binding.region_attention_scatter(q, kf, vf, kc, vc, nq, nq, nc, full, rows, workspace=ws,
                                                              dev_status=status)) == 1
    torch.cuda.synchronize()
    assert int(status[0]) == binding.DEV_BOUNDS
    want = _want(q, torch.cat([kf, kc], 1), torch.cat([vf, vc], 1))
    keep = np.setdiff1d(np.arange(NQ), bad)
    to = rows[0].long().cpu().numpy()[keep]
    assert_close(host_f64(full)[0, to], want[keep], f"scattered rows, D={D}")
    rest = torch.ones(NQ + NC, dtype=torch.bool)
    rest[to] = False
    assert bool((full[0, rest.cuda()] == -3.0).all())


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("rows", ["all", "one"])
def test_first_share_merges_rows_that_outgrow_their_reference(D, rows):
    """Keys of the second and third tile, of the middle and of the end raise the logits of every row, or of one row of the
    lone tile and one of a pair, by more than the probabilities' exponent range: segments are walked again, among them
    heads and tails of cut items."""
    import torch
    q, kf, vf, kc, vc, nq, nc, ws, status = _case(D)
    q, kf, kc = q * 0.3, kf * 0.3, kc * 0.3
    q[..., 0] = 16.0 if rows == "all" else 0.0
    q[:, [3, NQ - 1], :, 0] = 16.0
    kf[..., 0] = kc[..., 0] = 0.0
    for at, by in ((200, 40.0), (290, 80.0), (4000, 120.0), (7800, 160.0)):
        kc[:, at, :, 0] = by
    out = torch.zeros_like(q)
    assert _launched(lambda: binding.region_attention(q, kf, vf, kc, vc, nq, nq, nc, out, workspace=ws, dev_status=status)) == 1
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    assert_close(host_f64(out)[0], _want(q, torch.cat([kf, kc], 1), torch.cat([vf, vc], 1)), f"outgrown rows ({rows}), D={D}")


def _step(D, grid, n_text, heads, ratio, ne_cap, store=True, spread=False):
    """A step, the kernels it launched, and its attention rows against the equation."""
    import torch
    wl, lat, x, qkv = _inputs(1, grid, n_text, heads, D, ratio)
    if spread:                                   # some logits outgrow the first key tile's by far
        for a in qkv[:2]:
            a *= 0.3
            a[..., 0] = 0
        qkv[0][:, ::7, :, 0] = 16.0
        for at, by in ((200, 40.0), (1500, 80.0), (5000, 120.0)):
            qkv[1][:, at, :, 0] = by
    step = RegionStep(StepShapes(1, wl.n_img, n_text, wl.n_ref, wl.channels, heads, D, ne_cap, binding.METRIC_COSINE, wl.threshold))
    step.k_cache.copy_(qkv[1]); step.v_cache.copy_(qkv[2])
    if not store:                                # the cache of the step itself, left by an earlier call
        step.run(*x, *qkv, lat["t"], 0.97, 0.1, 0.2)
    step.o_full.zero_()
    n = _launched(lambda: step.run(*x, *qkv, lat["t"], 0.97, 0.1, 0.2, store_cache=store))
    torch.cuda.synchronize()
    assert int(step.dev_status[0]) == 0
    nq, nc = int(step.n_q[0]), int(step.n_cache[0])
    assert nq > 0 and nq + nc == step.shp.n_full
    rows, kept = step.query_rows[0, :nq].long(), step.cache_rows[0, :nc].long()
    assert_close(host_f64(step.o_full[0, rows]), _want(qkv[0][:, rows], qkv[1], qkv[2]), "attention rows")
    assert not bool(step.o_full[0, kept].any())
    for full, cache, fresh in ((qkv[1], step.k_cache, step.k_fresh), (qkv[2], step.v_cache, step.v_fresh)):
        assert torch.equal(cache[0, :nc], full[0, kept]) and torch.equal(fresh[0, :nq], full[0, rows])
    return n, step


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("spread", [False, True])
def test_first_share_merges_beside_the_copies_of_a_storing_step(D, spread):
    n, step = _step(D, (64, 64), 512, H, 0.2, 896, spread=spread)
    assert n == step.kernel_launches == 3        # partition, moves, attention


@pytest.mark.parametrize("n_text,store", [
    (224, True), (225, True),                    # n_full = 1024 | 1025: rows taken along up to 16 x (128 - 64)
    (128, False), (129, False),                  # n_full + 128 = 768 | 769: clusters up to 12 x (128 - 64)
])
@pytest.mark.parametrize("D", [64, 128])
def test_step_on_both_sides_of_its_rules(D, n_text, store):
    grid = (20, 20) if store else (16, 16)
    n, step = _step(D, grid, n_text, 4, 0.25, 128, store=store)
    assert step.shp.n_full == 2 * grid[0] * grid[1] + n_text
    assert n == (3 if n_text == 128 else 4)      # (the storing steps are far below the line of the clusters)
