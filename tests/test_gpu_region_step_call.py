"""The one-call region step against the separate library calls it stands for, bit for bit where the
operations are the same and within the attention's tolerance where the key order differs."""
import numpy as np
import pytest

from gpu_util import assert_close, dev_bf16, host_f64
from paper_2510_25590_b200 import binding, synth
from paper_2510_25590_b200.step import RegionStep, StepShapes

pytestmark = pytest.mark.gpu


def _inputs(B, grid, n_text, H, D, ratio, seed=0):
    wl = synth.scaled_workload(synth.WORKLOADS[5], grid=grid, n_text=n_text, heads=H, head_dim=D, batch=B)
    lat = synth.make_latents(wl, ratio, stream=seed)
    qkv = synth.make_qkv_full(wl, stream=seed)
    return wl, lat, [dev_bf16(lat[k]) for k in ("x_t", "v", "ref")], [dev_bf16(qkv[k]) for k in ("q", "k", "v")]


def _separate(step, lat, qkv, t, scale, dt, dt_u, store):
    s, b, st = step.shp, binding, step.dev_status
    x_t, v, ref = lat
    b.partition_rows(x_t, v, ref, t, s.metric, s.threshold, step.mask, step.edit_idx, step.keep_idx, step.slot, step.n_edit,
                     s.n_text, s.n_ref, s.membership, step.query_rows, step.n_q, step.cache_rows, step.n_cache, dev_status=st)
    b.gather_multi([x_t, v], step.edit_idx, step.n_edit, [step.x_e, step.v_e], dev_status=st)
    b.velocity_decay(step.v_e, scale, dt, step.x_e, step.n_edit, v_cache_out=step.v_avd, dev_status=st)
    b.merge(x_t, v, step.x_e, step.slot, dt_u, step.x_out, dev_status=st)
    if store:
        b.rikv_store(qkv[1], qkv[2], step.cache_rows, step.n_cache, step.k_cache, step.v_cache, dev_status=st)
    b.gather_multi(qkv, step.query_rows, step.n_q, [step.q_e, step.k_fresh, step.v_fresh], dev_status=st)
    b.region_attention_scatter(step.q_e, step.k_fresh, step.v_fresh, step.k_cache, step.v_cache, step.n_q, step.n_q,
                               step.n_cache, step.o_full, step.query_rows, workspace=step.workspace, dev_status=st)


@pytest.mark.parametrize("B,grid,n_text,H,D,ratio,ne_cap", [
    (1, (24, 24), 70, 4, 128, 0.2, 128),
    (3, (17, 23), 33, 5, 64, 0.4, 256),
    (2, (16, 16), 16, 2, 128, 1.0, 256),        # everything edited
    (2, (16, 16), 16, 2, 128, 0.0, 128),        # nothing edited: no query, the cache is still refreshed
    (2, (24, 24), 20, 3, 128, 0.5, 128),        # more edited tokens than the capacity holds
])
@pytest.mark.parametrize("membership", [binding.ROWS_EDITED_QUERIES, binding.ROWS_PAPER])
@pytest.mark.parametrize("store", [True, False])
def test_one_call_leaves_what_the_separate_calls_leave(B, grid, n_text, H, D, ratio, ne_cap, membership, store):
    import torch
    wl, lat, x, qkv = _inputs(B, grid, n_text, H, D, ratio)
    shp = StepShapes(B, wl.n_img, n_text, wl.n_ref, wl.channels, H, D, ne_cap, binding.METRIC_COSINE, wl.threshold, membership)
    one, sep = RegionStep(shp), RegionStep(shp)
    t, scale, dt, dt_u = [lat["t"]] * B, [0.97] * B, [1 / 28.0] * B, [5 / 28.0] * B
    if not store:                                # the cache of an earlier step
        for s in (one, sep):
            s.k_cache.copy_(qkv[2]); s.v_cache.copy_(qkv[1])
    one.run(*x, *qkv, t, scale, dt, dt_u, store_cache=store)
    _separate(sep, x, qkv, t, scale, dt, dt_u, store)
    torch.cuda.synchronize()
    over = int(lat["mask"].sum(1).max()) > ne_cap
    want = binding.DEV_BOUNDS if over else 0
    assert int(one.dev_status[0]) == want and int(sep.dev_status[0]) == want
    for name in ("mask", "slot", "n_edit", "n_q", "n_cache", "query_rows", "cache_rows", "x_e", "v_e", "v_avd", "x_out",
                 "k_cache", "v_cache", "q_e"):
        assert torch.equal(getattr(one, name), getattr(sep, name)), name
    if store and over:
        return                                   # (the rows that do not fit are neither fresh nor cached there)
    a, b = host_f64(one.o_full), host_f64(sep.o_full)
    if not store:
        assert np.array_equal(a, b)
    assert_close(a, b, "attention rows")


def test_requests_that_sit_out_and_requests_in_a_batch_of_three():
    """NaN scalars: a request keeps its partition, its Euler step or its merge from before."""
    import torch
    B = 3
    wl, lat, x, qkv = _inputs(B, (16, 20), 24, 2, 64, 0.3)
    shp = StepShapes(B, wl.n_img, 24, wl.n_ref, wl.channels, 2, 64, 128, binding.METRIC_COSINE, wl.threshold)
    one, sep = RegionStep(shp), RegionStep(shp)
    nan = float("nan")
    for t, scale, dt, dt_u in (([lat["t"]] * B, 0.9, 0.1, 0.2), ([lat["t"], nan, nan], [nan, 0.5, 0.25], 0.125, [0.5, nan, 0.25])):
        one.run(*x, *qkv, t, scale, dt, dt_u)
        _separate(sep, x, qkv, t, scale, dt, dt_u, True)
        torch.cuda.synchronize()
        assert int(one.dev_status[0]) == 0
        for name in ("mask", "slot", "n_edit", "x_e", "v_e", "v_avd", "x_out", "k_cache", "v_cache"):
            assert torch.equal(getattr(one, name), getattr(sep, name)), name
        assert_close(host_f64(one.o_full), host_f64(sep.o_full), "attention rows")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,grid,n_text,ne_cap", [
    (3, (24, 24), 20, 256),      # few items: shared by clusters
    (24, (30, 30), 30, 512),     # shares of the cost axis
])
@pytest.mark.parametrize("membership", [binding.ROWS_EDITED_QUERIES, binding.ROWS_PAPER])
def test_storing_step_with_more_edited_tokens_than_the_capacity_holds(D, H, grid, n_text, ne_cap, membership):
    """A request whose edited tokens do not fit attends over the rows of its lists alone (the dropped tokens' keys are
    neither fresh nor cached), beside one that fits and attends over K and V in place."""
    import torch
    wl, lat, x, qkv = _inputs(2, grid, n_text, H, D, 0.9)
    x[0][1, 200:] = x[2][1, 200:]                # request 1: the tokens from 200 on equal their reference, v = 0
    x[1][1, 200:] = 0
    shp = StepShapes(2, wl.n_img, n_text, wl.n_ref, wl.channels, H, D, ne_cap, binding.METRIC_COSINE, wl.threshold, membership)
    assert 16 * (shp.q_cap - 64) >= shp.n_full   # the attention reads K and V in place
    one, sep = RegionStep(shp), RegionStep(shp)
    one.run(*x, *qkv, lat["t"], 0.97, 0.1, 0.2)
    _separate(sep, x, qkv, lat["t"], 0.97, 0.1, 0.2, True)
    torch.cuda.synchronize()
    assert int(one.n_edit[0]) > ne_cap >= int(one.n_edit[1]) > 0
    assert int(one.dev_status[0]) == int(sep.dev_status[0]) == binding.DEV_BOUNDS
    for name in ("n_q", "n_cache", "query_rows", "cache_rows", "k_cache", "v_cache", "q_e", "x_out", "k_fresh",
                 "v_fresh"):
        assert torch.equal(getattr(one, name), getattr(sep, name)), name
    for b in range(2):
        assert_close(host_f64(one.o_full[b]), host_f64(sep.o_full[b]), f"attention rows, request {b}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,grid,n_text,ratio", [(2, (24, 24), 20, 0.3), (24, (30, 30), 30, 0.5), (70, (16, 16), 16, 1.0)])
@pytest.mark.parametrize("membership", [binding.ROWS_EDITED_QUERIES, binding.ROWS_PAPER])
def test_storing_step_leaves_its_fresh_rows_too(D, H, grid, n_text, ratio, membership):
    """k_fresh and v_fresh after a step whose attention reads K and V in place: rows of this step, those behind the
    live ones as they were.  Row lengths below and above what one copy moves."""
    import torch
    wl, lat, x, qkv = _inputs(2, grid, n_text, H, D, ratio)
    shp = StepShapes(2, wl.n_img, n_text, wl.n_ref, wl.channels, H, D, wl.n_img, binding.METRIC_COSINE, wl.threshold, membership)
    assert 16 * (shp.q_cap - 64) >= shp.n_full
    one, sep = RegionStep(shp), RegionStep(shp)
    for s in (one, sep):
        s.k_fresh.fill_(-3.0); s.v_fresh.fill_(-3.0)
    one.run(*x, *qkv, lat["t"], 0.97, 0.1, 0.2)
    _separate(sep, x, qkv, lat["t"], 0.97, 0.1, 0.2, True)
    torch.cuda.synchronize()
    assert int(one.dev_status[0]) == 0
    for name in ("k_fresh", "v_fresh", "k_cache", "v_cache", "q_e"):
        assert torch.equal(getattr(one, name), getattr(sep, name)), name
