"""The one-call region step names its buffers by address: buffers that are replaced, re-pointed or of other shapes than
planned, sizes changed in place, and inputs of other shapes give what the separate library calls give, or are refused."""
import pytest

from gpu_util import assert_close, host_f64
from paper_2510_25590_b200 import binding
from paper_2510_25590_b200.step import RegionStep, StepShapes
from test_gpu_region_step_call import _inputs, _separate

pytestmark = pytest.mark.gpu

SCALARS = (0.97, 0.1, 0.2)


def _steps(B=2, membership=binding.ROWS_EDITED_QUERIES, n=2):
    wl, lat, x, qkv = _inputs(B, (20, 20), 30, 3, 64, 0.4)
    shp = lambda: StepShapes(B, wl.n_img, 30, wl.n_ref, wl.channels, 3, 64, 256, binding.METRIC_COSINE, wl.threshold, membership)
    return x, qkv, lat["t"], [RegionStep(shp()) for _ in range(n)]


def _same(one, sep, rows=slice(None)):
    import torch
    torch.cuda.synchronize()
    assert int(one.dev_status[0]) == int(sep.dev_status[0]) == 0
    for name in ("query_rows", "n_q", "n_cache", "x_e", "v_avd", "x_out", "q_e"):
        assert torch.equal(getattr(one, name), getattr(sep, name)), name
    assert_close(host_f64(one.o_full[:, rows]), host_f64(sep.o_full[:, rows]), "attention rows")


def test_replaced_and_repointed_buffers_receive_the_results():
    import torch
    x, qkv, t, (one, sep) = _steps()
    one.run(*x, *qkv, t, *SCALARS)
    old = one.x_out, one.k_cache, one.o_full.clone()
    one.k_cache = torch.zeros_like(one.k_cache)
    one.run(*x, *qkv, t, *SCALARS)
    held = one.x_out.data
    one.x_out.data = torch.zeros_like(one.x_out)         # another address behind the same object
    held.fill_(-5.0)
    old[1].fill_(-5.0)
    one.run(*x, *qkv, t, *SCALARS)
    _separate(sep, x, qkv, t, *SCALARS, True)
    _same(one, sep)
    assert torch.equal(one.k_cache, sep.k_cache)
    assert bool((held == -5.0).all()) and bool((old[1] == -5.0).all())


def test_buffers_with_another_number_of_rows():
    import torch
    x, qkv, t, (one, sep) = _steps()
    n = one.shp.n_full
    one.o_full = torch.zeros((2, n + 40, 3, 64), dtype=torch.bfloat16, device="cuda")
    one.run(*x, *qkv, t, *SCALARS)
    _separate(sep, x, qkv, t, *SCALARS, True)
    _same(one, sep, slice(0, n))
    assert not bool(one.o_full[:, n:].any())

    x, qkv, t, (one, sep) = _steps(B=1)                  # a cache of exactly the rows that it receives
    _separate(sep, x, qkv, t, *SCALARS, True)
    nc = int(sep.n_cache[0])
    guard = torch.full((nc + 8, 3, 64), -5.0, dtype=torch.bfloat16, device="cuda")
    one.k_cache, one.v_cache = guard[:nc][None], torch.zeros_like(guard[:nc][None])
    one.run(*x, *qkv, t, *SCALARS)
    _same(one, sep)
    assert torch.equal(one.k_cache[0], sep.k_cache[0, :nc]) and bool((guard[nc:] == -5.0).all())


def test_unfit_buffers_and_inputs_are_refused():
    import torch
    x, qkv, t, (one,) = _steps(n=1)
    whole = one.k_cache
    one.k_cache = torch.zeros((2, whole.shape[1], 3, 128), dtype=torch.bfloat16, device="cuda")[..., :64]
    with pytest.raises(binding.RegionEError):            # strided
        one.run(*x, *qkv, t, *SCALARS)
    one.k_cache = whole[:, :100].contiguous()            # fewer rows than the list of them is laid out for
    with pytest.raises(binding.RegionEError):
        one.run(*x, *qkv, t, *SCALARS)
    one.k_cache = whole.half()
    with pytest.raises(binding.RegionEError):
        one.run(*x, *qkv, t, *SCALARS)
    one.k_cache, v_avd = whole, one.v_avd
    one.v_avd = v_avd[:, :100].contiguous()
    with pytest.raises(binding.RegionEError):
        one.run(*x, *qkv, t, *SCALARS)
    one.v_avd = v_avd
    with pytest.raises(binding.RegionEError):            # more tokens than the buffers hold
        one.run(*(torch.cat([a, a], 1) for a in x), *qkv, t, *SCALARS)
    with pytest.raises(binding.RegionEError):            # longer rows than the buffers hold
        one.run(*x, *(torch.cat([a, a], 2) for a in qkv), t, *SCALARS)
    one.run(*x, *qkv, t, *SCALARS)
    torch.cuda.synchronize()
    assert int(one.dev_status[0]) == 0


def test_sizes_changed_in_place_count_at_the_next_run():
    x, qkv, t, (one, sep) = _steps(membership=binding.ROWS_PAPER)
    one.run(*x, *qkv, t, *SCALARS)
    one.shp.membership = sep.shp.membership = binding.ROWS_EDITED_QUERIES
    for s in (one, sep):
        s.query_rows.zero_(); s.q_e.zero_(); s.o_full.zero_()
    one.run(*x, *qkv, t, *SCALARS)
    _separate(sep, x, qkv, t, *SCALARS, True)
    _same(one, sep)


def test_inputs_with_rows_as_one_dimension_or_more_rows():
    import torch
    x, qkv, t, (one, sep) = _steps()
    for s in (one, sep):                                 # the cache of an earlier step
        s.k_cache.copy_(qkv[2]); s.v_cache.copy_(qkv[1])
    flat = [torch.cat([a.flatten(2), a.flatten(2)[:, :9]], 1) for a in qkv]
    one.run(x[0], x[1], x[2].flatten(1), *flat, t, *SCALARS, store_cache=False)
    _separate(sep, x, qkv, t, *SCALARS, False)
    _same(one, sep)
