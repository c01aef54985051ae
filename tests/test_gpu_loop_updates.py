"""The sampler loop's updates of all tokens in one launch against the calls that they stand for, bit for bit."""
import numpy as np
import pytest

from gpu_util import dev_bf16
from paper_2510_25590_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,C,n_steps", [(1, 1, 8, 1), (1, 300, 16, 5), (3, 37, 24, 1), (9, 65, 16, 16), (130, 5, 8, 2)])
@pytest.mark.parametrize("new_velocity", [True, False])
def test_updates_leave_what_the_calls_leave(B, N, C, n_steps, new_velocity):
    """9 requests of 16 steps, or 130 requests, are more than a launch carries scalars for."""
    import torch
    rng = np.random.default_rng(B + N)
    r = lambda: dev_bf16(rng.standard_normal((B, N, C)).astype(np.float32))
    mask = rng.random((B, N)) < 0.4
    n = mask.sum(1)
    slot = np.where(mask, np.cumsum(mask, 1) - 1, -1)
    idx = np.zeros((B, N), np.int64)
    for b in range(B):
        idx[b, :n[b]] = np.flatnonzero(mask[b])
    slot, idx, n = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in (slot, idx, n))
    n_all = torch.full_like(n, N)
    dt, dt_e, scale, dt_u = rng.uniform(0.01, 0.1, B), rng.uniform(0.01, 0.1, (n_steps, B)), rng.uniform(0.8, 1.2, (n_steps, B)), \
        rng.uniform(0.1, 0.4, B)
    if B > 2:
        dt[1] = dt_e[0, 1] = dt_u[2] = np.nan                # sit the call, the update or the merge out
    x, x_e, v_last, v_cache, v, v_e = (r() for _ in range(6))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = [t.clone() for t in (x, x_e, v_last, v_cache)]
    got = [t.clone() for t in (x, x_e, v_last, v_cache)]
    lib, s = binding.load(), binding._stream()
    host = lambda a: binding._per_request(np.asarray(a).reshape(-1).tolist(), np.size(a), "scalars")
    plan = binding.LoopPlan(B, N, C, *(t.data_ptr() for t in (*got, slot, n, status)))

    binding.velocity_decay(v, [1.0] * B, dt.tolist(), want[0], n_all, v_cache_out=want[2], dev_status=status)
    starts = n.clone()
    if B > 2:
        starts[1] = 0                                        # (a request that sits out starts no run either)
    binding.gather(want[0], idx, starts, want[1], dev_status=status)
    assert lib.regione_loop_full_step(plan, v.data_ptr(), host(dt), 1, s) == binding.OK
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    if B > 2:
        assert torch.equal(got[1][1], x_e[1]) and not torch.equal(got[1][2], x_e[2])
    assert lib.regione_loop_full_step(plan, v_e.data_ptr(), host(dt), 0, s) == binding.OK
    binding.velocity_decay(v_e, [1.0] * B, dt.tolist(), want[0], n_all, v_cache_out=want[2], dev_status=status)
    for a, b in zip(want, got):
        assert torch.equal(a, b)

    for k in range(n_steps):
        binding.velocity_decay(v_e if new_velocity else want[3].clone(), scale[k].tolist(), dt_e[k].tolist(), want[1], n,
                               v_cache_out=want[3] if new_velocity and k == 0 else None, dev_status=status)
        if B > 2 and k == 0:
            dt_e[1:, 1] = np.nan                             # (a request whose first step is NaN sits all of them out)
    binding.merge(want[0], want[2], want[1], slot, dt_u.tolist(), want[0], dev_status=status)
    assert lib.regione_loop_region_steps(plan, v_e.data_ptr() if new_velocity else None, host(scale), host(dt_e), n_steps,
                                         host(dt_u), s) == binding.OK
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    assert int(status[0]) == 0


def test_updates_report_what_they_do_not_follow():
    import torch
    B, N, C = 1, 40, 16
    z = [torch.zeros((B, N, C), dtype=torch.bfloat16, device="cuda") for _ in range(6)]
    slot, n = torch.full((B, N), -1, dtype=torch.int32, device="cuda"), torch.full((B,), 3, dtype=torch.int32, device="cuda")
    slot[0, 7] = N
    lib, s, one = binding.load(), binding._stream(), binding._per_request(0.5, 1, "dt")
    for call in (lambda p: lib.regione_loop_full_step(p, z[4].data_ptr(), one, 1, s),
                 lambda p: lib.regione_loop_region_steps(p, z[5].data_ptr(), one, one, 1, one, s)):
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        plan = binding.LoopPlan(B, N, C, *(t.data_ptr() for t in (*z[:4], slot, n, status)))
        assert call(plan) == binding.OK
        torch.cuda.synchronize()
        assert int(status[0]) == binding.DEV_BOUNDS
        plan.C = 12
        assert call(plan) == binding.UNSUPPORTED
        plan.x = None
        assert call(plan) == binding.INVALID_ARG
