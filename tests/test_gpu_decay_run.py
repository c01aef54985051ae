"""Several Euler updates with one velocity in one launch against the same updates call by call, bit for bit,
and the sampler loop that uses them against the loop that a hook makes go step by step."""
import numpy as np
import pytest

from gpu_util import dev_bf16
from paper_2510_25590_b200 import binding, loop as gloop
from test_gpu_loop import TorchStraightLine, _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_steps,keep", [(1, 1, True), (3, 5, False), (9, 16, True), (2, 128, True)])
def test_one_call_leaves_what_the_calls_leave(B, n_steps, keep):
    """9 requests of 16 steps are one more than a launch carries scalars for; 128 steps are one request each."""
    import torch
    rng = np.random.default_rng(n_steps)
    cap, C = 37, 24
    v, x0 = (dev_bf16(rng.standard_normal((B, cap, C)).astype(np.float32)) for _ in range(2))
    n = torch.tensor([cap - b for b in range(B)], dtype=torch.int32, device="cuda")
    scale, dt = rng.uniform(0.8, 1.2, (n_steps, B)), rng.uniform(0.01, 0.1, (n_steps, B))
    if B > 1:
        dt[:, 1] = np.nan                                    # sits the call out
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want, got, v_kept, v_got = x0.clone(), x0.clone(), torch.zeros_like(v), torch.zeros_like(v)
    for k in range(n_steps):
        binding.velocity_decay(v, scale[k].tolist(), dt[k].tolist(), want, n, v_cache_out=v_kept if keep else None,
                               dev_status=status)
    host = lambda a: binding._per_request(a.reshape(-1).tolist(), a.size, "scalars")
    assert binding.load().regione_velocity_decay_run(
        v.data_ptr(), host(scale), host(dt), n_steps, got.data_ptr(), v_got.data_ptr() if keep else None, n.data_ptr(), B,
        cap, C, status.data_ptr(), binding._stream()) == binding.OK
    assert torch.equal(want, got) and torch.equal(v_kept, v_got) and int(status[0]) == 0


@pytest.mark.parametrize("schedule", ["alternating", "paper"])
def test_loop_is_the_loop_that_goes_step_by_step(schedule):
    import torch
    _, ref, _, target, noise = _case()
    kinds, after = gloop.alternating_schedule() if schedule == "alternating" else gloop.paper_schedule()
    T = len(kinds)
    cfg = gloop.LoopConfig(kinds, after, [1.0 - k / T for k in range(T + 1)], [1.0] * (T + 1), 0.05,
                           binding.METRIC_COSINE, 0.9)
    done = []
    for hook in (None, lambda *a: None):
        lp = gloop.RegionELoop(*noise.shape, cfg)
        lp.hook = hook
        x, trace = lp.run(dev_bf16(noise), dev_bf16(ref), TorchStraightLine(dev_bf16(target)))
        done.append((x, lp.x_e, lp.v_cache, trace))
    for a, b in zip(done[0][:3], done[1][:3]):
        assert torch.equal(a, b)
    a, b = done[0][3], done[1][3]
    assert a.per_request == b.per_request and a.model_region_calls == b.model_region_calls
    assert a.launches < b.launches


def test_long_runs_of_reused_steps_are_split():
    """20 reused steps behind one computed step: more than one update carries."""
    import torch
    _, ref, _, target, noise = _case()
    T = 24
    cfg = gloop.LoopConfig("FF" + "R" * 21 + "F", 2, [1.0 - k / (4 * T) for k in range(T + 1)], [1.0] * (T + 1), 100.0,
                           binding.METRIC_COSINE, 0.9)
    done = []
    for hook in (None, lambda *a: None):
        lp = gloop.RegionELoop(*noise.shape, cfg)
        lp.hook = hook
        x, trace = lp.run(dev_bf16(noise), dev_bf16(ref), TorchStraightLine(dev_bf16(target)))
        done.append((x, trace.per_request))
        assert trace.model_region_calls == 1
    assert torch.equal(done[0][0], done[1][0]) and done[0][1] == done[1][1]
