"""What the sampler loop takes from its velocity model: velocities of other shapes that hold the same rows, and streams
that the model makes current."""
import pytest

from gpu_util import dev_bf16
from paper_2510_25590_b200 import binding, loop as gloop
from test_gpu_loop import TorchStraightLine, _case

pytestmark = pytest.mark.gpu


class _Shaped(TorchStraightLine):
    def __init__(self, target, full=lambda v: v, region=lambda v: v):
        super().__init__(target)
        self.shape_full, self.shape_region = full, region

    def full(self, x, t, store):
        return self.shape_full(super().full(x, t, store))

    def region(self, x_e, t, edit_idx, n_edit):
        return self.shape_region(super().region(x_e, t, edit_idx, n_edit))


def _loop(noise):
    kinds, after = gloop.alternating_schedule()
    T = len(kinds)
    cfg = gloop.LoopConfig(kinds, after, [1.0 - k / T for k in range(T + 1)], [1.0] * (T + 1), 0.05, binding.METRIC_COSINE, 0.9)
    return gloop.RegionELoop(*noise.shape, cfg)


@pytest.mark.parametrize("hooked", [False, True])
def test_velocities_of_other_shapes_with_the_same_rows(hooked):
    import torch
    def run(B, **shapes):
        _, ref, _, target, noise = _case(B=B)
        lp = _loop(noise)
        lp.hook = (lambda *a: None) if hooked else None
        x, _ = lp.run(dev_bf16(noise), dev_bf16(ref), _Shaped(dev_bf16(target), **shapes))
        torch.cuda.synchronize()
        assert int(lp.dev_status[0]) == 0
        return x, int(lp.n_edit.max())
    want, n = run(1)
    # one request: without its dimension; only the rows of the edited tokens; more rows than tokens
    for region in (lambda v: v[:, :n].contiguous(), lambda v: v[0, :n + 3].contiguous(), lambda v: torch.cat([v, v], 1)):
        assert torch.equal(run(1, full=lambda v: v[0], region=region)[0], want)
    want, _ = run(2)
    assert torch.equal(run(2, region=lambda v: v.flatten(0, 1))[0], want)
    for shapes in (dict(full=lambda v: v[:1]), dict(full=lambda v: v[0]), dict(region=lambda v: v[:, :n].contiguous()),
                   dict(full=lambda v: v.float()), dict(region=lambda v: v.transpose(0, 1))):
        with pytest.raises(binding.RegionEError):
            run(2, **shapes)


@pytest.mark.parametrize("hooked", [False, True])
def test_a_region_velocity_with_too_few_rows_is_reported(hooked):
    """A single request's velocity of fewer rows than it has edited tokens: its rows are applied, none is read behind them."""
    import torch
    _, ref, _, target, noise = _case(B=1)
    before = []
    class Model(_Shaped):
        def region(self, x_e, t, edit_idx, n_edit):
            before.append(x_e[0].clone())
            return super().region(x_e, t, edit_idx, n_edit)
    lp = _loop(noise)
    lp.hook = (lambda *a: None) if hooked else None
    lp.run(dev_bf16(noise), dev_bf16(ref), Model(dev_bf16(target), region=lambda v: v[:, :5].contiguous()))
    torch.cuda.synchronize()
    n = int(lp.n_edit[0])
    assert n > 5 and int(lp.dev_status[0]) == binding.DEV_BOUNDS
    assert torch.equal(lp.x_e[0, 5:n], before[-1][5:n]) and not torch.equal(lp.x_e[0, :5], before[-1][:5])
    assert not lp.v_cache[0, 5:].any()


@pytest.mark.parametrize("hooked", [False, True])
def test_loop_follows_the_stream_that_the_model_makes_current(hooked):
    """A model that leaves another stream current, its velocity still being computed there when it returns."""
    import torch
    class Elsewhere(TorchStraightLine):
        def switch(self):
            old, new = torch.cuda.current_stream(), torch.cuda.Stream()
            new.wait_stream(old)
            torch.cuda.set_stream(new)
            torch.cuda._sleep(200_000)
        def full(self, x, t, store):
            self.switch()
            return super().full(x, t, store)
        def region(self, x_e, t, edit_idx, n_edit):
            self.switch()
            return super().region(x_e, t, edit_idx, n_edit)
    _, ref, _, target, noise = _case()
    first, done = torch.cuda.current_stream(), []
    for model in (TorchStraightLine, Elsewhere):
        lp = _loop(noise)
        lp.hook = (lambda *a: None) if hooked else None
        try:
            done.append(lp.run(dev_bf16(noise), dev_bf16(ref), model(dev_bf16(target)))[0])
            torch.cuda.synchronize()
        finally:
            torch.cuda.set_stream(first)
        done.append(lp.x_e)
    assert torch.equal(done[0], done[2]) and torch.equal(done[1], done[3])


@pytest.mark.parametrize("which", ["region velocity in x", "full velocity in x_e"])
def test_velocities_that_lie_in_the_loop_s_buffers(which):
    """A model whose velocity lies in rows that the loop writes next: read by every block before it is written over.
    (65536 tokens of 64 channels are twice the blocks that are resident at once.)"""
    import torch
    N, C = 65536, 64
    g = torch.Generator(device="cuda").manual_seed(11)
    r = lambda: torch.randn((1, N, C), generator=g, device="cuda").bfloat16()
    ref, noise, target = r(), r(), r()
    edited = torch.rand((1, N, 1), generator=g, device="cuda") < 0.4
    target = torch.where(edited, target, ref)

    class Model(TorchStraightLine):
        def full(self, x, t, store):
            self.x = x
            v = super().full(x, t, store)
            return lp.x_e.copy_(v) if which == "full velocity in x_e" else v

        def region(self, x_e, t, edit_idx, n_edit):
            return self.x if which == "region velocity in x" else super().region(x_e, t, edit_idx, n_edit)

    done = []
    for hook in (lambda *a: None, None):                     # a call for each of the loop's operations; the short path
        lp = _loop(noise)
        lp.hook = hook
        x, _ = lp.run(noise.clone(), ref, Model(target))
        torch.cuda.synchronize()
        assert int(lp.dev_status[0]) == 0 and 0 < int(lp.n_edit[0]) < N
        done.append((x, lp.x_e))
    assert all(torch.equal(a, b) for a, b in zip(*done))
