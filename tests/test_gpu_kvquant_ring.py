"""The 8-bit cache store at the sizes where its two forms can go wrong: the ring (rows of several pieces, pieces that do not fill
a warp's last pass, rings that wrap and batches of pieces that follow one another), the block per row (passes that are full,
partly full or repeated), both sides of the rule between them, counts and rows out of range."""
import numpy as np
import pytest

from gpu_util import dev_bf16, dev_i32
from oracle import regione_oracle as orc
from paper_2510_25590_b200 import binding, synth

pytestmark = pytest.mark.gpu
REST = 0x55                                          # what the destination holds before the call


def _store(k, v, keep, n_keep):
    import torch
    (B, _, H, D), cap = k.shape, keep.shape[1]
    codes = [torch.full((B, cap, H, D), REST, dtype=torch.uint8, device="cuda") for _ in range(2)]
    scales = [torch.full((B, cap, H), -7.0, dtype=torch.float32, device="cuda") for _ in range(2)]
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.rikv_store_e4m3(k, v, dev_i32(keep), dev_i32(n_keep), *codes, *scales, dev_status=st)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in codes + scales], int(st[0])


@pytest.mark.parametrize("D,H,N,cap,n_keep", [
    (128, 1, 31000, 30000, [30000, 29999]),          # more than one batch of pieces a warp
    (64, 3, 9000, 8000, [8000, 1]),
    (128, 33, 400, 300, [300, 0]),                   # (few rows: a block per row, two passes, the second one short)
    (64, 130, 200, 150, [3, 150]),
    (128, 33, 1500, 1300, [1300, 30]),               # two pieces of 17 and 16 heads
    (64, 73, 1500, 1300, [3, 1300]),                 # three pieces, the last one shorter
    (128, 2, 1300, 1184, [1184, 1184]),              # 2368 rows: a block per row | rings
    (128, 2, 1300, 1185, [1185, 1185]),
    (64, 48, 1400, 1200, [1200, 1]),                 # full passes: a block per row
    (128, 20, 1400, 1200, [1199, 1200]),             # passes filled to five sixths | to less than four fifths
    (128, 19, 1400, 1200, [1199, 1200]),
    (64, 47, 9100, 9000, [9000, 200]),               # one pass, nearly full, 18000 rows: rings
])
def test_codes_and_scales(D, H, N, cap, n_keep):
    rng = np.random.default_rng(D + H)
    k, v = (synth.bf16_round(rng.standard_normal((2, N, H, D), dtype=np.float32) * np.float32(s)) for s in (0.09, 3.0))
    keep = np.stack([rng.permutation(N)[:cap] for _ in range(2)]).astype(np.int32)
    (kq, vq, ks, vs), status = _store(dev_bf16(k), dev_bf16(v), keep, np.array(n_keep, np.int32))
    assert status == 0
    for b, n in enumerate(n_keep):
        for got, scale, x in ((kq, ks, k), (vq, vs, v)):
            rows = x[b, keep[b, :n]].astype(np.float64)
            m, e = np.frexp(np.abs(rows).max(-1))
            want = np.ldexp(1.0, e - 9 + (m > 0.875))
            assert np.array_equal(scale[b, :n].astype(np.float64), want) and np.all(scale[b, n:] == -7.0)
            codes = orc.e4m3_encode(rows / want[..., None])
            zero = (codes & 0x7f) == 0                                       # (+0 and -0 are the same value)
            assert np.array_equal(np.where(zero, 0, got[b, :n]), np.where(zero, 0, codes))
            assert np.all((got[b, :n][zero] & 0x7f) == 0) and np.all(got[b, n:] == REST)


@pytest.mark.parametrize("cap", [6, 2400])           # a block per row, rings
def test_special_values_and_bounds(cap):
    import torch
    x = torch.ones((1, 8, 2, 128), dtype=torch.bfloat16, device="cuda")
    x[0, 1, 0, 5], x[0, 1, 1, 127] = float("inf"), float("nan")
    x[0, 2, 0], x[0, 2, 1] = 2.0 ** -130, 1.75                               # subnormal; the edge of the scale rule
    x[0, 3, 0], x[0, 3, 1] = -3.3e38, -1.7578125
    rest = [4] * (cap - 6)
    (kq, vq, ks, vs), status = _store(x, x, np.array([[1, 2, 3, 8, -1, 4] + rest], np.int32), np.array([6], np.int32))
    assert status == binding.DEV_BOUNDS
    for q, s in ((kq, ks), (vq, vs)):
        assert np.array_equal(np.log2(s[0, :3]), [[120, -8], [-100, -8], [120, -7]])
        assert q[0, 0, 0, 5] == 0x7e and np.all(q[0, 0, 0, :5] == 0) and q[0, 0, 1, 127] & 0x7f == 0x7f
        assert np.all(q[0, 1, 0] == 0) and np.all(q[0, 1, 1] == 0x7e) and np.all(q[0, 0, 1, :127] == 0x78)
        assert np.all(q[0, 3:5] == REST) and np.all(q[0, 5] == 0x78)          # rows out of range are left out
    (kq, *_), status = _store(x, x, np.zeros((1, cap), np.int32), np.array([cap + 1], np.int32))
    assert status == binding.DEV_BOUNDS and np.all(kq == 0x78)               # a count beyond the capacity is clamped
