"""GPU parity of the attention where its walk over the key tiles changes course: rows whose logits outgrow
the reference maximum of the first key tile (the segment is walked again), and key tiles whose second
half has no live key, in the middle of the walk and at its end."""
import numpy as np
import pytest

from gpu_util import dev_bf16, dev_i32, host_f64
from oracle import regione_oracle as orc
from paper_2510_25590_b200 import binding
from test_gpu_attention import _rand_bf16, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("n_q,n_f,n_c", [
    (300, 300, 1000),      # a full query pair and a lone tile, items cut between thread blocks
    (100, 100, 300),       # a lone tile
    (256, 0, 128 * 3),     # whole tiles only
])
@pytest.mark.parametrize("rows", ["all", "one"])
@pytest.mark.parametrize("H", [3, 40])     # items shared by clusters; items cut between the shares of the cost axis
def test_logits_that_outgrow_the_first_key_tile(D, n_q, n_f, n_c, rows, H):
    """Later keys raise the logits of every row, or of one row, by far more than the exponent range of the
    probabilities: the softmax is then almost one-hot on those keys and the tolerance is that of the plain case."""
    rng = np.random.default_rng(D + n_q)
    B = 2
    q = _rand_bf16(rng, (B, n_q, H, D), 0.3)
    kf, vf = _rand_bf16(rng, (B, max(n_f, 1), H, D), 0.3), _rand_bf16(rng, (B, max(n_f, 1), H, D))
    kc, vc = _rand_bf16(rng, (B, n_c, H, D), 0.3), _rand_bf16(rng, (B, n_c, H, D))
    # dimension 0 of q is 16 (or 0 for rows that stay ordinary); key 200 (second tile) gives +16 * 40 / sqrt(D),
    # key 290 (third tile) twice that
    q[..., 0] = 16.0 if rows == "all" else 0.0
    if rows == "one":
        q[:, n_q - 1, :, 0] = 16.0
    kc[..., 0] = 0.0
    kf[..., 0] = 0.0
    kc[:, 200, :, 0] = 40.0
    kc[:, 290, :, 0] = 80.0
    check(q, kf, vf, kc, vc, [n_q] * B, [n_f] * B, [n_c] * B, what=f"outgrown rows ({rows}), D={D}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("n_q", [100, 256, 700])
@pytest.mark.parametrize("n_f,n_c", [(60, 1000 + 24), (64, 128 * 7 + 1), (65, 128 * 7 + 64), (1, 128 * 4 + 56)])
@pytest.mark.parametrize("H", [12, 38])
def test_key_tiles_with_a_dead_second_half(D, n_q, n_f, n_c, H):
    rng = np.random.default_rng(n_q + n_f + n_c + D)
    B = 2
    q = _rand_bf16(rng, (B, n_q, H, D))
    kf, vf = _rand_bf16(rng, (B, n_f + 5, H, D)), _rand_bf16(rng, (B, n_f + 5, H, D))
    kc, vc = _rand_bf16(rng, (B, n_c + 9, H, D)), _rand_bf16(rng, (B, n_c + 9, H, D))
    check(q, kf, vf, kc, vc, [n_q] * B, [n_f] * B, [n_c] * B, what=f"dead second half, D={D}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H", [1, 24, 70])
def test_cache_refresh_row_lengths_and_outgrown_rows(D, H):
    """The refreshing call with rows shorter and longer than a copy slot, its attention walked twice over."""
    import torch
    rng = np.random.default_rng(D + H)
    B, N = 2, 300
    q, k, v = (_rand_bf16(rng, (B, N, H, D), 0.3) for _ in range(3))
    q[..., 0] = 16.0
    k[..., 0] = 0.0
    k[:, 200, :, 0] = 40.0
    n_rows = [300, 211]
    keep = np.zeros((B, N), np.int32)
    for b, n in enumerate((251, 40)):
        keep[b, :n] = np.sort(rng.permutation(n_rows[b])[:n])
    out = torch.full((B, N, H, D), -3.0, dtype=torch.bfloat16, device="cuda")
    kc, vc = torch.full_like(out, -3.0), torch.full_like(out, -3.0)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(binding.full_attention_store_workspace(B, N, H, D), 256), dtype=torch.uint8, device="cuda")
    binding.full_attention_store(dev_bf16(q), dev_bf16(k), dev_bf16(v), dev_i32(n_rows), dev_i32(keep),
                                 dev_i32([251, 40]), kc, vc, out, workspace=ws, dev_status=st)
    torch.cuda.synchronize()
    assert int(st[0]) == 0
    for b, n in enumerate((251, 40)):
        assert np.array_equal(host_f64(kc)[b, :n], k[b, keep[b, :n]].astype(np.float64))
        assert np.array_equal(host_f64(vc)[b, :n], v[b, keep[b, :n]].astype(np.float64))
        assert np.all(host_f64(kc)[b, n:] == -3.0) and np.all(host_f64(vc)[b, n:] == -3.0)
    empty = np.zeros((B, 0, H, D))
    want = orc.region_attention(q, k, v, empty, empty, n_rows, n_rows, [0, 0])
    from gpu_util import assert_close
    for b in range(B):
        assert_close(host_f64(out)[b, :n_rows[b]], want[b, :n_rows[b]], f"attention, request {b}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("counts", [
    [(1, 1, 0)],                                        # one key tile: nothing to share
    [(200, 100, 128 * 2 + 5), (0, 3, 40), (130, 0, 128)],   # fewer key tiles than ranks, an empty request
    [(256, 256, 3000)],                                 # more key tiles than ranks
    [(40, 0, 0), (40, 10, 1000)],                       # a request without keys beside one with them
])
def test_items_shared_by_clusters(D, counts):
    """Capacities of few items: ranks without key tiles, rows of one and of two query tiles, dead items."""
    rng = np.random.default_rng(D + len(counts))
    B, H = len(counts), 4
    cap_q, cap_f, cap_c = (max(c[i] for c in counts) + 7 for i in range(3))
    q = _rand_bf16(rng, (B, cap_q, H, D))
    kf, vf = _rand_bf16(rng, (B, cap_f, H, D)), _rand_bf16(rng, (B, cap_f, H, D))
    kc, vc = _rand_bf16(rng, (B, cap_c, H, D)), _rand_bf16(rng, (B, cap_c, H, D))
    check(q, kf, vf, kc, vc, [c[0] for c in counts], [c[1] for c in counts], [c[2] for c in counts], what=f"clusters {counts}")


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,n_q,n_f,n_c", [(3, 300, 300, 2000), (40, 100, 0, 1500), (24, 819, 819, 7000)])
def test_rows_that_one_key_dominates_are_exact_to_the_rounding_of_the_output(D, H, n_q, n_f, n_c):
    """Each query meets one key, anywhere in the sequence, whose logit is 15 (the others' deviate by 1 / 4): its weight is
    above 0.99.  Whatever reference the probabilities are rounded against, that key's rounding cancels between the
    product and the sum, and what is left is the rounding of the output to bf16, which the exact result shows when it is
    rounded.  1.1 of that leaves room for the other keys; a rounding that does not cancel gives 1.17 to 2.3."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(D + H)
    r = lambda n: torch.randn((1, n, H, D), generator=g, device="cuda").bfloat16()
    q, k, v = r(n_q), r(n_f + n_c) * 0.25, r(n_f + n_c)
    at = torch.randperm(n_f + n_c, generator=torch.Generator().manual_seed(D)).cuda()[:n_q]
    k[0, at] = (q[0].float() * (15.0 * D ** 0.5 / q[0].float().pow(2).sum(-1, keepdim=True))).bfloat16()
    out, status = torch.zeros_like(q), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(max(binding.region_attention_workspace(1, n_q, n_f, n_c, H, D), 256), dtype=torch.uint8, device="cuda")
    kf, vf = (k[:, :n_f].contiguous(), v[:, :n_f].contiguous()) if n_f else (None, None)
    binding.region_attention(q, kf, vf, k[:, n_f:].contiguous(), v[:, n_f:].contiguous(), dev_i32([n_q]), dev_i32([n_f]),
                             dev_i32([n_c]), out, workspace=ws, dev_status=status)
    want = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for h in range(H):
        s = q[0, :, h].double() @ k[0, :, h].double().T * D ** -0.5
        want[0, :, h] = torch.softmax(s, -1) @ v[0, :, h].double()
    assert int(status[0]) == 0
    error = lambda a: float((a.double() - want).norm() / want.norm())
    assert error(out) <= 1.1 * error(want.bfloat16()), (error(out), error(want.bfloat16()))
