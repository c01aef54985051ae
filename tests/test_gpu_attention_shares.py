"""Items cut between thread blocks and merged by their first share: hand-over through the workspace whatever it
holds, repeated from a CUDA graph, and beside another launch on a second stream."""
import numpy as np
import pytest

from gpu_util import dev_bf16, dev_i32
from paper_2510_25590_b200 import binding
from test_gpu_attention import _rand_bf16, check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("H,n_q,n_f,n_c", [
    (24, 819, 819, 7000),       # three pairs and a lone tile; an item meets two or three shares
    (24, 1800, 300, 4500),      # more items than thread blocks, some whole
    (24, 819, 819, 900),        # short shares: merged by the second kernel
])
def test_first_share_merges(D, H, n_q, n_f, n_c):
    rng = np.random.default_rng(D + H + n_q)
    r = lambda n: _rand_bf16(rng, (1, n, H, D))
    check(r(n_q), r(n_f), r(n_f), r(n_c), r(n_c), [n_q], [n_f], [n_c], what=f"cut items, D={D}")


def test_any_workspace_content_graphs_and_streams():
    import torch
    rng = np.random.default_rng(5)
    H, D, n_q, n_c = 24, 128, 1000, 8000
    r = lambda n: dev_bf16(_rand_bf16(rng, (1, n, H, D)))
    q, kf, vf, kc, vc = r(n_q), r(n_q), r(n_q), r(n_c), r(n_c)
    nq, nc = dev_i32([n_q]), dev_i32([n_c])
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    size = binding.region_attention_workspace(1, n_q, n_q, n_c, H, D)

    def call(out, ws, stream=None):
        binding.region_attention(q, kf, vf, kc, vc, nq, nq, nc, out, workspace=ws, dev_status=status, stream=stream)

    outs = []
    for fill in (0, 255, 1):
        ws, out = torch.full((size,), fill, dtype=torch.uint8, device="cuda"), torch.zeros_like(q)
        call(out, ws)
        outs.append(out)
    ws, out = torch.full((size,), 7, dtype=torch.uint8, device="cuda"), torch.zeros_like(q)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(out, ws)
    for _ in range(5):
        out.zero_()
        graph.replay()
        outs.append(out.clone())
    streams = [torch.cuda.Stream() for _ in range(2)]
    pairs = [(torch.empty(size, dtype=torch.uint8, device="cuda"), torch.zeros_like(q)) for _ in streams]
    torch.cuda.synchronize()
    for _ in range(20):
        for s, (w, o) in zip(streams, pairs):
            call(o, w, s)
    torch.cuda.synchronize()
    outs += [o for _, o in pairs]
    assert int(status[0]) == 0
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
