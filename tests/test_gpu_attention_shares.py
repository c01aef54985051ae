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


def _captured_epoch(graph):
    """The number that tells a captured launch's flags from others': in the kernel's parameters, ahead of the bound of
    its waits (4e9 cycles)."""
    import ctypes
    from cuda.bindings import driver
    err, _, n = driver.cuGraphGetNodes(driver.CUgraph(graph.raw_cuda_graph()), 0)
    assert int(err) == 0
    err, nodes, n = driver.cuGraphGetNodes(driver.CUgraph(graph.raw_cuda_graph()), n)
    assert int(err) == 0
    kernels = [k for k in nodes if driver.cuGraphNodeGetType(k)[1] == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL]
    assert len(kernels) == 1                                   # merged by the first shares: no second kernel
    err, params = driver.cuGraphKernelNodeGetParams(kernels[0])
    assert int(err) == 0
    at = (ctypes.c_void_p * 6).from_address(int(params.kernelParams))[5]      # (five tensor maps ahead of it)
    words = (ctypes.c_uint64 * 18).from_address(at)
    assert words[17] == 4_000_000_000
    return words[16]


def test_a_launch_that_timed_out_is_not_repeated_over_its_leftovers():
    """A repetition by a graph has the epoch of the launch that timed out: told so by the workspace's last word, it
    records the time-out again and merges nothing, whatever flags lie there; with the word overwritten it works as before."""
    import torch
    rng = np.random.default_rng(6)
    H, D, n_q, n_c = 24, 128, 1000, 8000
    r = lambda n: dev_bf16(_rand_bf16(rng, (1, n, H, D)))
    q, kf, vf, kc, vc = r(n_q), r(n_q), r(n_q), r(n_c), r(n_c)
    nq, nc = dev_i32([n_q]), dev_i32([n_c])
    status, out = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros_like(q)
    ws = torch.zeros(binding.region_attention_workspace(1, n_q, n_q, n_c, H, D), dtype=torch.uint8, device="cuda")
    call = lambda: binding.region_attention(q, kf, vf, kc, vc, nq, nq, nc, out, workspace=ws, dev_status=status)
    call()
    want = out.clone()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    epoch = _captured_epoch(graph)
    graph.instantiate()
    last = torch.frombuffer(bytearray(int(epoch).to_bytes(8, "little")), dtype=torch.uint8).cuda()
    for failed in (False, True, False):
        out.fill_(-3.0)
        status.zero_()
        ws[-8:] = last if failed else 0
        graph.replay()
        torch.cuda.synchronize()
        assert int(status[0]) == (binding.DEV_TIMEOUT if failed else 0)
        assert failed or torch.equal(out, want)
        rows = ((out == -3.0).all(-1) | (out == want).all(-1))                 # left out or as they should be
        assert bool(rows.all()) and (not failed or bool((out == -3.0).all(-1).any()))
    call()                                                     # (a launch of its own has another epoch)
    assert torch.equal(out, want)
