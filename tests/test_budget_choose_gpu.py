"""The budget selector around the sizes where its kernels change (2048 candidates, as many requests as SMs) and with
scores that stress the threshold search: zeros, one value for everything, denormals, every budget from
the roots alone to all nodes.  Bit for bit against the oracle, as whole numbers are."""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from oracle import budget_oracle as bo

pytestmark = pytest.mark.gpu

SIZES = [(2, 1), (16, 128), (683, 3), (64, 128), (65, 127), (1024, 8), (1000, 9), (7, 97), (148, 13), (149, 13), (148, 1)]


@pytest.mark.parametrize("scores", ["uniform", "few", "zeros", "ones", "denormal"])
@pytest.mark.parametrize("B,Tc", SIZES)
def test_choose(B, Tc, scores):
    rng = np.random.Generator(np.random.Philox(key=B * 1000 + Tc))
    par = np.stack([inputs.tree_frontier(Tc, rng) for _ in range(B)])
    p = {"uniform": lambda: rng.uniform(0.02, 1.0, (B, Tc)), "few": lambda: rng.choice([0.0, 0.5, 1.0], (B, Tc)),
         "zeros": lambda: np.zeros((B, Tc)), "ones": lambda: np.ones((B, Tc)),
         "denormal": lambda: rng.uniform(0.0, 1e-40, (B, Tc))}[scores]().astype(np.float32)
    N = B * Tc
    for budget in sorted({B, min(B + 1, N), (B + N) // 2, N, N + 5}):
        ref = bo.select(par, p, budget)
        got = tv.budget_select(torch.from_numpy(par).cuda(), torch.from_numpy(p).cuda(), budget)
        torch.cuda.synchronize()
        K = min(budget, N)
        for n in ("counts", "offsets", "parent_packed"):
            assert np.array_equal(got[n].cpu().numpy(), ref[n]), (n, budget)
        node_id = got["node_id"].cpu().numpy()
        assert np.array_equal(node_id[:K], ref["node_id"][:K]) and (node_id[K:] == -1).all()


@pytest.mark.parametrize("B,Tc,few", [(16, 128, True), (0, 13, True), (1, 13, False), (17, 121, False), (1024, 2, False),
                                      (683, 3, False), (1024, 8, False)])
def test_launches(B, Tc, few):
    """Every request's CTA of the two-launch form searches the whole batch's keys: it takes at most 2048
    candidates and one CTA per SM (B = 0, 1: as many requests as SMs, one more)."""
    import ctypes
    if B < 2:
        B += torch.cuda.get_device_properties(0).multi_processor_count
    par = torch.full((B, Tc), -1, dtype=torch.int32, device="cuda")
    p = torch.rand(B, Tc, device="cuda")
    out = tv.budget_select(par, p, B)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        tv.budget_select(par, p, B, out=out)
    n = ctypes.c_size_t()
    runtime = ctypes.CDLL("libcudart.so.12")
    assert runtime.cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    assert n.value == (2 if few else 3)
