"""The budget selector around the sizes where its kernels change (2048 and 8192 candidates) and with
scores that stress the threshold search: zeros, one value for everything, denormals, every budget from
the roots alone to all nodes.  Bit for bit against the oracle, as whole numbers are."""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from oracle import budget_oracle as bo

pytestmark = pytest.mark.gpu

SIZES = [(2, 1), (16, 128), (683, 3), (64, 128), (65, 127), (1024, 8), (1000, 9), (7, 97)]


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
