"""Gated tensor-core kernel, two items on a CTA and operands that land before the state does.

Stage 1 leaves q, k and v in L2 while the states come from memory, so the second item's q and k can
have landed before the first item's state.  The order in which a CTA asks for its loads must not depend
on which of them is there first: the kernel's waits are bounded, and one that runs out is reported by
``device_status``."""
import dataclasses

import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,T", [(16, 16, 17), (10, 15, 64), (37, 8, 5)])
def test_operands_before_the_state(B, H, T):
    wl = dataclasses.replace(inputs.workload("c3"), B=B, H=H, T=T, L=1, seed=31 + T, tree="frontier")
    parents, accepted = inputs.make_trees(wl)
    tree = tv.tree_build(parents).upload()
    acc = torch.from_numpy(accepted).cuda()
    dims = dict(H=H, dk=128, dv=128)
    empty = lambda: torch.empty(B, H, T, 128, device="cuda", dtype=torch.bfloat16)
    sets = []
    for s in range(3):
        g = inputs.make_conv_inputs(dataclasses.replace(wl, seed=s), device="cuda", W=4)
        S = inputs.make_tensors(dataclasses.replace(wl, T=1, seed=s), device="cuda")["S_pre"]
        y = dict(q=empty(), k=empty(), v=empty(), alpha=torch.empty(B, H, T, device="cuda"),
                 beta=torch.empty(B, H, T, device="cuda"))
        sets.append((g, S, y, torch.zeros(B, H, T, 128, device="cuda")))
    for i in range(900):
        g, S, y, O = sets[i % 3]
        q, k, v, alpha, _ = tv.tree_conv(tree, g["x"], g["ctx"], g["weight"], g["bias"], gate_a=g["gate_a"],
                                         gate_b=g["gate_b"], A_log=g["A_log"], dt_bias=g["dt_bias"],
                                         normalize_qk=True, **dims, **y)
        tv.tree_verify(tree, S, q, k, v, alpha, rule=tv.GATED, O=O)
        tv.commit_path(tree, acc, S, k, v, alpha, rule=tv.GATED)
        tv.conv_commit(tree, acc, g["x"], g["ctx"], **dims)
    tree.device_status()   # raises if a wait ran out in any of the passes
    for _, S, _, O in sets:
        assert torch.isfinite(S).all() and torch.isfinite(O).all()
