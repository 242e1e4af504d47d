"""The commit kernel for dk = 64 and 128 where its CTA shapes change (few, some, many rows per launch),
at value widths that end inside a CTA, with paths shorter and longer than the 16 rows it stages at a
time, rejected requests, from corrections and from values, in place and out of place.

Tolerance: fp32 sums over a path of at most 128 nodes, 1e-5 as for all-fp32 operands elsewhere.
"""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from oracle import tree_oracle as orc
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [inputs.F32, inputs.BF16])
@pytest.mark.parametrize("dk,dv", [(64, 64), (64, 24), (128, 128), (128, 104), (128, 8)])
@pytest.mark.parametrize("B,H,T,tree", [(3, 2, 33, "chain"), (9, 16, 17, "chain"), (48, 16, 40, "frontier"),
                                        (5, 2, 128, "chain"), (40, 16, 1, "chain")])
def test_rows(B, H, T, tree, dk, dv, dtype):
    wl = inputs.workload("c4", B=B, H=H, T=T, dk=dk, dv=dv, tree=tree, rule=inputs.GATED, qkv_dtype=dtype, seed=B + T)
    tens = inputs.make_tensors(wl)
    parents, _ = inputs.make_trees(wl)
    rng = np.random.default_rng(T)
    accepted = rng.integers(-1, T, size=B).astype(np.int32)
    accepted[0], accepted[-1] = T - 1, -1
    dev = {n: None if x is None else x.cuda() for n, x in tens.items()}
    U = torch.randn(B, H, T, dv, device="cuda")
    tree_ = tv.tree_build(parents).upload()
    acc = torch.from_numpy(accepted).cuda()
    f = {n: inputs.to_f64(x) for n, x in tens.items()}
    for u in (None, U):
        value = f["v"] if u is None else inputs.to_f64(u)
        for in_place in (True, False):
            S = dev["S_pre"].clone()
            out = tv.commit_path(tree_, acc, S, dev["k"], dev["v"], dev["alpha"], U=u,
                                 S_new=None if in_place else torch.full_like(S, float("nan")))
            got = inputs.to_f64(out)
            for b in sorted({0, 1, B // 2, B - 1}):
                for h in (0, H - 1):
                    ref = orc.commit_walk(f["S_pre"][b, h].T, f["k"][b, h], value[b, h], f["alpha"][b, h], None,
                                          parents[b], int(accepted[b]), "gated").T
                    assert pu.rel_fro(got[b, h], ref) <= 1e-5
            assert in_place or torch.equal(S, dev["S_pre"])
            assert torch.equal(out[accepted < 0], dev["S_pre"][accepted < 0])


def test_many_64_wide_states():
    """Enough of them that the commit is an ordinary launch (30 CTAs per SM), accepted and rejected requests."""
    B, H, T, d = 160, 32, 20, 64
    wl = inputs.workload("c3", B=B, H=H, T=T, dk=d, dv=d, tree="frontier", seed=17)
    assert B * H >= 30 * torch.cuda.get_device_properties(0).multi_processor_count
    tens = inputs.make_tensors(wl)
    parents, accepted = inputs.make_trees(wl)
    accepted[::7] = -1
    dev = {n: None if x is None else x.cuda() for n, x in tens.items()}
    tree_ = tv.tree_build(parents).upload()
    out = tv.commit_path(tree_, torch.from_numpy(accepted).cuda(), dev["S_pre"].clone(), dev["k"], dev["v"], dev["alpha"])
    got = inputs.to_f64(out)
    f = {n: inputs.to_f64(x) for n, x in tens.items()}
    for b in (0, 1, 7, 80, 159):
        for h in (0, 31):
            ref = orc.commit_walk(f["S_pre"][b, h].T, f["k"][b, h], f["v"][b, h], f["alpha"][b, h], None, parents[b],
                                  int(accepted[b]), "gated").T
            assert pu.rel_fro(got[b, h], ref) <= 1e-5
    assert torch.equal(out[torch.from_numpy(accepted < 0)], dev["S_pre"][torch.from_numpy(accepted < 0)])
