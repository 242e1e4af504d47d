"""Delta-rule tensor-core kernels (one and two row blocks of 64 nodes): edges of the blocks, many items per
CTA, requests that share a box with another request's rows."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from tests.parity_util import compare, gpu_round, oracle_round

pytestmark = pytest.mark.gpu

# State, V' and the rows of W and A enter the tensor core as two bf16 each, 16 bits and a rounding: a term of
# a sum is off by at most 3 * 2^-17 of itself, and the terms of these sums are up to eight times their result.
BOUND = 8 * 3 * 2.0 ** -17


@pytest.mark.parametrize("T,tree,want_U", [(1, "chain", True), (15, "chain", True), (33, "frontier", True), (63, "spine", False),
                                           (64, "frontier", True), (65, "frontier", True), (96, "spine", False),
                                           (97, "frontier", True), (128, "spine", True)])
def test_blocks_and_rounds(T, tree, want_U):
    # a persistent CTA works through three or four items; the last round is incomplete
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    H = 7
    B = (3 * sms + 5) // H + 1
    wl = dataclasses.replace(inputs.workload("c4"), B=B, H=H, T=T, tree=tree, seed=100 + T)
    parents, accepted = inputs.make_trees(wl)
    tens = inputs.make_tensors(wl)
    items = [(0, 0), (0, H - 1), (B // 3, 3), (B // 2, 1), (B - 1, 0), (B - 1, H - 1)]
    O, U, Sn, tree_h = gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_TC, want_U=want_U, commit_with_U=want_U)
    tree_h.device_status()
    ver, com = oracle_round(wl, parents, accepted, tens, items=items)
    eO, eU, eS = compare(wl, O, U, Sn, ver, com)
    assert eO < BOUND and eU < BOUND and eS < BOUND, (eO, eU, eS)


@pytest.mark.parametrize("n_max,sizes", [(64, [33, 1, 64, 40, 9, 17]), (128, [65, 3, 128, 64, 100, 1])])
def test_non_finite_rows_stay_in_their_request(n_max, sizes):
    # boxes reach into the rows of the next request: its values, whatever they are, must not
    H = 3
    rng = np.random.default_rng(n_max)
    parents = [np.array([-1] + [int(rng.integers(max(0, i - 4), i)) for i in range(1, n)], dtype=np.int32) for n in sizes]
    def depth(par):
        d = np.zeros(len(par), dtype=int)
        for i, p in enumerate(par):
            d[i] = d[p] + 1 if p >= 0 else 0
        return d.max()

    parents = [p if depth(p) <= 15 else np.array([-1] + [(i - 1) // 2 for i in range(1, len(p))], dtype=np.int32) for p in parents]
    cap = sum(sizes)
    wl = dataclasses.replace(inputs.workload("c4"), B=1, H=H, T=cap, seed=5)
    t = {n: None if x is None else x[0].cuda() for n, x in inputs.make_tensors(wl).items()}
    S = inputs.make_tensors(dataclasses.replace(wl, B=len(sizes), T=1))["S_pre"].cuda()
    forest = tv.forest_build(parents, n_max=n_max).upload()
    off = forest.offsets

    def run(x):
        O = torch.zeros(H, cap, 128, device="cuda")
        U = torch.zeros_like(O)
        tv.tree_verify(forest, S, x["q"], x["k"], x["v"], x["alpha"], x["beta"], rule=tv.DELTA, O=O, U=U, impl=tv.IMPL_TC)
        forest.device_status()
        return O, U

    O0, U0 = run(t)
    assert torch.isfinite(O0).all() and torch.isfinite(U0).all()
    for bad in (1, 3, 5):
        x = {n: v.clone() for n, v in t.items() if v is not None}
        for n in ("q", "k", "v"):
            x[n][:, off[bad]:off[bad + 1]] = float("nan")
        O, U = run(x)
        for r in range(len(sizes)):
            rows = slice(off[r], off[r + 1])
            if r == bad:
                assert torch.isnan(O[:, rows]).all()
            else:
                assert torch.equal(O[:, rows], O0[:, rows]) and torch.equal(U[:, rows], U0[:, rows])


@pytest.mark.parametrize("T,tree", [(1, "chain"), (15, "chain"), (40, "frontier"), (64, "frontier"), (100, "spine"), (128, "frontier")])
@pytest.mark.parametrize("gate,value", [("alpha", float("nan")), ("alpha", float("inf")), ("beta", float("nan"))])
def test_non_finite_gate_reaches_its_subtree_alone(T, tree, gate, value):
    # a node's output depends on its root path: a gate elsewhere, whatever it is, does not change it
    wl = dataclasses.replace(inputs.workload("c4"), B=2, H=2, T=T, tree=tree, seed=11)
    parents, _ = inputs.make_trees(wl)
    t = {n: x.cuda() for n, x in inputs.make_tensors(wl).items()}
    tree_h = tv.tree_build(parents).upload()
    anc, _, _ = tree_h.meta()

    def run(t):
        return tv.tree_verify(tree_h, *[t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")], rule=tv.DELTA, want_U=True,
                              impl=tv.IMPL_TC)

    O0, U0 = run(t)
    for node in sorted({0, T // 3, T // 2, T - 1}):
        x = dict(t)
        x[gate] = t[gate].clone()
        x[gate][1, 0, node] = value
        O, U = run(x)
        tree_h.device_status()
        hit = np.array([i == node or bool(int(anc[1, i, node >> 6]) >> (node & 63) & 1) for i in range(T)])
        free = torch.from_numpy(~hit).cuda()
        assert torch.isnan(O[1, 0][~free]).all() and torch.isnan(U[1, 0][~free]).all()
        assert torch.equal(O[1, 0][free], O0[1, 0][free]) and torch.equal(U[1, 0][free], U0[1, 0][free])
        assert torch.equal(O[0], O0[0]) and torch.equal(O[1, 1], O0[1, 1]) and torch.equal(U[0], U0[0]) and torch.equal(U[1, 1], U0[1, 1])


@pytest.mark.parametrize("T", [40, 100])
def test_states_beyond_the_largest_bf16(T):
    # the largest fp32 numbers round to infinity in bf16; the two pieces together must still hold them
    wl = dataclasses.replace(inputs.workload("c4"), B=1, H=2, T=T, tree="frontier", seed=3)
    parents, accepted = inputs.make_trees(wl)
    t = inputs.make_tensors(wl)
    t["S_pre"][0, 0, 5, 7] = 3.4e38
    t["S_pre"][0, 1, 9, 7] = -3.4028234e38
    t["k"][..., 7] = 0                      # the keys leave the entry alone, the queries read a part of it
    t["q"] = t["q"] * 2.0 ** -20
    O, U, Sn, tree_h = gpu_round(wl, parents, accepted, t, impl=tv.IMPL_TC)
    tree_h.device_status()
    ver, com = oracle_round(wl, parents, accepted, t)
    eO, eU, eS = compare(wl, O, U, Sn, ver, com)
    assert eO < BOUND and eU < BOUND and eS < BOUND, (eO, eU, eS)
