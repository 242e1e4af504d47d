"""The general fp32 verify kernels where their tiles, forms and column chunks change: row tiles of 16
nodes, one or two row blocks, path form (at most 15 ancestors) and block form, chunks of 32, 64 and
128 value columns, widths that are no multiple of a tile, packed forests with both kinds of trees.

Tolerance: fp32 sums of at most 128 products and 128 corrections, 1e-5 as everywhere for all-fp32
operands; chains of more than 64 nodes 5e-5 (128 sequential fp32 steps).
"""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def _check(wl, parents, accepted, tens, tol):
    O, U, Sn, tree = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT, commit_with_U=True)
    items = [(0, 0), (wl.B - 1, wl.H - 1), (wl.B // 2, wl.H // 2)]
    ver, com = pu.oracle_round(wl, parents, accepted, tens, items=items)
    errs = pu.compare(wl, O, U, Sn, ver, com)
    assert max(errs) <= tol, errs


SIZES = [1, 15, 16, 17, 31, 33, 48, 49, 64, 65, 95, 96, 97, 128]


@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
@pytest.mark.parametrize("tree", ["frontier", "chain"])
@pytest.mark.parametrize("T", SIZES)
def test_row_tiles_and_forms(T, tree, rule):
    # 6, 60 and 200 items: chunks of 32, 64 and 128 of the value columns
    for B, H in ((2, 3), (10, 6), (25, 8)):
        wl = inputs.workload("c4", B=B, H=H, T=T, rule=rule, tree=tree, qkv_dtype=inputs.F32, seed=10 * T + B)
        tens = inputs.make_tensors(wl)
        tens["k"] = tens["k"] * (8.0 / wl.dk ** 0.5)
        parents, accepted = inputs.make_trees(wl)
        _check(wl, parents, accepted, tens, 5e-5 if tree == "chain" and T > 64 else 1e-5)


@pytest.mark.parametrize("dk,dv,dtype", [(4, 4, inputs.F32), (36, 100, inputs.F32), (8, 72, inputs.BF16),
                                         (120, 40, inputs.BF16), (64, 128, inputs.F32)])
@pytest.mark.parametrize("T,tree", [(23, "frontier"), (40, "chain"), (70, "frontier"), (100, "chain")])
def test_odd_widths(dk, dv, dtype, T, tree):
    for B, H in ((1, 2), (16, 16)):
        wl = inputs.workload("c4", B=B, H=H, T=T, dk=dk, dv=dv, tree=tree, qkv_dtype=dtype, seed=T + dk)
        tens = inputs.make_tensors(wl)
        if dtype == inputs.F32:
            tens["k"] = tens["k"] * (8.0 / dk ** 0.5)
        parents, accepted = inputs.make_trees(wl)
        _check(wl, parents, accepted, tens, 5e-5 if tree == "chain" and T > 64 else 1e-5)


@pytest.mark.parametrize("n_max", [60, 128])
def test_forest_with_shallow_and_deep_trees(n_max):
    """A request picks its form by its own tree (up to 64 nodes), and a tree of one block may share a
    launch with trees of two."""
    rng = np.random.default_rng(3)
    H, d = 4, 128
    par = [inputs.tree_chain(n_max), inputs.tree_frontier(n_max, rng), inputs.tree_chain(16), inputs.tree_chain(17),
           inputs.tree_frontier(1, rng), inputs.tree_frontier(n_max // 2, rng)]
    forest = tv.forest_build(par, n_max=n_max).upload()
    N = int(forest.offsets[-1])
    wl = inputs.workload("c4", B=1, H=H, T=N, qkv_dtype=inputs.F32, seed=77)
    t = inputs.make_tensors(wl)
    t["k"] = t["k"] * (8.0 / d ** 0.5)
    S = inputs.make_tensors(inputs.workload("c4", B=len(par), H=H, T=1, seed=78))["S_pre"]
    dev = {n: t[n][0].cuda() for n in ("q", "k", "v", "alpha", "beta")}
    O, U = tv.tree_verify(forest, S.cuda(), dev["q"], dev["k"], dev["v"], dev["alpha"], dev["beta"], rule=tv.DELTA,
                          want_U=True, impl=tv.IMPL_SIMT)
    torch.cuda.synchronize()
    from oracle import tree_oracle as orc
    for b, p in enumerate(par):
        lo, hi = int(forest.offsets[b]), int(forest.offsets[b + 1])
        cut = {n: inputs.to_f64(t[n][:, :, lo:hi]) for n in dev}
        ver = orc.verify_batch(inputs.to_f64(S[b:b + 1]), cut["q"], cut["k"], cut["v"], cut["alpha"], cut["beta"],
                               p[None], "delta")
        for h in range(H):
            Or, Ur = ver[(0, h)]
            assert pu.rel_l2_rows(inputs.to_f64(O[h, lo:hi]), Or) <= 5e-5
            assert pu.rel_l2_rows(inputs.to_f64(U[h, lo:hi]), Ur) <= 5e-5


@pytest.mark.parametrize("T,tree", [(30, "frontier"), (40, "chain"), (100, "frontier"), (100, "chain")])
def test_nan_stays_on_its_paths(T, tree):
    """A non-finite value row reaches the nodes below it and no others."""
    wl = inputs.workload("c4", B=2, H=2, T=T, tree=tree, qkv_dtype=inputs.F32, seed=T)
    tens = inputs.make_tensors(wl)
    tens["k"] = tens["k"] * (8.0 / wl.dk ** 0.5)
    parents, accepted = inputs.make_trees(wl)
    clean = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[0]
    bad = T // 2
    tens["v"][0, :, bad] = float("nan")
    O = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[0]
    from oracle import tree_oracle as orc
    hit = np.array([bad in orc.path_to(parents[0], i) for i in range(T)])
    assert np.isnan(O[0][:, hit]).all()
    assert np.array_equal(O[0][:, ~hit], clean[0][:, ~hit]) and np.array_equal(O[1], clean[1])


@pytest.mark.parametrize("zero", ["gate", "key"])
@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
@pytest.mark.parametrize("T,tree", [(30, "frontier"), (40, "chain"), (100, "frontier"), (100, "chain")])
def test_a_zero_coefficient_does_not_hide_a_nan(T, tree, rule, zero):
    """The coefficients below a non-finite value row are exactly zero, from a gate of zero or from the
    row's own key: 0 x NaN is NaN for every node of the paths through it, in both forms."""
    wl = inputs.workload("c4", B=2, H=2, T=T, rule=rule, tree=tree, qkv_dtype=inputs.F32, seed=T)
    tens = inputs.make_tensors(wl)
    tens["k"] = tens["k"] * (8.0 / wl.dk ** 0.5)
    parents, accepted = inputs.make_trees(wl)
    from oracle import tree_oracle as orc
    below = [sum(n in orc.path_to(parents[0], i) for i in range(T)) for n in range(T)]
    bad = max(range(1, T), key=lambda n: below[n] if n >= T // 8 else 0)   # a node with many below it
    hit = np.array([bad in orc.path_to(parents[0], i) for i in range(T)])
    assert hit.sum() > 1
    if zero == "gate":
        tens["alpha"][0][:, torch.from_numpy(parents[0] == bad)] = 0.0
    else:
        tens["k"][0, :, bad] = 0.0
    O0, U0 = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[:2]
    assert np.isfinite(O0).all()
    tens["v"][0, :, bad] = float("nan")
    O, U = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[:2]
    assert np.isnan(O[0][:, hit]).all()
    assert np.array_equal(O[0][:, ~hit], O0[0][:, ~hit]) and np.array_equal(O[1], O0[1])
    if rule == inputs.DELTA:
        assert np.isnan(U[0][:, hit]).all() and np.array_equal(U[0][:, ~hit], U0[0][:, ~hit])


@pytest.mark.parametrize("dtype", [inputs.F32, inputs.BF16])
@pytest.mark.parametrize("T", [40, 64, 90, 128])
def test_corrections_of_long_chains_keep_their_precision(T, dtype):
    """A correction is its right-hand side (three roundings) less two sums over its path, each summed from
    zero and subtracted once: five roundings of 2^-24 / sqrt(3) root mean square at the size of the result,
    7.7e-8, and the sums' own errors, which are smaller as the sums are.  Subtracting the path's terms one
    by one rounds at that size up to 127 times: 1.2e-7 at 40 nodes, 2.1e-7 at 128."""
    wl = inputs.workload("c4", B=2, H=8, T=T, tree="chain", qkv_dtype=dtype, seed=T)
    tens = inputs.make_tensors(wl)
    if dtype == inputs.F32:
        tens["k"] = tens["k"] * (8.0 / wl.dk ** 0.5)
    parents, accepted = inputs.make_trees(wl)
    U = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[1]
    ver, _ = pu.oracle_round(wl, parents, accepted, tens)
    ref = np.stack([np.stack([ver[(b, h)][1] for h in range(wl.H)]) for b in range(wl.B)])
    assert pu.rel_fro(U, ref) <= 1e-7


def _tree_of_depth(T, depth, rng):
    """T nodes, the deepest with exactly `depth` ancestors (node `depth` is one of them)."""
    return inputs.tree_frontier(T, rng, max_depth=depth, spine=depth + 1)


@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
@pytest.mark.parametrize("depth", [15, 16])
@pytest.mark.parametrize("T", [17, 64, 65, 96, 97, 128])
def test_the_depth_where_the_forms_change(T, depth, rule):
    """15 ancestors fill the path form's tables; one more takes the block form."""
    rng = np.random.default_rng(T)
    for B, H in ((2, 3), (10, 6), (25, 8)):
        wl = inputs.workload("c4", B=B, H=H, T=T, rule=rule, qkv_dtype=inputs.F32, seed=T + depth)
        tens = inputs.make_tensors(wl)
        tens["k"] = tens["k"] * (8.0 / wl.dk ** 0.5)
        parents = np.stack([_tree_of_depth(T, depth, rng) for _ in range(B)])
        assert inputs.node_depths(parents[0]).max() == depth
        accepted = rng.integers(-1, T, size=B).astype(np.int32)
        accepted[0], accepted[-1], accepted[B // 2] = depth, T - 1, depth
        _check(wl, parents, accepted, tens, 1e-5)


@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
def test_forest_from_the_device_at_the_path_forms_depth(rule):
    """A bound of 15 on more than 64 nodes selects the path form: the deepest trees it admits."""
    from oracle import tree_oracle as orc
    rng = np.random.default_rng(5)
    B, H, n, d = 3, 2, 100, 128
    par = np.stack([_tree_of_depth(n, 15, rng) for _ in range(B)])
    forest = tv.forest_build([np.array([-1], dtype=np.int32)] * B, n_max=n, capacity=B * n)
    forest.upload_device(torch.from_numpy(par).cuda(), torch.arange(0, (B + 1) * n, n, dtype=torch.int32, device="cuda"),
                         max_depth_bound=15)
    wl = inputs.workload("c4", B=1, H=H, T=B * n, rule=rule, qkv_dtype=inputs.F32, seed=9)
    t = inputs.make_tensors(wl)
    t["k"] = t["k"] * (8.0 / d ** 0.5)
    S = inputs.make_tensors(inputs.workload("c4", B=B, H=H, T=1, seed=10))["S_pre"]
    names = ("q", "k", "v", "alpha", "beta")
    dev = {m: None if t[m] is None else t[m][0].cuda() for m in names}
    O, U = tv.tree_verify(forest, S.cuda(), *[dev[m] for m in names], rule=rule, want_U=True, impl=tv.IMPL_SIMT)
    forest.device_status()
    for b in range(B):
        cut = {m: None if t[m] is None else inputs.to_f64(t[m][:, :, b * n:(b + 1) * n]) for m in names}
        ver = orc.verify_batch(inputs.to_f64(S[b:b + 1]), *[cut[m] for m in names], par[b][None], wl.rule_name)
        for h in range(H):
            assert pu.rel_l2_rows(inputs.to_f64(O[h, b * n:(b + 1) * n]), ver[(0, h)][0]) <= 1e-5
            assert pu.rel_l2_rows(inputs.to_f64(U[h, b * n:(b + 1) * n]), ver[(0, h)][1]) <= 1e-5
