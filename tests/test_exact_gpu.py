"""The verify kernels at fp32 accuracy on the tensor cores (what `auto` takes for f32 operands, for the delta
rule on trees deeper than the other tensor-core kernels hold, and for 64-wide heads): blocks of 16 nodes, path
and block form, one or two halves of the value columns, several items on a CTA.

Tolerances: 1e-5 per node as everywhere for all-fp32 operands.  Whole tensors: 1.5e-7.  An operand in three
bf16 pieces is exact to 2^-24; a product drops three of nine piece products, each below 2^-24 of it; the sums are
fp32, four truncated steps on top of smaller ones in two halves, 2^-23 each at most and half of that on average, then
at most four roundings: 1.4e-7 of the result's norm where partial sums are no larger than it."""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from oracle import tree_oracle as orc
from paper_2608_01651_b200 import inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def _inputs(B, H, T, rule, tree, dtype, dk=128, dv=128, seed=0):
    wl = inputs.workload("c4", B=B, H=H, T=T, dk=dk, dv=dv, rule=rule, tree=tree, qkv_dtype=dtype, seed=seed + T)
    tens = inputs.make_tensors(wl)
    if dtype == inputs.F32:
        tens["k"] = tens["k"] * (8.0 / dk ** 0.5)
    return (wl,) + inputs.make_trees(wl) + (tens,)


def _takes(wl, parents, tens):
    """The call goes to this kernel: with another rule the cases here would test another one."""
    t = {n: None if x is None else x.cuda() for n, x in tens.items()}
    tree = tv.tree_build(parents).upload()
    O = torch.empty(t["v"].shape, device="cuda")
    launched = pu.kernels_of(lambda: tv.tree_verify(tree, *[t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")], rule=wl.rule, O=O))
    return len(launched) == 1 and "verify_exact_kernel" in launched[0][0]


def _check(wl, parents, accepted, tens, whole=1.5e-7):
    assert _takes(wl, parents, tens)
    O, U, Sn, tree = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_AUTO, commit_with_U=True)
    tree.device_status()
    n = wl.B * wl.H
    items = sorted({(i // wl.H, i % wl.H) for i in (0, 1, n // 2, n - 1, min(n - 1, 148), min(n - 1, 149))})
    ver, com = pu.oracle_round(wl, parents, accepted, tens, items=items)
    errs = pu.compare(wl, O, U, Sn, ver, com)
    assert max(errs) <= 1e-5, errs
    for x, which in ((O, 0),) + (((U, 1),) if wl.rule == inputs.DELTA else ()):
        got, ref = (np.stack(y) for y in ([x[i] for i in items], [ver[i][which] for i in items]))
        assert pu.rel_fro(got, ref) <= whole


@pytest.mark.parametrize("tree", ["frontier", "chain"])
@pytest.mark.parametrize("T", [17, 32, 33, 48, 49, 63, 64])
def test_delta(T, tree):
    # 6 items: halves; 80: whole columns; 200: two items on a CTA
    for B, H in ((2, 3), (10, 8), (25, 8)):
        if T > 32 or B == 10 or (B == 25 if tree == "chain" else T == 32 and B == 2):   # others: the general kernel's
            _check(*_inputs(B, H, T, inputs.DELTA, tree, inputs.F32, seed=B))
    if tree == "chain":
        for B, H in ((2, 3), (25, 8)):
            _check(*_inputs(B, H, T, inputs.DELTA, tree, inputs.BF16, seed=B))


@pytest.mark.parametrize("T", [49, 64])
@pytest.mark.parametrize("tree", ["frontier", "chain"])
def test_gated(T, tree):
    for B, H in ((5, 8), (10, 8), (25, 8)):
        _check(*_inputs(B, H, T, inputs.GATED, tree, inputs.F32, seed=B))


@pytest.mark.parametrize("dk,dv", [(64, 64), (64, 128), (128, 64)])
@pytest.mark.parametrize("dtype", [inputs.F32, inputs.BF16])
@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
def test_other_widths(rule, dtype, dk, dv):
    if dtype == inputs.BF16 and rule == inputs.GATED and dk == dv:
        pytest.skip("a kernel of its own")
    for T, tree in ((31, "chain"), (50, "frontier"), (64, "chain")):
        for B, H in ((3, 2), (10, 8), (25, 8)):
            # the general kernel's
            if rule == inputs.GATED and (T < 49 or B == 3 or B == 25 and dv == 64):
                continue
            if rule == inputs.DELTA and dtype == inputs.F32 and tree == "chain" and (B != 10 if T < 33 else B == 3 and dk == 64):
                continue
            if rule == inputs.DELTA and dtype == inputs.BF16 and T < 33 and B == 3 and dk < dv:
                continue
            _check(*_inputs(B, H, T, rule, tree, dtype, dk=dk, dv=dv, seed=B))


@pytest.mark.parametrize("rule,dtype,dk,dv,T,tree,B", [
    (inputs.DELTA, inputs.BF16, 128, 128, 40, "chain", 80),      # 640 items: four and five a CTA, q and k in two sets of rows
    (inputs.DELTA, inputs.BF16, 64, 128, 50, "frontier", 80),
    (inputs.DELTA, inputs.BF16, 64, 64, 33, "chain", 63),        # 504
    (inputs.DELTA, inputs.F32, 128, 128, 64, "chain", 57),       # 456
    (inputs.GATED, inputs.F32, 64, 128, 49, "frontier", 57),
    (inputs.GATED, inputs.BF16, 128, 64, 64, "chain", 57),
    (inputs.GATED, inputs.BF16, 64, 128, 49, "frontier", 1),     # 8: halves
    (inputs.GATED, inputs.BF16, 64, 128, 64, "chain", 1)])
def test_many_items_and_few(rule, dtype, dk, dv, T, tree, B):
    _check(*_inputs(B, 8, T, rule, tree, dtype, dk=dk, dv=dv, seed=B))


def test_packed_forest_of_64_wide_heads_under_the_gated_rule():
    """bf16 operands: dense batches of these have a kernel of their own, packed ones come here."""
    rng = np.random.default_rng(4)
    H, d = 6, 64
    par = [inputs.tree_chain(64), inputs.tree_frontier(40, rng), inputs.tree_frontier(1, rng), inputs.tree_frontier(64, rng), inputs.tree_chain(49)]
    forest = tv.forest_build(par, n_max=64).upload()
    N = int(forest.offsets[-1])
    t = _inputs(1, H, N, inputs.GATED, "chain", inputs.BF16, dk=d, dv=d)[3]
    S = inputs.make_tensors(inputs.workload("c4", B=len(par), H=H, T=1, dk=d, dv=d, seed=78))["S_pre"]
    dev = [S.cuda()] + [t[n][0].cuda() for n in ("q", "k", "v", "alpha")] + [None]
    O, U = torch.full((H, N, d), 7.0, device="cuda"), torch.full((H, N, d), 7.0, device="cuda")
    call = lambda: tv.tree_verify(forest, *dev, rule=tv.GATED, O=O, U=U)
    (name, _), = pu.kernels_of(call)
    assert "verify_exact_kernel" in name
    call()
    forest.device_status()
    for b, p in enumerate(par):
        lo, hi = int(forest.offsets[b]), int(forest.offsets[b + 1])
        cut = {n: inputs.to_f64(t[n][:, :, lo:hi]) for n in ("q", "k", "v", "alpha")}
        ver = orc.verify_batch(inputs.to_f64(S[b:b + 1]), *cut.values(), None, p[None], "gated")
        for h in range(H):
            assert pu.rel_l2_rows(inputs.to_f64(O[h, lo:hi]), ver[(0, h)][0]) <= 1e-5
            assert torch.equal(U[h, lo:hi].cpu(), t["v"][0, h, lo:hi].float())


@pytest.mark.parametrize("depth", [15, 16])
def test_the_depth_where_the_forms_change(depth):
    rng = np.random.default_rng(depth)
    for T in (25, 40, 64):
        wl, _, _, tens = _inputs(5, 8, T, inputs.DELTA, "frontier", inputs.F32)
        parents = np.stack([inputs.tree_frontier(T, rng, max_depth=depth, spine=depth + 1) for _ in range(5)])
        accepted = np.array([depth, T - 1, -1, 0, depth], dtype=np.int32)
        _check(wl, parents, accepted, tens)


def test_more_items_than_a_cta_keeps_a_record_of():
    wl, parents, accepted, tens = _inputs(160, 32, 33, inputs.DELTA, "frontier", inputs.F32, dk=64, dv=64)
    _check(wl, parents, accepted, tens)


@pytest.mark.parametrize("full,more", [(0, 1), (1, 0), (1, 1), (32, 0), (32, 1), (33, 5), (64, 0), (64, 1)])
def test_every_sm_gets_as_many_ctas_as_the_others(full, more):
    """A CTA takes at most 32 items and an SM to itself; a few CTAs beyond a multiple of the SMs would run alone at the end."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = full * sms + more
    t = {x: torch.empty(n, 1, 64, d, device="cuda") for x, d in (("S_pre", 64), ("q", 64), ("k", 64), ("v", 64), ("O", 64), ("U", 64))}
    gates = torch.empty(n, 1, 64, device="cuda")
    tree = tv.tree_build(np.stack([inputs.tree_chain(64)])).upload()
    call = lambda: tv.tree_verify(tree, *[t[x] for x in ("S_pre", "q", "k", "v")], gates, gates, rule=tv.DELTA, O=t["O"], U=t["U"])
    if n < 33:   # the general kernel's
        tree = tv.tree_build(np.stack([inputs.tree_frontier(64, np.random.default_rng(1))])).upload()
    (name, grid), = pu.kernels_of(call)
    assert "verify_exact_kernel" in name
    assert grid == (n if n < sms else sms * -(-n // (32 * sms)))


@pytest.mark.parametrize("rule,dtype,tree,T,dk,dv,line", [
    (inputs.DELTA, inputs.F32, "chain", 24, 64, 64, "half"), (inputs.DELTA, inputs.F32, "chain", 32, 128, 64, "half"),
    (inputs.DELTA, inputs.F32, "chain", 17, 64, 128, "quarter"), (inputs.DELTA, inputs.F32, "chain", 32, 128, 128, "quarter"),
    (inputs.GATED, inputs.F32, "chain", 56, 64, 128, "quarter"), (inputs.GATED, inputs.F32, "frontier", 64, 128, 128, "quarter"),
    (inputs.GATED, inputs.F32, "chain", 49, 128, 64, "half"), (inputs.DELTA, inputs.F32, "frontier", 29, 128, 128, 2),
    (inputs.DELTA, inputs.F32, "frontier", 32, 64, 64, 2)])
def test_the_general_kernel_keeps_few_items(rule, dtype, tree, T, dk, dv, line):
    """As long as the general kernel has an SM for every part of an item's columns (four of 128, two of 64), and on one or
    two small trees, it is the faster one: 7.7 us against 8.6 on 64 chains of 24 nodes, 64 x 64."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = {"half": sms // 2, "quarter": sms // 4}.get(line, line)
    trees = tv.tree_build(np.stack([inputs.tree_chain(T) if tree == "chain" else inputs.tree_frontier(T, np.random.default_rng(T))])).upload()
    for items, name in ((n, "verify_simt"), (n + 1, "verify_exact")):
        t = [torch.empty(items, 1, r, d, device="cuda") for r, d in ((dv, dk), (T, dk), (T, dk), (T, dv))]
        gates, O = torch.empty(items, 1, T, device="cuda"), torch.empty(items, 1, T, dv, device="cuda")
        launched = pu.kernels_of(lambda: tv.tree_verify(trees, *t, gates, gates if rule else None, rule=rule, O=O))
        assert len(launched) == 1 and name in launched[0][0], (items, launched)


def test_packed_forest_and_strides():
    """Requests of 1 to 64 nodes, shallow and deep; grouped key heads and token-major rows against dense ones."""
    rng = np.random.default_rng(3)
    H = 4
    par = [inputs.tree_chain(64), inputs.tree_frontier(40, rng), inputs.tree_chain(17),
           inputs.tree_frontier(1, rng), inputs.tree_frontier(64, rng)]
    forest = tv.forest_build(par, n_max=64).upload()
    N = int(forest.offsets[-1])
    t = _inputs(1, H, N, inputs.DELTA, "chain", inputs.F32)[3]
    S = inputs.make_tensors(inputs.workload("c4", B=len(par), H=H, T=1, seed=78))["S_pre"]
    dev = {n: t[n][0].cuda() for n in ("q", "k", "v", "alpha", "beta")}
    O, U = tv.tree_verify(forest, S.cuda(), *dev.values(), rule=tv.DELTA, want_U=True)
    forest.device_status()
    for b, p in enumerate(par):
        lo, hi = int(forest.offsets[b]), int(forest.offsets[b + 1])
        cut = {n: inputs.to_f64(t[n][:, :, lo:hi]) for n in dev}
        ver = orc.verify_batch(inputs.to_f64(S[b:b + 1]), *cut.values(), p[None], "delta")
        for h in range(H):
            assert pu.rel_l2_rows(inputs.to_f64(O[h, lo:hi]), ver[(0, h)][0]) <= 1e-5
            assert pu.rel_l2_rows(inputs.to_f64(U[h, lo:hi]), ver[(0, h)][1]) <= 1e-5
    for dtype, rule in ((inputs.F32, tv.GATED), (inputs.F32, tv.DELTA), (inputs.BF16, tv.DELTA)):
        wl, parents, _, t = _inputs(20, 10, 50, rule, "chain", dtype)
        x = {n: y.cuda() if y is not None else None for n, y in t.items()}
        x["q"], x["k"] = x["q"][:, ::2].contiguous(), x["k"][:, ::2].contiguous()
        tree = tv.tree_build(parents).upload()
        names = ("S_pre", "q", "k", "v", "alpha", "beta")
        dense = tv.tree_verify(tree, *[x[n] for n in names], rule=rule, want_U=True)
        token = lambda y: y if y is None else y.transpose(1, 2).contiguous().transpose(1, 2)
        moved = [x["S_pre"]] + [token(x[n]) for n in names[1:]]
        out = [token(torch.zeros_like(dense[0])) for _ in range(2)]
        tv.tree_verify(tree, *moved, rule=rule, O=out[0], U=out[1])
        assert torch.equal(out[0], dense[0]) and torch.equal(out[1], dense[1])


@pytest.mark.parametrize("what", ["q", "coefficients", "state and v", "v", "large q", "large state and v"])
@pytest.mark.parametrize("rule,dtype,T,tree", [(inputs.DELTA, inputs.F32, 64, "frontier"), (inputs.DELTA, inputs.F32, 50, "chain"),
                                               (inputs.GATED, inputs.F32, 64, "frontier"), (inputs.DELTA, inputs.BF16, 40, "chain")])
def test_numbers_near_the_ends_of_the_range(rule, dtype, T, tree, what):
    """The recurrence is linear in q and in (S_pre, v): a power of two on them is the same power on the outputs, and changes no
    other bit of any sum as long as its terms are normal numbers.  Results down here are some 2^-120; a last place lost
    to subnormal numbers is 2^-149, less than 2^-24 of a tensor's norm.  bf16 operands are used as they are: 2^-108 on
    q leaves their scores normal.  What passes 2^112 is worked out row by row in fp32: the tolerance per node."""
    wl, parents, accepted, tens = _inputs(10, 8, T, rule, tree, dtype)
    if what in ("coefficients", "v"):
        tens["S_pre"].zero_()
    up = {"q": -116, "coefficients": -116, "state and v": -114, "v": -114, "large q": 113, "large state and v": 113}[what]
    if dtype == inputs.BF16 and up == -116:
        up = -108
    if dtype == inputs.BF16:   # nothing that the power leaves with fewer than its 8 bits
        for n in ("q", "v"):
            tens[n] = tens[n] * (tens[n].abs() >= 2.0 ** -11)
    moved = dict(tens)
    for n in ("q",) if what in ("q", "coefficients", "large q") else ("S_pre", "v"):
        moved[n] = tens[n] * 2.0 ** up
        assert torch.isfinite(moved[n]).all()
    O0, U0 = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_AUTO)[:2]
    O, U, _, tree = pu.gpu_round(wl, parents, accepted, moved, impl=tv.IMPL_AUTO)
    tree.device_status()
    items = [(0, 0), (4, 3), (9, 7)]
    f = {n: inputs.to_f64(x) for n, x in moved.items()}
    ver = orc.verify_batch(f["S_pre"], f["q"], f["k"], f["v"], f["alpha"], f["beta"], parents, wl.rule_name, memo=True, items=items)
    by_q = what in ("q", "coefficients", "large q")
    for x, x0, which in ((O, O0, 0),) + (((U, U0, 1),) if rule == inputs.DELTA else ()):
        got, ref = (np.stack(y) for y in ([x[i] for i in items], [ver[i][which] for i in items]))
        assert pu.rel_l2_rows(got, ref) <= 1e-5
        if up < 0:
            assert pu.rel_fro(x, x0 * (1.0 if by_q and which else 2.0 ** up)) <= 2.0 ** -24


@pytest.mark.parametrize("what", ["v", "k", "alpha", "beta", "zero gate", "state"])
@pytest.mark.parametrize("rule", [inputs.GATED, inputs.DELTA])
@pytest.mark.parametrize("T,tree", [(50, "frontier"), (49, "chain")])
def test_values_that_are_not_finite(T, tree, rule, what):
    """They reach the rows that the recurrence takes them to -- a node's subtree, an entry of the state its value
    column -- and change no bit of any other row, whatever the coefficients between them."""
    if what == "beta" and rule == inputs.GATED:
        pytest.skip("no beta")
    wl, parents, accepted, tens = _inputs(20, 8, T, rule, tree, inputs.F32)
    bad = T // 3
    if what == "zero gate":
        tens["alpha"][3][:, torch.from_numpy(parents[3] == bad)] = 0.0
    run = lambda: pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_AUTO)[:2]
    O0, U0 = run()
    if what == "state":
        tens["S_pre"][3, 2, 5, 7] = float("inf")
    elif what == "zero gate":
        tens["v"][3, 2, bad] = float("nan")
    else:
        tens[what][3, 2, bad] = float("nan")
    O, U = run()
    hit = np.array([bad in orc.path_to(parents[3], i) for i in range(T)])
    O_is, U_is = np.ones_like(O, dtype=bool), np.ones_like(O, dtype=bool)   # where nothing may change
    if what == "state":
        O_is[3, 2, :, 5] = U_is[3, 2, :, 5] = False
        assert not np.isfinite(O[3, 2, :, 5]).any()
    else:
        O_is[3, 2, hit] = False
        U_is[3, 2, hit] = False
        if not (what == "k" and rule == inputs.GATED and hit.sum() == 1):
            assert np.isnan(O[3, 2, hit]).all()
    if what == "state":   # every row of the item is worked out again, in fp32
        np.testing.assert_allclose(O[3, 2][O_is[3, 2]], O0[3, 2][O_is[3, 2]], rtol=0, atol=1e-5 * np.abs(O0[3, 2]).max())
        O_is[3, 2] = U_is[3, 2] = False
    assert np.array_equal(O[O_is], O0[O_is])
    if rule == inputs.DELTA:
        assert np.array_equal(U[U_is], U0[U_is])


@pytest.mark.parametrize("B,H,T,tree,rule,dtype,dk,dv", [
    (6, 8, 64, "frontier", inputs.DELTA, inputs.F32, 128, 128),     # halves of the columns
    (4, 8, 40, "chain", inputs.DELTA, inputs.BF16, 64, 128),
    (20, 16, 40, "chain", inputs.DELTA, inputs.BF16, 128, 128),     # three items on a CTA
    (20, 16, 50, "frontier", inputs.DELTA, inputs.BF16, 64, 64),
    (20, 16, 64, "chain", inputs.DELTA, inputs.F32, 64, 128),
    (10, 8, 33, "frontier", inputs.DELTA, inputs.F32, 128, 64),
    (20, 16, 49, "frontier", inputs.GATED, inputs.F32, 128, 128),
    (20, 16, 64, "chain", inputs.GATED, inputs.BF16, 64, 128),
    (20, 16, 64, "frontier", inputs.GATED, inputs.BF16, 128, 64),
])
def test_values_that_are_not_finite_on_every_variant(B, H, T, tree, rule, dtype, dk, dv):
    """In the first and the last item of a CTA, single entries left and right: what they reach and what comes out elsewhere are
    the general kernel's, whose sums run over a node's own path; rows that they do not reach keep every bit."""
    wl, parents, accepted, tens = _inputs(B, H, T, rule, tree, dtype, dk=dk, dv=dv)
    clean = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_AUTO)[:2]
    last = (B * H - 1) // 148 * 148
    items = sorted({(i // H, i % H) for i in (0, 1, 2, last, last + 1)})
    bad = T // 3
    tens["v"][items[0]][bad, dv - 1] = float("nan")
    tens["k"][items[1]][bad, 5] = float("inf")
    tens["S_pre"][items[2]][dv - 2, 3] = float("inf")
    for b, h in items[3:]:
        tens["alpha"][b, h, bad] = float("nan")
        tens["v"][b, h, 0, 1] = float("-inf")
    got = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_AUTO)[:2]
    ref = pu.gpu_round(wl, parents, accepted, tens, impl=tv.IMPL_SIMT)[:2]
    for x, y, c in list(zip(got, ref, clean))[:2 if rule == inputs.DELTA else 1]:
        assert np.array_equal(np.isfinite(x), np.isfinite(y))
        rest = np.ones((B, H), dtype=bool)
        for i in items:
            rest[i] = False
            ok = np.isfinite(y[i])
            assert not ok.all()
            np.testing.assert_allclose(x[i][ok], y[i][ok], rtol=0, atol=1e-5 * np.abs(y[i][ok]).max())
        assert np.array_equal(x[rest], c[rest])


def test_a_poisoned_request_does_not_hold_up_the_batch():
    """Items that hold such values are worked out a second time, in fp32: some four times what the general kernel takes."""
    wl, parents, _, tens = _inputs(8, 16, 63, inputs.DELTA, "frontier", inputs.F32)
    tens["S_pre"][3] = float("nan")
    t = {n: x.cuda() for n, x in tens.items()}
    tree = tv.tree_build(parents).upload()
    O, U = torch.empty_like(t["v"]), torch.empty_like(t["v"])
    us = {}
    for impl in (tv.IMPL_SIMT, tv.IMPL_AUTO):
        call = lambda: tv.tree_verify(tree, *[t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")], rule=tv.DELTA, O=O, U=U, impl=impl)
        us[impl] = pu.device_us(call)
    assert us[tv.IMPL_AUTO] <= 8 * us[tv.IMPL_SIMT], us
