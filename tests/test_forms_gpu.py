"""Calls whose form (shapes, strides, types) was seen before: same results, same refusals."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs

pytestmark = pytest.mark.gpu


def _token_major(x, dims):
    h = x.dim() - dims + 1
    return x.transpose(h, h + 1).contiguous().transpose(h, h + 1)


def test_repeated_forms_agree_and_refuse_as_before():
    wl = dataclasses.replace(inputs.workload("c4"), B=3, H=4, T=20, seed=9)
    parents, accepted = inputs.make_trees(wl)
    t = inputs.make_tensors(wl, device="cuda")
    tree = tv.tree_build(parents).upload()
    acc = torch.from_numpy(accepted).cuda()
    args = [t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")]
    strided = [t["S_pre"]] + [_token_major(t[n], 4) for n in ("q", "k", "v")] + [_token_major(t[n], 3) for n in ("alpha", "beta")]
    first = tv.tree_verify(tree, *args, rule=tv.DELTA, want_U=True)
    first_S = tv.commit_path(tree, acc, args[0], *args[2:], rule=tv.DELTA, U=first[1], S_new=torch.empty_like(args[0]))
    for x in (args, strided, args, strided):          # alternating forms, new buffers each time
        O, U = tv.tree_verify(tree, *[y.clone(memory_format=torch.preserve_format) for y in x], rule=tv.DELTA, want_U=True)
        assert torch.equal(O, first[0]) and torch.equal(U, first[1])
        Sn = tv.commit_path(tree, acc, x[0], *x[2:], rule=tv.DELTA, U=first[1], S_new=torch.empty_like(x[0]))
        assert torch.equal(Sn, first_S)
    S, q, k, v, al, be = args
    O, U = first
    bad = [(S.double(), q, k, v, al, be), (S, q.float(), k, v, al, be), (S, q, k, v, al.bfloat16(), be),
           (S, strided[1], k, v, al, be), (S, q, k, v, strided[4], be), (S.cpu(), q, k, v, al, be),
           (S.transpose(-1, -2), q, k, v, al, be), (S, q, k[..., ::2], v, al, be)]
    for _ in range(2):
        for x in bad:
            with pytest.raises(ValueError):
                tv.tree_verify(tree, *x, rule=tv.DELTA, O=O, U=U)
        with pytest.raises(ValueError):
            tv.tree_verify(tree, *args, rule=tv.DELTA, O=O.double(), U=U)
        with pytest.raises(ValueError):
            tv.tree_verify(tree, *args, rule=tv.DELTA, O=O, U=_token_major(U, 4))
        with pytest.raises(ValueError):
            tv.commit_path(tree, acc.long(), S, k, v, al, be, rule=tv.DELTA, U=U)
        with pytest.raises(tv.TreeVerifyError):       # a form that passes here, refused by the library
            tv.tree_verify(tree, *args, rule=7, O=O, U=U)
        other = tv.tree_build(parents[:, :10]).upload()
        with pytest.raises(tv.TreeVerifyError):
            tv.tree_verify(other, *args, rule=tv.DELTA, O=O, U=U)
        with pytest.raises(TypeError):
            tv.tree_verify(tree, *args, rule=1.0, O=O, U=U)



def test_front_end_values_are_read_anew():
    # sizes and switches of one element that are not plain numbers: their value counts, in every call
    wl = dataclasses.replace(inputs.workload("c4"), B=2, H=2, T=12, seed=4)
    parents, _ = inputs.make_trees(wl)
    g = {n: x.cuda() for n, x in inputs.make_conv_inputs(wl, device="cpu", W=4).items()}
    tree = tv.tree_build(parents).upload()

    def conv(**kw):
        return tv.tree_conv(tree, g["x"], g["ctx"], g["weight"], g["bias"], H=2, dk=128, dv=128, **kw)[:2]

    eps, norm = torch.tensor(1e-6), torch.tensor(True)
    for value, on in ((1e-6, True), (3.0, True), (3.0, False), (1e-6, True)):
        eps.fill_(value)
        norm.fill_(on)
        want = conv(eps=value, normalize_qk=on)
        for e, n in ((eps, norm), (np.array(value), np.array(on)), (np.float64(value), int(on))):
            got = conv(eps=e, normalize_qk=n)
            assert all(torch.equal(a, b) for a, b in zip(got, want)), (value, on)
    a, b = conv(eps=1e-6, normalize_qk=True), conv(eps=3.0, normalize_qk=True)
    assert not torch.equal(a[0], b[0])


def test_refused_inputs_allocate_no_outputs():
    wl = dataclasses.replace(inputs.workload("c4"), B=2, H=2, T=12, seed=4)
    parents, _ = inputs.make_trees(wl)
    t = inputs.make_tensors(wl, device="cuda")
    tree = tv.tree_build(parents).upload()
    args = [t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")]
    tv.tree_verify(tree, *args, rule=tv.DELTA)
    torch.cuda.synchronize()
    for bad in ([args[0].double()] + args[1:], args[:3] + [t["v"].cpu()] + args[4:], args[:1] + [t["q"].float()] + args[2:]):
        held = torch.cuda.memory_allocated()
        torch.cuda.reset_peak_memory_stats()
        with pytest.raises(ValueError):
            tv.tree_verify(tree, *bad, rule=tv.DELTA, want_U=True)
        assert torch.cuda.max_memory_allocated() == held


def test_other_calls_repeat_and_refuse_by_form():
    # alternating forms of the calls without strides: every result as from a table that holds nothing
    wls = [dataclasses.replace(inputs.workload("c4"), B=B, H=2, T=T, seed=T) for B, T in ((3, 12), (2, 12), (3, 13))]
    cases = []
    for i, wl in enumerate(wls):
        parents, accepted = inputs.make_trees(wl)
        t = inputs.make_tensors(wl, device="cuda")
        W = 4 if i else 3
        g = {n: x.cuda() for n, x in inputs.make_conv_inputs(wl, device="cpu", W=W).items()}
        cases.append((wl, tv.tree_build(parents).upload(), torch.from_numpy(parents).cuda(), torch.from_numpy(accepted).cuda(), t, g))

    def calls(case, one_tree, norm, eps):
        wl, tree, par, acc, t, g = case
        args = [t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")]
        O = torch.zeros(wl.B, wl.H, wl.T, 128, device="cuda")
        U = torch.zeros_like(O)
        tv.tree_verify_static(par[0] if one_tree else par, *args, rule=tv.DELTA, O=O, U=U)
        dims = dict(H=wl.H, dk=128, dv=128)
        y = tv.tree_conv(tree, g["x"], g["ctx"], g["weight"], g["bias"], gate_a=g["gate_a"], gate_b=g["gate_b"],
                         A_log=g["A_log"], dt_bias=g["dt_bias"], normalize_qk=norm, eps=eps, **dims)
        ctx = tv.conv_commit(tree, acc, g["x"], g["ctx"], ctx_new=torch.zeros_like(g["ctx"]), **dims)
        return [O, U, *y, ctx]

    variants = [(c, one, norm, eps) for c in cases for one in (False, True) for norm, eps in ((True, 1e-6), (True, 0.5), (False, 1e-6))]
    want = []
    for v in variants:
        tv._forms.clear()
        want.append(calls(*v))
    for v, w in list(zip(variants, want)) * 2:
        assert all(torch.equal(a, b) for a, b in zip(calls(*v), w))
    # a neighbour of an accepted form is refused, before and after
    wl, tree, par, acc, t, g = cases[0]
    args = [t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")]
    O = torch.zeros(wl.B, wl.H, wl.T, 128, device="cuda")
    for _ in range(2):
        for bad in (par[:2], par[:, :-1].contiguous(), par.long(), par.t().contiguous(), par.cpu()):
            with pytest.raises(ValueError):
                tv.tree_verify_static(bad, *args, rule=tv.DELTA, O=O)
        with pytest.raises(ValueError):
            tv.tree_verify_static(par, *args, rule=tv.DELTA, O=O.transpose(1, 2).contiguous().transpose(1, 2))
        with pytest.raises(ValueError):
            tv.tree_conv(tree, g["x"], g["ctx"][:, :-1].contiguous(), g["weight"], H=wl.H, dk=128, dv=128)
        with pytest.raises(ValueError):
            tv.tree_conv(tree, g["x"], g["ctx"], g["weight"], H=wl.H, dk=64, dv=128)
        with pytest.raises(ValueError):
            tv.conv_commit(tree, acc.long(), g["x"], g["ctx"], H=wl.H, dk=128, dv=128)
        with pytest.raises(ValueError):
            tv.conv_commit(tree, acc, g["x"], g["ctx"], H=wl.H + 1, dk=128, dv=128)


def test_more_forms_than_the_table_keeps():
    S = torch.randn(4, 2, 128, 128, device="cuda") * 0.05
    rows = {n: (torch.randn(4, 2, 128, 128, device="cuda") / 8).bfloat16() for n in ("q", "k", "v")}
    gates = torch.rand(2, 4, 2, 128, device="cuda")
    trees = {}

    def verify(B, T):
        if (B, T) not in trees:
            trees[B, T] = tv.tree_build(np.tile(np.concatenate([[-1], np.arange(T - 1) // 2]).astype(np.int32), (B, 1))).upload()
        cut = lambda x: x[:B, :, :T].contiguous()
        return tv.tree_verify(trees[B, T], S[:B], *[cut(rows[n]) for n in ("q", "k", "v")], cut(gates[0]), cut(gates[1]),
                              rule=tv.DELTA)

    sizes = [(B, T) for T in range(1, 129) for B in (1, 2, 4)]
    assert len(sizes) > tv._FORMS_KEPT
    first = [verify(*s) for s in sizes]
    assert len(tv._forms) <= tv._FORMS_KEPT
    for s, x in zip(sizes, first):
        assert torch.equal(verify(*s), x)
