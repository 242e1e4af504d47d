"""Whole rounds queued on one stream without any synchronisation: upload -> Stage 1 -> verify ->
commit, twice over, every kernel a dependent launch of the one in front of it.  The results must be
bit for bit those of the same calls issued one at a time with a device synchronisation after each:
a kernel that read an input before the kernel producing it had finished, or wrote a buffer that an
older kernel was still reading, would show up as a difference."""
import numpy as np
import pytest
import torch

import paper_2608_01651_b200 as tv
from paper_2608_01651_b200 import inputs
from tests import parity_util as pu

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _round_calls(wl, rule, impl):
    parents, accepted = inputs.make_trees(wl)
    tree = tv.tree_build(parents)
    acc = torch.from_numpy(np.asarray(accepted, dtype=np.int32)).to(DEV)
    B, H, T, dk, dv = wl.B, wl.H, wl.T, wl.dk, wl.dv
    ci = [{k: v.to(DEV) for k, v in inputs.make_conv_inputs(wl, layer=r, device="cpu").items()} for r in range(2)]
    S0 = inputs.make_tensors(wl)["S_pre"].to(DEV)
    delta = rule == tv.DELTA

    def run(sync):
        S = S0.clone()
        ctx = [c["ctx"].clone() for c in ci]
        outs = []
        torch.cuda.synchronize()
        pause = torch.cuda.synchronize if sync else (lambda: None)
        for r in range(2):
            c = ci[r]
            tree.upload(); pause()
            q, k, v, al, be = tv.tree_conv(tree, c["x"], ctx[r], c["weight"], c["bias"], H=H, dk=dk, dv=dv,
                                           gate_a=c["gate_a"], gate_b=c["gate_b"], A_log=c["A_log"],
                                           dt_bias=c["dt_bias"], normalize_qk=True)
            pause()
            O = torch.empty(B, H, T, dv, device=DEV)
            U = torch.empty_like(O) if delta else None
            tv.tree_verify(tree, S, q, k, v, al, be if delta else None, rule=rule, O=O, U=U, impl=impl)
            pause()
            tv.commit_path(tree, acc, S, k, v, al, be if delta else None, rule=rule, U=U)   # in place
            pause()
            tv.conv_commit(tree, acc, c["x"], ctx[r], H=H, dk=dk, dv=dv)                      # in place
            pause()
            outs.append((q, k, v, al, be, O, U))
        torch.cuda.synchronize()
        tree.device_status()
        return S, ctx, outs

    return run


@pytest.mark.parametrize("name,B,H,T,rule,impl", [
    ("c3", 32, 32, 64, tv.GATED, tv.IMPL_AUTO),
    ("c3", 6, 8, 40, tv.GATED, tv.IMPL_AUTO),
    ("c4", 16, 32, 64, tv.DELTA, tv.IMPL_AUTO),
    ("c5", 24, 16, 128, tv.GATED, tv.IMPL_AUTO),
    ("c3", 5, 4, 33, tv.GATED, tv.IMPL_SIMT),
])
def test_unsynchronised_rounds_equal_synchronised_ones(name, B, H, T, rule, impl):
    wl = inputs.workload(name, B=B, H=H, T=T, L=1, seed=1234 + T)
    run = _round_calls(wl, rule, impl)
    S_ref, ctx_ref, outs_ref = run(sync=True)
    assert torch.isfinite(S_ref).all()
    for rep in range(3):
        S, ctx, outs = run(sync=False)
        assert torch.equal(S, S_ref), f"state differs (repeat {rep})"
        for a, b in zip(ctx, ctx_ref):
            assert torch.equal(a, b), f"context rows differ (repeat {rep})"
        for r, (got, ref) in enumerate(zip(outs, outs_ref)):
            for i, (x, y) in enumerate(zip(got, ref)):
                if y is None:
                    assert x is None
                else:
                    assert torch.equal(x, y), f"round {r}, output {i} differs (repeat {rep})"


@pytest.mark.parametrize("rule", [tv.GATED, tv.DELTA])
@pytest.mark.parametrize("d,T,impl", [(64, 64, tv.IMPL_SIMT), (128, 64, tv.IMPL_SIMT), (64, 128, tv.IMPL_SIMT), (128, 128, tv.IMPL_SIMT),
                                      (64, 64, tv.IMPL_AUTO), (128, 64, tv.IMPL_AUTO)])
def test_commit_that_rejects_every_request_keeps_the_order(d, T, impl, rule):
    """verify -> in-place commit in which no request accepts anything -> other trees -> verify, queued
    without synchronisation.  The commit has nothing to do, and must still not end before the verify in
    front of it: the upload behind it waits for the commit only and then overwrites the masks."""
    wl = inputs.workload("c4", B=12, H=16, T=T, dk=d, dv=d, rule=rule, qkv_dtype=inputs.F32, seed=T + d)
    t = {n: None if x is None else x.to(DEV) for n, x in inputs.make_tensors(wl).items()}
    t["k"] = t["k"] * (8.0 / d ** 0.5)
    trees = [inputs.make_trees(wl)[0], np.stack([inputs.tree_chain(T)] * wl.B)]
    none = torch.full((wl.B,), -1, dtype=torch.int32, device=DEV)
    tree = tv.tree_build(trees[0])

    def run(sync):
        pause = torch.cuda.synchronize if sync else (lambda: None)
        S = t["S_pre"].clone()
        outs = [torch.zeros(wl.B, wl.H, T, d, device=DEV) for _ in range(4)]
        torch.cuda.synchronize()
        for r in range(2):
            tree.rebuild(trees[r]).upload(); pause()
            tv.tree_verify(tree, S, t["q"], t["k"], t["v"], t["alpha"], t["beta"], rule=rule, O=outs[2 * r],
                           U=outs[2 * r + 1], impl=impl); pause()
            tv.commit_path(tree, none, S, t["k"], t["v"], t["alpha"], t["beta"], rule=rule, U=outs[2 * r + 1]); pause()
        tree.rebuild(trees[0]).upload()      # over the masks of the last verify
        torch.cuda.synchronize()
        return [S] + outs

    ref = run(sync=True)
    assert torch.equal(ref[0], t["S_pre"]) and torch.isfinite(ref[3]).all()
    for rep in range(3):
        for i, (x, y) in enumerate(zip(run(sync=False), ref)):
            assert torch.equal(x, y), (rep, i)


def _compare(run):
    S_ref, ctx_ref, outs_ref = run(sync=True)
    assert torch.isfinite(S_ref).all()
    for rep in range(3):
        S, ctx, outs = run(sync=False)
        assert torch.equal(S, S_ref), rep
        assert all(torch.equal(a, b) for a, b in zip(ctx, ctx_ref)), rep
        for r, (got, ref) in enumerate(zip(outs, outs_ref)):
            for i, (x, y) in enumerate(zip(got, ref)):
                assert (x is None and y is None) or torch.equal(x, y), (rep, r, i)


@pytest.mark.parametrize("rule", [tv.GATED, tv.DELTA])
@pytest.mark.parametrize("tree,T,d,dtype,B,H", [
    ("frontier", 63, 128, inputs.F32, 9, 16),     # path form, whole columns
    ("frontier", 40, 64, inputs.F32, 5, 8),       # 64-wide states: column chunks, the commit kernel of dk = 64
    ("chain", 40, 128, inputs.BF16, 9, 16),       # block form
    ("chain", 40, 64, inputs.F32, 12, 16),
    ("frontier", 100, 128, inputs.F32, 6, 16),    # two row blocks, path form
    ("chain", 128, 128, inputs.BF16, 6, 16),      # two row blocks, block form: its second block is loaded late
    ("chain", 90, 64, inputs.F32, 6, 16),
])
def test_queued_rounds_of_the_general_kernel(tree, T, d, dtype, B, H, rule):
    """The fp32 kernel asks for the state before its wait, and so does the commit behind it."""
    wl = inputs.workload("c4", B=B, H=H, T=T, dk=d, dv=d, tree=tree, qkv_dtype=dtype, rule=rule, seed=T + d)
    _compare(_round_calls(wl, rule, tv.IMPL_SIMT))


@pytest.mark.parametrize("tree,T,dk,dv,dtype,B,H,rule", [
    ("frontier", 63, 128, 128, inputs.F32, 9, 16, tv.DELTA),     # path form, whole columns
    ("frontier", 63, 128, 128, inputs.F32, 16, 16, tv.DELTA),    # two items on a CTA
    ("frontier", 40, 128, 128, inputs.F32, 4, 16, tv.DELTA),     # halves
    ("chain", 40, 128, 128, inputs.BF16, 9, 16, tv.DELTA),       # block form; the state goes to registers before the wait
    ("chain", 40, 128, 128, inputs.BF16, 28, 16, tv.DELTA),      # four items on a CTA
    ("chain", 24, 128, 128, inputs.BF16, 4, 8, tv.DELTA),
    ("chain", 50, 64, 64, inputs.F32, 12, 16, tv.DELTA),
    ("chain", 40, 64, 64, inputs.BF16, 12, 16, tv.DELTA),
    ("frontier", 64, 64, 128, inputs.BF16, 12, 16, tv.DELTA),
    ("frontier", 63, 128, 128, inputs.F32, 12, 16, tv.GATED),
    ("chain", 64, 64, 128, inputs.BF16, 12, 16, tv.GATED),
])
def test_queued_rounds_of_the_kernel_of_fp32_accuracy(tree, T, dk, dv, dtype, B, H, rule):
    """It asks for the state before its wait and releases the commit behind it at once, and runs between an in-place commit
    and an upload that overwrites its masks."""
    wl = inputs.workload("c4", B=B, H=H, T=T, dk=dk, dv=dv, tree=tree, qkv_dtype=dtype, rule=rule, seed=T + dk)
    t = {n: None if x is None else x.to(DEV) for n, x in inputs.make_tensors(wl).items()}
    trees = tv.tree_build(inputs.make_trees(wl)[0]).upload()
    O = torch.empty(B, H, T, dv, device=DEV)
    (name, _), = pu.kernels_of(lambda: tv.tree_verify(trees, *[t[n] for n in ("S_pre", "q", "k", "v", "alpha", "beta")], rule=rule, O=O))
    assert "verify_exact_kernel" in name
    _compare(_round_calls(wl, rule, tv.IMPL_AUTO))


@pytest.mark.parametrize("B,Tc,rule,dtype", [
    (32, 64, tv.GATED, inputs.BF16),    # 2048 candidates
    (32, 64, tv.DELTA, inputs.BF16),
    (24, 100, tv.DELTA, inputs.F32),    # 2400, general verify kernel
    (24, 60, tv.DELTA, inputs.F32),     # the verify kernel of fp32 accuracy
    (100, 90, tv.GATED, inputs.BF16),   # 9000
    (700, 3, tv.GATED, inputs.F32),     # many small requests
])
def test_queued_rounds_with_selection(B, Tc, rule, dtype):
    """selection -> metadata from device memory -> verify -> commit in place, twice, with other candidates
    the second time: the keys, the packed parents and the masks of one round are overwritten by the next."""
    H, d, N = 4, 128, max(B, B * Tc * 6 // 10)
    wl = inputs.workload("c4", B=1, H=H, T=N, rule=rule, qkv_dtype=dtype, seed=7)
    rng = np.random.default_rng(B)
    par = [torch.from_numpy(np.stack([inputs.tree_frontier(Tc, rng) for _ in range(B)])).to(DEV) for _ in range(2)]
    p = [torch.from_numpy(rng.uniform(0.1, 1.0, (B, Tc)).astype(np.float32)).to(DEV) for _ in range(2)]
    t = {n: None if x is None else x[0].to(DEV) for n, x in inputs.make_tensors(wl).items()}
    if dtype == inputs.F32:
        t["k"] = t["k"] * (8.0 / d ** 0.5)
    S0 = inputs.make_tensors(inputs.workload("c4", B=B, H=H, T=1, seed=8))["S_pre"].to(DEV)
    acc = torch.zeros(B, dtype=torch.int32, device=DEV)      # the root: every request keeps it
    forest = tv.forest_build([np.array([-1], dtype=np.int32)] * B, n_max=Tc, capacity=N)
    sel = tv.budget_select(par[0], p[0], N)

    def run(sync):
        pause = torch.cuda.synchronize if sync else (lambda: None)
        S = S0.clone()
        outs = [(torch.zeros(H, N, d, device=DEV), torch.zeros(H, N, d, device=DEV)) for _ in range(2)]
        torch.cuda.synchronize()
        for r in range(2):
            O, U = outs[r]
            tv.budget_select(par[r], p[r], N, out=sel); pause()
            forest.upload_device(sel["parent_packed"], sel["offsets"], max_depth_bound=min(8, Tc - 1)); pause()
            tv.tree_verify(forest, S, t["q"], t["k"], t["v"], t["alpha"], t["beta"], rule=rule, O=O, U=U); pause()
            tv.commit_path(forest, acc, S, t["k"], t["v"], t["alpha"], t["beta"], rule=rule, U=U); pause()
        torch.cuda.synchronize()
        forest.device_status()
        return S, [], outs

    _compare(run)
