"""Calls whose form (shapes, strides, types) was seen before: same results, same refusals."""
import dataclasses

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
    for x in (args, strided, args, strided):          # alternating forms, new buffers each time
        O, U = tv.tree_verify(tree, *[y.clone(memory_format=torch.preserve_format) for y in x], rule=tv.DELTA, want_U=True)
        assert torch.equal(O, first[0]) and torch.equal(U, first[1])
        Sn = tv.commit_path(tree, acc, x[0], *x[2:], rule=tv.DELTA, U=first[1], S_new=torch.empty_like(x[0]))
        assert torch.isfinite(Sn).all()
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
