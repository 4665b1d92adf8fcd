"""The calls of a step through the CPython module: the same results whether outputs are given or
allocated and whichever form the descriptors come in, and the same errors as the checks in Python."""
import numpy as np
import pytest
import torch

from paper_2602_24082_b200 import workloads as W

pytestmark = pytest.mark.gpu

W1 = W.Workload("binding", [[(70, (33, 5))], [(9, (140,))]], 4, 2, 64, seed=3)


def _inputs():
    from paper_2602_24082_b200 import binding as B
    return B, B.plan_for(W1), [x.cuda() for x in W1.tensors()]


@pytest.mark.parametrize("form", [tuple, list, lambda d: [a.astype(np.int64) for a in d],
                                  lambda d: [a.tolist() for a in d],
                                  lambda d: [np.repeat(a, 2)[::2] for a in d]],
                         ids=["tuple", "list", "int64", "lists", "strided"])
def test_descriptor_forms_give_the_same_plan(form):
    from paper_2602_24082_b200 import binding as B
    want = B.plan_for(W1)
    got = B.pp_build_plan(form(W1.descriptors()), 4, 2, 64, W1.total_tokens,
                          workspace=torch.empty(want.plan_bytes, dtype=torch.uint8, device="cuda"))
    assert got.status() == (0, 0) and got.problem.num_responses == 3
    nb = len(want.read_bwd_tiles())
    (tiles, fwd_order, bwd_order, key_end), expected = got.read(), want.read()
    for a, b in zip((tiles, fwd_order, bwd_order[:nb], key_end), (*expected[:2], expected[2][:nb], expected[3])):
        assert np.array_equal(a, b)              # (bwd_order is valid up to the backward's tiles)
    assert np.array_equal(got.read_bwd_tiles(), want.read_bwd_tiles())


def test_given_and_allocated_outputs_agree():
    B, plan, (q, k, v, do) = _inputs()
    o, lse = B.pp_attn_fwd(plan, q, k, v, 0.125)
    o2, lse2 = torch.full_like(o, 7.0), torch.full_like(lse, 7.0)
    r = B.pp_attn_fwd(plan, q, k, v, 0.125, o=o2, lse=lse2)
    assert r[0].data_ptr() == o2.data_ptr() and torch.equal(o, o2) and torch.equal(lse, lse2)
    a = B.pp_attn_bwd(plan, q, k, v, o, lse, do, 0.125)
    out = [torch.full_like(x, 7.0) for x in a]
    b = B.pp_attn_bwd(plan, q, k, v, o, lse, do, 0.125, *out)
    assert [x.data_ptr() for x in b] == [x.data_ptr() for x in out]
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert [x.shape for x in a] == [q.shape, k.shape, v.shape] and all(not x.requires_grad for x in a)


@pytest.mark.parametrize("what,bad", [("q", lambda t: t.float()), ("k", lambda t: t[:-1]), ("v", lambda t: t.cpu()),
                                      ("q", lambda t: t.transpose(0, 1).contiguous().transpose(0, 1))],
                         ids=["type", "shape", "cpu", "strides"])
def test_unsuitable_tensors_are_refused(what, bad):
    B, plan, (q, k, v, do) = _inputs()
    args = {"q": q, "k": k, "v": v}
    args[what] = bad(args[what])
    with pytest.raises(ValueError, match=f"^{what}: expected contiguous CUDA"):
        B.pp_attn_fwd(plan, args["q"], args["k"], args["v"], 0.125)
    o, lse = B.pp_attn_fwd(plan, q, k, v, 0.125)
    with pytest.raises(ValueError, match=f"^{what}: expected contiguous CUDA"):
        B.pp_attn_bwd(plan, args["q"], args["k"], args["v"], o, lse, do, 0.125)


@pytest.mark.parametrize("bad", [lambda t: t.float(), lambda t: t[:-1].contiguous(), lambda t: t[:, :1].contiguous(),
                                 lambda t: t.cpu(), lambda t: t.transpose(0, 1).contiguous().transpose(0, 1),
                                 lambda t: t.float().cpu().numpy()],
                         ids=["type", "tokens", "heads", "cpu", "strides", "array"])
def test_unsuitable_outputs_are_refused(bad):
    """Before anything is launched: no gradient changes."""
    B, plan, (q, k, v, do) = _inputs()
    o, lse = B.pp_attn_fwd(plan, q, k, v, 0.125)
    with pytest.raises(ValueError, match="^o: expected contiguous CUDA"):
        B.pp_attn_fwd(plan, q, k, v, 0.125, o=bad(o))
    out = {n: torch.full_like(t, 7.0) for n, t in (("d_q", q), ("d_k", k), ("d_v", v))}
    for n, t in out.items():
        with pytest.raises(ValueError, match=f"^{n}: expected contiguous CUDA"):
            B.pp_attn_bwd(plan, q, k, v, o, lse, do, 0.125, **{**out, n: bad(t)})
    assert all(bool((t == 7.0).all()) for t in out.values())


@pytest.mark.parametrize("bad", [lambda t: t.cpu(), lambda t: t[:1].expand(t.numel()), lambda t: t.cpu().numpy()],
                         ids=["cpu", "strides", "array"])
def test_unsuitable_buffers_are_refused(bad):
    B, plan, (q, k, v, do) = _inputs()
    o, lse = B.pp_attn_fwd(plan, q, k, v, 0.125)
    plan._bwd_scratch = bad(plan.bwd_scratch())
    with pytest.raises(ValueError, match="^scratch: expected a contiguous CUDA"):
        B.pp_attn_fwd(plan, q, k, v, 0.125, for_backward=True)
    with pytest.raises(ValueError, match="^scratch: expected a contiguous CUDA"):
        B.pp_attn_bwd(plan, q, k, v, o, lse, do, 0.125)
    for desc in (W1.descriptors(), [a.tolist() for a in W1.descriptors()]):
        with pytest.raises((ValueError, AttributeError)):
            B.pp_build_plan(desc, 4, 2, 64, W1.total_tokens, workspace=bad(plan.workspace))


def test_library_errors_are_raised():
    B, plan, (q, k, v, do) = _inputs()
    with pytest.raises(B.PPError) as e:
        B.pp_attn_fwd(plan, q, k, v, -1.0)
    assert e.value.code == -1
    with pytest.raises(ValueError, match="too small"):
        B.pp_build_plan(W1.descriptors(), 4, 2, 64, W1.total_tokens, workspace=plan.workspace[:64])
    with pytest.raises(B.PPError) as e:
        B.pp_build_plan(W1.descriptors(), 4, 2, 64, W1.total_tokens + 1, workspace=plan.workspace)
    assert e.value.code == -1
    with pytest.raises(ValueError, match="CUDA"):
        B.pp_build_plan(W1.descriptors(), 4, 2, 64, W1.total_tokens, workspace=plan.workspace.cpu())
