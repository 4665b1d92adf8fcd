"""Forward with two query tiles of a segment in a unit's slots (an odd number of query heads per KV head, more
units than SMs): each row's arithmetic is that of a unit with one tile, so a head of a large problem
has the bits it has alone, where there are too few units for it."""
import pytest
import torch

from paper_2602_24082_b200 import workloads as W

pytestmark = pytest.mark.gpu

ROWS = [[(257, (5, 128, 31)), (1, (1, 385))], [(128, (256, 129))], [(384, (640,)), (130, (127, 512))]]


def _run(w, tens, clear):
    from paper_2602_24082_b200 import binding as B
    plan = B.plan_for(w)
    if clear:
        plan.bwd_scratch().fill_(0xFF)
    o, lse = B.pp_attn_fwd(plan, *tens[:3], w.softmax_scale, for_backward=clear)
    grads = B.pp_attn_bwd(plan, *tens[:3], o, lse, tens[3], w.softmax_scale) if clear else ()
    torch.cuda.synchronize()
    assert plan.status() == (0, 0)
    return (o, lse) + tuple(grads)


@pytest.mark.parametrize("hq,hkv", [(12, 12), (21, 7), (42, 6)])
@pytest.mark.parametrize("d", [64, 96, 128])
def test_a_head_has_the_bits_it_has_alone(hq, hkv, d):
    w = W.Workload("paired", ROWS, hq, hkv, d, seed=hq)
    # more units than SMs, also without the mixed tiles that many short segments would bring
    tiles = sum((p + 127) // 128 + sum((r + 127) // 128 for r in rs) for row in ROWS for p, rs in row)
    assert tiles * hkv * ((hq // hkv + 1) // 2) > 148
    tens = [x.cuda() for x in w.tensors()]
    o, lse, dq, _, _ = _run(w, tens, clear=True)
    assert torch.isfinite(dq).all()      # (a row of the accumulator that was not cleared would show)
    r = hq // hkv
    for h in (0, r - 1, hq // 2, hq - 1):
        one = W.Workload("alone", ROWS, 1, 1, d, seed=0)
        kv = h // r
        part = [tens[0][:, h:h + 1].contiguous(), tens[1][:, kv:kv + 1].contiguous(),
                tens[2][:, kv:kv + 1].contiguous()]
        o1, lse1 = _run(one, part, clear=False)
        assert torch.equal(o[:, h], o1[:, 0]) and torch.equal(lse[h], lse1[0])
