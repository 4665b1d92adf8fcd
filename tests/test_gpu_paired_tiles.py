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


def _units(w):
    from paper_2602_24082_b200 import binding as B
    plan = B.plan_for(w)
    assert plan.status() == (0, 0)
    return plan.read_fwd_units(len(plan.read()[0]))


def _split(length, n, ratio):
    r = max(1, length // (n + ratio))
    return (length - n * r, (r,) * n)


@pytest.mark.parametrize("lens,hq,hkv,d,some_alone", [
    ([6000] + [600] * 30, 3, 3, 64, True),
    ([8000, 4000, 4000] + [500] * 20, 3, 3, 64, True),
    ([14384] + [600] * 40, 2, 2, 128, True), ([14384] + [600] * 40, 8, 8, 96, False),
    ([20000] + [300] * 100, 1, 1, 128, True),          # (more than 512 tiles: ordered by sorting)
    ([30000] + [(120, (100,))] * 800, 1, 1, 128, True),        # (more than 2048: several kernels)
    ([3000] * 4, 16, 16, 128, False), ([2600] * 5, 21, 3, 64, False)])
def test_which_tiles_share_a_unit(lens, hq, hkv, d, some_alone):
    """By twos from a segment's start, but each alone where the two would take longer than an SM's share of the
    forward: 1.4 (head_dim 64: 1.6) times a tile's key tiles, as much as two heads of a tile take."""
    w = W.Workload("which", [[x if isinstance(x, tuple) else _split(x, 2, 2)] for x in lens], hq, hkv, d, seed=1)
    from paper_2602_24082_b200 import binding as B
    plan = B.plan_for(w)
    assert plan.status() == (0, 0)
    tiles = plan.read()[0]
    mode, units = plan.read_fwd_units(len(tiles))
    assert mode == 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    start, work = tiles[:, 0].tolist(), tiles[:, 7].tolist()
    cost = 16 if d == 64 else 14
    share = hkv * sum(work) * (10 + cost * (hq // hkv // 2))   # tenths of a key tile, of all SMs
    segments = {s: (n + 127) // 128 for s, n, *_ in w.segments()}
    expect, t = [], 0
    for s in sorted(segments):
        assert start[t] == s
        for i in range(segments[s]):
            two = i % 2 == 1 or i + 1 < segments[s]
            longer = work[t + i] if i % 2 else work[t + i] + 1
            expect.append(1 if not two or cost * sms * longer > share else 2 if i % 2 else 0)
        t += segments[s]
    assert units.tolist() == expect
    by_twos = [2 if i % 2 else 1 if i + 1 == segments[s] else 0 for s in sorted(segments) for i in range(segments[s])]
    assert (expect != by_twos) == some_alone and 2 in expect


def test_uneven_batches_keep_their_bits():
    """Pairs and single tiles side by side in a segment: each head has the bits it has alone."""
    w = W.Workload("uneven", [[_split(x, 2, 2)] for x in [2600] + [400] * 12], 7, 7, 64, seed=3)
    mode, units = _units(w)
    assert mode == 2 and {0, 1, 2} == set(units.tolist())
    tens = [x.cuda() for x in w.tensors()]
    o, lse, dq, _, _ = _run(w, tens, clear=True)
    assert torch.isfinite(dq).all()
    for h in range(7):
        one = W.Workload("alone", w.rows, 1, 1, 64, seed=0)
        assert _units(one)[0] == 0
        o1, lse1 = _run(one, [x[:, h:h + 1].contiguous() for x in tens[:3]], clear=False)
        assert torch.equal(o[:, h], o1[:, 0]) and torch.equal(lse[h], lse1[0])


@pytest.mark.parametrize("hq,hkv", [(12, 12), (20, 20), (21, 7), (42, 6)])
@pytest.mark.parametrize("d", [64, 96, 128])
def test_a_head_has_the_bits_it_has_alone(hq, hkv, d):
    w = W.Workload("paired", ROWS, hq, hkv, d, seed=hq)
    mode, units = _units(w)
    assert mode == (0 if hq == 12 else 2)     # (12 heads: too little work for it)
    assert mode == 0 or (set(units.tolist()) == {0, 1, 2} and (units == 2).sum() >= 10)
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
