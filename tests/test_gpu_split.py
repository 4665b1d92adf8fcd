"""Backward units cut into parts by query heads (small batches with several query heads per KV
head): parity with the fp64 oracle, and the same dK / dV bit for bit from every way to run it.

The parts' sums are fp32, as the whole unit's accumulator is, and are rounded to bf16 once, so the
tolerance is that of the whole units (relative L2 2e-2 for unit-normal bf16 inputs)."""
import pytest
import torch

from paper_2602_24082_b200 import workloads as W
from test_gpu_parity import TOL_GRAD, _run_gpu, check_against_oracle

pytestmark = pytest.mark.gpu

CASES = [
    # rows, Hq, Hkv, D, parts per unit
    ([[(1, (1,))]], 8, 1, 64, 8),                              # one tile of two rows, a head per part
    ([[(129, (127, 1))], [(31, (97,))]], 2, 1, 128, 2),        # tile edges, quarter edges
    ([[(100, (60, 128, 1)), (3, (30,))]], 7, 1, 64, 4),        # 1, 2, 2, 2 heads per part
    ([[(257, (5, 128, 31))]], 14, 2, 96, 4),
    ([[(640, (200, 73))]], 48, 8, 128, 4),                     # more parts than SMs, 1 or 2 heads each
    ([[(100, (90, 87))]], 64, 8, 128, 8),
    ([[(900, (700, 300, 148))]], 4, 1, 128, 4),                # units of 16 query tiles
    ([[(1200, (700, 512))]], 8, 1, 128, 8),                    # dQ of more than 592 blocks: sums in two rounds
]


@pytest.mark.parametrize("rows,hq,hkv,d,parts", CASES, ids=[f"{c[1]}q{c[2]}kv-d{c[3]}" for c in CASES])
def test_parts_add_up(rows, hq, hkv, d, parts):
    from paper_2602_24082_b200 import binding as B
    w = W.Workload("split", rows, hq, hkv, d, seed=7)
    tens = w.tensors()
    plan = B.plan_for(w)
    tiles = len(plan.read_bwd_tiles())
    assert plan.bwd_scratch_bytes >= 4 * w.total_tokens * hq * d + tiles * hkv * parts * 1024 * d
    gpu = _run_gpu(w, tens, for_backward=True)
    check_against_oracle(w, tens, gpu)

    q, k, v, do = (x.cuda() for x in tens)
    o, lse = B.pp_attn_fwd(plan, q, k, v, w.softmax_scale)
    want = [torch.from_numpy(x).cuda() for x in gpu[2:]]
    det = [B.pp_attn_bwd(plan, q, k, v, o, lse, do, w.softmax_scale, deterministic=True) for _ in range(2)]
    assert all(torch.equal(a, b) for a, b in zip(*det))
    noalloc = [torch.full_like(x, 9.0) for x in (q, k, v)]
    B.pp_attn_bwd_noalloc(plan, q, k, v, o, lse, do, w.softmax_scale, *noalloc)
    host = B.HostStep(w)
    host(*[x.contiguous().pin_memory() for x in tens])
    torch.cuda.synchronize()
    assert plan.status() == (0, 0)
    # (without room for the parts in the built-in scratch, units stay whole: another rounding)
    whole = plan.bwd_scratch_bytes > B.pp_attn_bwd_noalloc_max_bytes()
    for got in (det[0], noalloc, [x.cuda() for x in (host.dq, host.dk, host.dv)]):
        for i, (a, b) in enumerate(zip(got, want)):
            exact = i > 0 and not (whole and got is noalloc)
            assert float((a.double() - b).norm()) <= (0 if exact else TOL_GRAD) * float(b.norm())
