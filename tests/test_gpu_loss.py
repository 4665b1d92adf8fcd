"""GPU parity of the loss-side consumer against the numpy oracle (fp32 sums vs fp64)."""
import numpy as np
import pytest
import torch

from oracle import loss as L
from paper_2602_24082_b200 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    W.config0(),
    W.Workload("ragged", [[(257, (5, 128, 31))], [(1, (1, 300))]], 4, 2, 128, seed=4),
    W.Workload("single", [[(97, (64,)), (128, (128, 128, 7, 9, 40))], [(700, (1, 1))]], 2, 2, 64, seed=5),
    W.config2(),
    W.config4(3),
    # every team width of the kernel (mean segment 1 .. 4096 tokens), more responses than teams
    W.Workload("ones", [[(1, (1,) * 37)] for _ in range(9)], 1, 1, 64, seed=6),
    W.Workload("mean200", [[(200, (190, 210, 1, 399) * 5)]], 1, 1, 64, seed=7),
    W.Workload("mean400", [[(400, (511, 289, 400))], [(1, (799,))]], 1, 1, 64, seed=8),
    W.Workload("mean900", [[(900, (1023, 1, 1577))]], 1, 1, 64, seed=9),
    W.Workload("mean4096", [[(4096, (4095, 4097))]], 1, 1, 64, seed=10),
    # every number of warps per group (16 up to 296 groups on 148 SMs, then 8, 4, 2, 1), a last block
    # that is not full, more responses than a warp has lanes
    W.Workload("gang8", [[(3, (40, 2)), (1, (1,) * 17), (300, (200,))]] * 149, 1, 1, 64, seed=11),
    W.Workload("gang8-many", [[(3, (40, 2)), (1, (1,) * 33)]] * 401, 1, 1, 64, seed=15),
    W.Workload("gang4", [[(150, (140, 2, 130))]] * 701, 1, 1, 64, seed=12),
    W.Workload("gang2", [[(2, (3, 1)), (7, (130,)), (1, (1, 2, 3, 4))]] * 401, 1, 1, 64, seed=13),
    W.Workload("gang1", [[(2, (3, 1)), (9, (35, 1, 70, 33))]] * 1201, 1, 1, 64, seed=14),
] + [W.random_structure(s) for s in range(8)]


@pytest.mark.parametrize("w", CASES, ids=lambda w: w.name)
@pytest.mark.parametrize("with_ref", [True, False], ids=["dpo", "noref"])
def test_preference_loss_parity(w, with_ref):
    from paper_2602_24082_b200 import binding as B
    rng = np.random.default_rng(7)
    T = w.total_tokens
    lp = (-rng.gamma(2.0, 1.0, T)).astype(np.float32)
    ref = (-rng.gamma(2.0, 1.0, T)).astype(np.float32) if with_ref else None
    beta = 0.1 if with_ref else 0.01
    plan = B.plan_for(w, desc_on_device=True)
    out = B.pp_preference_loss(plan, torch.from_numpy(lp).cuda(),
                               torch.from_numpy(ref).cuda() if with_ref else None, beta)
    torch.cuda.synchronize()
    assert plan.status() == (0, 0)
    s, r, loss, grad = (x.cpu().numpy().astype(np.float64) for x in out)
    S, Rw, Ls, G = L.preference_loss(w.rows, lp, ref, beta)
    # fp32 sums of up to a few thousand O(1) terms: relative 1e-5 of the magnitude
    assert np.abs(s - S).max() <= 1e-5 * max(1.0, np.abs(S).max())
    assert np.abs(r - Rw).max() <= 2e-5 * max(1.0, np.abs(Rw).max()) + 1e-5
    assert np.abs(loss - Ls).max() <= 1e-4 * max(1.0, np.abs(Ls).max())
    assert np.abs(grad - G).max() <= 1e-4 * max(1e-3, np.abs(G).max())
    # prompt tokens carry no gradient: exactly zero
    prompt = np.zeros(T, dtype=bool)
    for (st, ln, _, _, seg) in w.segments():
        if seg == 0:
            prompt[st:st + ln] = True
    assert not grad[prompt].any()


@pytest.mark.parametrize("rows", [[[(100, (8192, 5000, 33))]], [[(9, (4097, 4000))], [(300, (1, 7000))]],
                                  [[(3, (150, 201)), (1, (7, 90, 8, 1))]] * 40, [[(5, (40, 30))]] * 5000],
                         ids=["long", "two", "short", "many"])
def test_sums_are_rounded_once(rows):
    """Multiples of 2^-16 below 4: the few dozen terms of a lane add up exactly in fp32, a response's sum
    does not fit 24 bits, so what comes out is the exact sum (and beta times the exact difference) rounded."""
    from paper_2602_24082_b200 import binding as B
    w = W.Workload("exact", rows, 1, 1, 64, seed=1)
    rng = np.random.default_rng(3)
    lp, ref = (-rng.integers(0, 1 << 18, w.total_tokens) / 65536.0 for _ in range(2))
    plan = B.plan_for(w)
    f32 = lambda x: torch.from_numpy(x.astype(np.float32)).cuda()
    s, r, _, _ = B.pp_preference_loss(plan, f32(lp), f32(ref), 0.1)
    spans = [(a, a + n) for a, n, _, _, seg in w.segments() if seg]
    S, Sr = (np.array([x[a:b].sum() for a, b in spans]) for x in (lp, ref))
    assert np.array_equal(s.cpu().numpy(), S.astype(np.float32))
    assert np.array_equal(r.cpu().numpy(), (np.float64(np.float32(0.1)) * (S - Sr)).astype(np.float32))
