"""Forward over query tiles whose rows belong to several segments (many short segments): parity with
the fp64 oracle through every form of the plan, and the tiles that each group should get.

The sums are those of the other tiles in another split, so the tolerances are the same (max-abs 2e-2
on O, 5e-3 on LSE, relative L2 2e-2 on the gradients, for unit-normal bf16 inputs)."""
import random

import numpy as np
import pytest
import torch

from paper_2602_24082_b200 import workloads as W
from test_gpu_parity import _run_gpu, check_against_oracle

pytestmark = pytest.mark.gpu


def _tiles(p, rs):
    """Work of the tiles of the segments, and of those of the group's grid."""
    up = lambda n: -(-n // 128)
    segs = [i + 1 for i in range(up(p))] + [up(p) + i + 1 for r in rs for i in range(up(r))]
    starts = np.cumsum([0, p] + list(rs))
    grid = []
    for q in range(0, starts[-1], 128):
        s = starts[np.searchsorted(starts, q, side="right") - 1]
        grid.append(q // 128 + 1 if q < p else up(p) + up(q - s) + 1)
    return segs, grid


def _many(n, seed):
    rng = random.Random(seed)
    return [[(rng.randint(1, 30), tuple(rng.randint(1, 25) for _ in range(rng.randint(1, 7))))] for _ in range(n)]


CASES = [
    # edges of segments on, before and behind edges of tiles and of quarters of a tile; a group
    # whose segments' tiles are less work; a prompt of one token; a response that begins one tile
    # and ends two tiles later
    ("edges", [[(100, (20, 8, 1, 127, 128)), (257, (5, 128, 31))], [(1, (1, 300, 2))],
               [(200, (128, 128, 128))], [(31, (1, 32, 64, 33, 95, 1)), (128, (1, 1, 126, 129))]], 24, 4, 64),
    ("d128", [[(100, (20, 8, 1, 127, 128)), (129, (5, 130, 31)), (3, (2, 1))]] * 3, 21, 3, 128),
    ("d96", [[(90, (39, 127, 1, 1, 60))], [(1, (126, 1, 1, 300))], [(250, (6, 7, 8))]], 40, 8, 96),
    ("sorted-orders", _many(150, 1), 2, 1, 64),         # more than 512 tiles
    ("multi-kernel-plan", _many(520, 2), 1, 1, 64),     # more than 2048 tiles
    # works of 1 to 24 key tiles, in groups of either kind of tile
    ("multi-kernel-long", _many(300, 3) + [[(1500, (1400, 1, 90)), (2, (300, 1, 1))]] + _many(250, 4), 2, 2, 64),
]


@pytest.mark.parametrize("name,rows,hq,hkv,d", CASES, ids=[c[0] for c in CASES])
def test_mixed_tiles(name, rows, hq, hkv, d):
    from paper_2602_24082_b200 import binding as B
    w = W.Workload(name, rows, hq, hkv, d, seed=11)
    tens = w.tensors()
    plan = B.plan_for(w)
    cost = lambda works: sum(works) + len(works)
    want = [min(_tiles(*g), key=cost) for row in rows for g in row]
    header = plan.workspace[:64].cpu().view(torch.int32)
    assert plan.status() == (0, 0) and int(header[9]) == sum(len(t) for t in want)
    results = [_run_gpu(w, tens, desc_on_device=dev, for_backward=dev) for dev in (False, True)]
    check_against_oracle(w, tens, results[0])
    for i in (0, 1, 3, 4):
        assert np.array_equal(results[0][i], results[1][i])
    host = B.HostStep(w)
    host(*[x.contiguous().pin_memory() for x in tens])
    torch.cuda.synchronize()
    for x, i in ((host.o, 0), (host.lse, 1), (host.dk, 3), (host.dv, 4)):
        assert np.array_equal(x.double().numpy(), results[0][i])
