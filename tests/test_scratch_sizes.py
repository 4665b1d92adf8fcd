"""Sizes of the backward scratch (host only)."""
import numpy as np
import pytest

from paper_2602_24082_b200 import binding as B

ALIGN = lambda n: -(-n // 256) * 256


def _scratch(rows, hq, hkv, d):
    groups = [g for row in rows for g in row]
    a = lambda x: np.asarray(x, np.int32)
    tokens = sum(p + sum(rs) for p, rs in groups)
    desc = (a(np.cumsum([0] + [len(r) for r in rows])), a([p for p, _ in groups]),
            a(np.cumsum([0] + [len(rs) for _, rs in groups])), a([r for _, rs in groups for r in rs]))
    problem, keep = B.make_problem(desc, hq, hkv, d, tokens)
    return B.pp_plan_workspace_bytes(problem)[2], tokens, len(groups)


@pytest.mark.parametrize("rows,hq,hkv,d,parts", [
    ([[(1000, (12,) * 64)]] * 4, 8, 1, 128, 8),            # many short responses
    ([[(2000, (2,) * 1000)]], 8, 1, 128, 8),
    ([[(100, (60, 128, 1)), (3, (30,))]], 7, 1, 64, 4),
    ([[(2000, (500, 300))]] * 60, 32, 8, 128, 1),          # enough units: whole
])
def test_parts_have_room_by_the_backwards_own_tiles(rows, hq, hkv, d, parts):
    """The backward's key tiles are cut per group, so responses add none: accumulator, two statistics,
    turn counters, and dV and dK in fp32 for each part of a (key tile, KV head)."""
    got, tokens, groups = _scratch(rows, hq, hkv, d)
    tiles = tokens // 128 + groups
    want = ALIGN(4 * tokens * hq * d) + 2 * ALIGN(4 * tokens * hq) + ALIGN(16 * tiles * hq)
    if parts > 1:
        want += tiles * hkv * parts * 2 * 128 * d * 4
    assert got == want
