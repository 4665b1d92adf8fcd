"""What the Python side of a plan keeps, without a GPU: the module that makes the calls is replaced."""
import types

import numpy as np
import pytest

from paper_2602_24082_b200 import binding as B


@pytest.fixture
def builds(monkeypatch):
    """pp_build_plan with a module that accepts int32 arrays and gives the null handle."""
    seen = []

    def build_plan(desc, *rest):
        if not all(getattr(a, "dtype", None) == np.int32 for a in desc):
            return None
        seen.append(tuple(a.tolist() for a in desc))
        return 0

    monkeypatch.setattr(B, "_ext", types.SimpleNamespace(build_plan=build_plan))
    return seen


DESC = [[0, 1, 2], [3, 4], [0, 2, 3], [5, 6, 7]]      # 2 groups, 3 responses, 25 tokens
arrays = lambda: [np.asarray(a, np.int32) for a in DESC]


def test_a_plan_is_that_of_the_arrays_at_the_call(builds):
    """A loader may keep one list and put the next batch's arrays into it."""
    desc = arrays()
    plan = B.pp_build_plan(desc, 4, 2, 64, 25, workspace=object())
    desc[:] = [np.asarray(a, np.int32) for a in ([0, 1], [3], [0, 1], [5])]
    p = plan.problem
    assert (p.num_rows, p.num_groups, p.num_responses, p.total_tokens) == (2, 2, 3, 25)
    want, _ = B.make_problem(arrays(), 4, 2, 64, 25)
    assert plan.bwd_scratch_bytes == B.pp_plan_workspace_bytes(want)[2]


@pytest.mark.parametrize("dtype", [np.int32, np.int64])
def test_descriptors_may_come_from_an_iterator(builds, monkeypatch, dtype):
    """An iterator can be gone through once, whichever way its arrays are taken."""
    monkeypatch.setattr(B, "_call", lambda index, where, fn, problem, *rest: builds.append(problem.num_responses))
    workspace = types.SimpleNamespace(is_cuda=True, get_device=lambda: 0, data_ptr=lambda: 0, numel=lambda: 0,
                                      is_contiguous=lambda: True)
    plan = B.pp_build_plan((np.asarray(a, dtype) for a in DESC), 4, 2, 64, 25, workspace=workspace)
    assert builds == [tuple(DESC)] if dtype is np.int32 else builds == [3]
    assert plan.problem.num_groups == 2
