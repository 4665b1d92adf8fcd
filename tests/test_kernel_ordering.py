"""Orders between threads that no run can show to hold: where one is missing, equal runs still agree
on the chip at hand.  They are read from the kernels' sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_24082_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_turns_of_the_deterministic_backward_are_released_and_acquired():
    """The reductions of one key tile come before those of the next: complete -> release -> acquire ->
    proxy fence -> issued, on every path."""
    assert ".relaxed." not in _source("pp_bwd.cu") + _source("pp_ptx.cuh")
    main = _source("pp_bwd.cu")
    dq = main[main.index("kBwdRegsDq, kBwdRegsLaunch>"):]
    assert dq.count("load_acquire_gpu(sem)") == 2
    assert re.search(r"auto publish = [^;]*store_release_gpu\(p, k_rel \+ 1\);", dq)
    for call in re.finditer(r"publish\(pend\);", dq):
        assert re.search(r"bulk_wait_group<[^>]*>\(\);\s*$", dq[:call.start()])
    # published before the unit waits for its next turn: no unit below waits for one that waits itself
    assert dq.index("publish(pend);") < dq.index("if (kDet && sem && c == 0)")
    turn, reduce = dq.index("if (kDet && sem && c == 0)"), dq.index("tma_reduce_add_3d(")
    assert re.search(r"fence_proxy_async_global\(\);\s*}\s*if \(32 \* quarter < qt.len\) $", dq[turn:reduce])


def test_tensor_memory_is_handed_back_behind_a_fence():
    """One lane arrives for its warp: what the other lanes did to tensor memory is ordered before it by
    their own fence and the warp barrier."""
    main = _source("pp_bwd.cu")
    for bar in ("kPReady", "kDsReady", "kDqDrained", "kDkvFree"):
        places = [m.start() for m in re.finditer(r"mbar_arrive\(bar\(%s\)\)" % bar, main)]
        assert places
        for at in places:
            assert re.search(r"tc_fence_before\(\);\s*__syncwarp\(\);\s*if \(lane == 0\) $", main[:at]), bar


def test_kernels_that_start_early_promise_nothing_about_their_inputs():
    """A kernel that waits for the one in front is resident while its inputs are still written: pointers that
    are restrict would let loads be moved before the wait."""
    early = 0
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            for kernel in _source(name).split("__global__")[1:]:
                if "dependency_wait();" in kernel:
                    early += 1
                    assert "__restrict__" not in kernel, (name, kernel[:120])
    assert early >= 12
