"""Rules that the kernel sources keep wherever a mistake could hang a GPU, checked on the text (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_08923_b200", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _functions(src):
    """(name, body) of the functions of sm100_ptx.cuh."""
    for m in re.finditer(r"__forceinline__ \w+ (\w+)\([^)]*\)\s*\{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m[1], src[m.end():i - 1]


def test_aligned_cluster_barriers_are_reached_by_converged_warps():
    """barrier.cluster with .aligned is undefined when the lanes of a warp arrive apart: every helper brings them together itself, and kernels use the helpers."""
    found = []
    for name, body in _functions(_source("sm100_ptx.cuh")):
        if re.search(r"barrier\.cluster\S*\.aligned", body):
            found.append(name)
            assert 0 <= body.find("__syncwarp()") < body.find("barrier.cluster"), name
    assert {"cluster_sync", "cluster_arrive_relaxed", "cluster_wait"} <= set(found)
    for f in os.listdir(CSRC):
        assert f == "sm100_ptx.cuh" or "barrier.cluster" not in _source(f), f


def test_warps_leave_a_wait_together_and_branch_on_one_answer():
    """In the tensor-core kernels a barrier is waited for through the helpers that bring the lanes together again, or by lane 0 for the others; and an
    answer that may differ between lanes is not branched on before a vote."""
    helpers = dict(_functions(_source("sm100_ptx.cuh")))
    assert "__syncwarp()" in helpers["mbar_wait_converged"] and "__all_sync" in helpers["mbar_wait_warp"]
    for f in ("gemm_tc.cuh", "attn_tc.cuh"):
        src = _source(f)
        for m in re.finditer(r"[^;{}]*\bmbar_wait\([^;]*;", src):
            assert "if (lane == 0)" in m[0], (f, m[0].strip())
        for call in ("mbar_wait_converged(", "wait_full("):
            assert not re.search(r"if \([^;{]*" + re.escape(call), src), (f, call)
