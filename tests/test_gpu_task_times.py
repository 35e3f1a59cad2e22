"""The library's task length is no worse than one moment group per task, at shapes whose tasks are few rounds of the
chip's resident ones (where a longer task can leave a large part of the last round idle) and at one with many."""
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

FLOW = dict(bc=[[0, 0], [2, 2], [0, 0]], bc_state=[[[0] * 5] * 2, [[0, 0.1, 0, 0, 1.0], [0, 0, 0, 0, 1.1]], [[0] * 5] * 2],
            body_force=(0.01, 0, 0))


@pytest.mark.parametrize("ne, p, n, opts, curved, G", [
    ([6, 6, 3], 2, 40, FLOW, False, 5), ([8, 11, 8], 2, 21, FLOW, False, 6), ([8, 13, 12], 1, 25, {}, False, 8),
    ([17, 12, 9], 1, 24, FLOW, False, 8), ([7, 6, 8], 1, 24, {}, True, 3), ([32, 16, 4], 2, 24, FLOW, False, 8)])
def test_own_length_against_single_groups(ne, p, n, opts, curved, G):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    ss = []
    for o in ({}, dict(vtiles_per_task=G)):
        s = bgk.Solver(3, ne, [0.0] * 3, [1.0] * 3, p, (n, n, n), (-5.0,) * 3, (5.0,) * 3, 0.02, chunks=8, **opts, **o)
        x = s.points()
        if curved:
            x = W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.1, "sine")
            s.set_geometry(x)
        s.set_state(W.smooth_prim(x, 3, seed=5, amp=0.02))
        ss.append(s)
    best = [1e30, 1e30]
    for rep in range(60):  # the best of six, and of more where another job on the machine held some up
        if rep >= 6 and best[0] <= 1.04 * best[1]:
            break
        for k, s in enumerate(ss):
            s.set_timing(True)
            s.step(1e-6, 2)
            t = s.timing()
            best[k] = min(best[k], t["stage_ms"] / t["stage_launches"])
    assert best[0] <= 1.04 * best[1], best
