"""A task of several moment groups writes its running sums out after each, so the results do not depend on the
task length: the library's own choice must equal, bit for bit, the same groups with one group per task."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim, ne, p, nv, opts, curved", [
    (1, [9001], 3, (16, 16, 14), {}, False), (1, [9001], 4, (16, 16, 14), {}, False), (2, [71, 63], 3, (18, 18, 8), {}, False),
    (3, [9, 7, 11], 2, (18, 18, 16), {}, False), (3, [9, 7, 11], 3, (16, 16, 16), dict(limiter=True), False),
    (3, [9, 7, 6], 3, (18, 18, 18), {}, True), (3, [9, 7, 11], 1, (24, 24, 22), {}, True)])
def test_library_task_length_equals_one_group_per_task(dim, ne, p, nv, opts, curved):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    tiles = max(-(-int(np.prod(c)) // 32) for c in
                [(-(-nv[0] // 2), -(-nv[1] // 2), -(-nv[2] // 2))])  # of the largest octant
    G = max(1, min(8, tiles * int(np.prod(ne)) // (152 * 32)))  # the library's moment group
    got = []
    for o in ({}, dict(vtiles_per_task=G)):
        s = bgk.Solver(dim, ne, [0.0] * 3, [1.0] * 3, p, nv, (-5.0,) * 3, (5.0,) * 3, 0.02, **opts, **o)
        x = s.points()
        if curved:
            s.set_geometry(W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.1, "sine"))
        s.set_state(W.smooth_prim(x, dim, seed=5, amp=0.1))
        s.step(1e-6, 2)
        got.append((s.moments(), s.equilibrium()))
        del s
    for a, b in zip(*got):
        assert np.array_equal(a, b)
