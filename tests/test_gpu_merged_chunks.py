"""Small problems launch all velocity chunks of a stage together: the same task groups as chunk by chunk. With
one tile per group the mixed-octant single chunk (opts.chunks = 1) has the same groups too, so the two must
agree bit for bit, for every kernel and form, with octants of different and of padded sizes."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

D = [[1, 1], [0, 0], [0, 0]]
DS = [[[1.0, 0.1, 0, 0, 1.0], [0.8, 0, 0, 0, 1.1]], [[0] * 5] * 2, [[0] * 5] * 2]
WALL = [[0, 0], [2, 2], [0, 0]]
WS = [[[0] * 5] * 2, [[0, 0.1, 0, 0, 1.0], [0, 0, 0, 0, 1.1]], [[0] * 5] * 2]


@pytest.mark.parametrize("dim, ne, p, nv, opts, curved", [
    (1, [7], 2, (9, 8, 11), dict(bc=D, bc_state=DS), False), (1, [18], 3, (10, 9, 1), {}, False),
    (2, [3, 5], 3, (9, 10, 1), {}, False), (2, [4, 2], 2, (8, 7, 9), dict(bc=D, bc_state=DS, limiter=True), False),
    (3, [2, 3, 2], 1, (7, 8, 9), {}, False), (3, [2, 2, 3], 2, (9, 9, 9), dict(bc=D, bc_state=DS, limiter=True), False),
    (3, [2, 3, 1], 2, (8, 8, 8), dict(bc=WALL, bc_state=WS, body_force=(0.01, 0, 0)), False),
    (3, [2, 3, 2], 3, (9, 8, 7), {}, False), (3, [3, 2, 1], 3, (8, 8, 8), dict(mu_ref=0.02, mu_omega=0.8, limiter=True), False),
    (3, [2, 3, 2], 3, (8, 9, 8), dict(bc=WALL, bc_state=WS, body_force=(0.01, 0, 0)), False),
    (3, [3, 3, 2], 2, (8, 9, 8), {}, True), (3, [2, 2, 2], 2, (8, 9, 8), dict(precision=1), False)])
def test_merged_chunks_equal_one_chunk(dim, ne, p, nv, opts, curved):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    got = []
    for chunks in (0, 1):
        s = bgk.Solver(dim, ne, [0.0] * 3, [1.0] * 3, p, nv, (-5.0,) * 3, (5.0,) * 3, 0.02, chunks=chunks,
                       vtiles_per_task=1, **opts)
        x = s.points()
        if curved:
            s.set_geometry(W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.1, "sine"))
        s.set_state(W.smooth_prim(x, dim, seed=5, amp=0.1))
        s.step(1e-3, 2)
        Q = s.moments()
        s.set_f(s.get_f())  # (the moments-only pass)
        s.step(1e-3, 1)
        got.append((Q, s.moments(), s.get_f()))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
