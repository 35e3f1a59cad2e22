"""The Newton solve's forms by point count (four lanes per point, a thread per point) form every sum in the
same order, so they give the same bits: a line whose elements are copies of one another is solved at point
counts on both sides of the limit and with ragged last warps, and every element must agree with the
shortest line's, exactly."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build

pytestmark = pytest.mark.gpu


def run(ne, nv, **opts):
    from paper_2308_06196_gb300 import bgk

    h = 0.5
    s = bgk.Solver(1, [ne], [0.0], [ne * h], 2, nv, (-6.0,) * 3, (6.0,) * 3, 1e-2, vtiles_per_task=3, **opts)
    P = np.zeros((3, 5))
    P[:, 0], P[:, 1], P[:, 2], P[:, 4] = [1.0, 1.2, 0.9], [0.1, -0.2, 0.3], 0.05, [1.0, 0.9, 1.1]
    s.set_state(np.tile(P, (ne, 1)))
    s.step(2e-3, 2)
    return s.moments().reshape(ne, 15), s.equilibrium().reshape(ne, 15)


@pytest.mark.parametrize("nv, opts", [((9, 8, 10), {}), ((12, 12, 12), dict(mu_ref=0.02, mu_omega=0.8)), ((10, 10, 1), {})])
def test_forms_agree_bit_for_bit(nv, opts):
    _build.build()
    Q0, P0 = run(2, nv, **opts)
    # 9,726 / 9,729 points: the last size of one form and the first of the other
    for ne in (5, 3242, 3243, 6486, 25942):
        Q, P = run(ne, nv, **opts)
        assert np.array_equal(Q, np.broadcast_to(Q0[0], Q.shape)) and np.array_equal(P, np.broadcast_to(P0[0], P.shape)), ne
