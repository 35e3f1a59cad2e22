"""The all-FP64 stage's line form against the oracle at the shapes the other tests leave out: degrees 4 and 5
on lines, one chunk of mixed octants, velocity grids whose axes differ (table columns)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim, ne, p, nv, opts", [
    (1, [7], 1, (9, 8, 10), {}), (1, [5], 4, (9, 8, 10), {}), (1, [3], 5, (12, 9, 1), {}),
    (2, [3, 2], 2, (8, 9, 10), {}), (3, [2, 3, 1], 3, (8, 9, 7), dict(chunks=1)),
    (3, [2, 1, 2], 1, (7, 8, 9), dict(chunks=1, body_force=(0.02, -0.01, 0.03)))])
def test_lines_match_oracle(dim, ne, p, nv, opts):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    lo, hi, vlo, vhi = [0.0] * dim, [1.0] * dim, (-5.0, -4.5, -5.5), (5.0, 5.5, 5.0)
    s = bgk.Solver(dim, ne, lo, hi, p, nv, vlo, vhi, 0.02, precision=bgk.FP64, **opts)
    o = orc.Problem(dim, ne, lo, hi, p, nv, vlo, vhi, 0.02, force=opts.get("body_force"))
    P = W.smooth_prim(o.points(), dim, seed=3, amp=0.1)
    s.set_state(P)
    o.set_state(P)
    dt = o.dt(0.1)
    s.step(dt, 2)
    o.step(dt, 2)
    f, g = s.get_f(), o.get_f()
    # round-off of six stages: some 50 operations per value and stage, each at most 2^-53 of max f
    assert np.abs(f - g).max() <= 6 * 50 * 2.0**-53 * 10 * np.abs(g).max()
    assert np.abs(s.moments() - o.moments()).max() <= 1e-10 * np.abs(o.moments()).max()
