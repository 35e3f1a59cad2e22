"""The Newton solve with a body force in both forms: up to 6,485 points four lanes share a point and each forms its own
axis's force sums, beyond that a thread forms them all. Every sum has the same order, so a row of elements that
are copies of one another, solved at point counts on both sides of the limit, must give the shortest row's
moments, equilibria and (through the force polynomials) f, exactly."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

FORCE = (0.3, -0.2, 0.1)


def run(ne, p, nv, **opts):
    from paper_2308_06196_gb300 import bgk

    h = 0.5
    s = bgk.Solver(3, [ne, 1, 1], [0.0] * 3, [ne * h, h, h], p, nv, (-6.0,) * 3, (6.0,) * 3, 1e-2, vtiles_per_task=2,
                   chunks=1, body_force=FORCE, **opts)
    rng = np.random.default_rng(4)
    P = np.zeros(((p + 1) ** 3, 5))
    P[:, 0], P[:, 1:4], P[:, 4] = rng.uniform(0.8, 1.2, len(P)), rng.uniform(-0.3, 0.3, (len(P), 3)), rng.uniform(0.9, 1.1, len(P))
    s.set_state(np.tile(P, (ne, 1)))
    s.step(2e-3, 2)
    return [a.reshape(ne, -1) for a in (s.moments(), s.equilibrium(), s.get_f())]


@pytest.mark.parametrize("p, nv, opts, counts", [
    (1, (8, 9, 10), {}, (810, 811, 1217)), (1, (9, 9, 9), dict(mu_ref=0.02, mu_omega=0.8), (810, 811)),
    (2, (8, 8, 8), dict(precision=1), (240, 241))])  # 6,480 points: four lanes; 6,488, 6,507 and more: one
def test_force_forms_agree_bit_for_bit(p, nv, opts, counts):
    _build.build()
    want = run(2, p, nv, **opts)
    for ne in counts:
        for a, b in zip(run(ne, p, nv, **opts), want):
            assert np.array_equal(a, np.broadcast_to(b[0], a.shape)), ne


def test_one_lane_force_matches_oracle():
    _build.build()
    from paper_2308_06196_gb300 import bgk

    # 7,168 points; the same discretisation element by element as 14 of them, which the oracle steps
    ne, lo, nv, v = [14, 8, 8], [0.0] * 3, (8, 8, 8), (5.0,) * 3
    hi, small, shi = [3.5, 2.0, 2.0], [14, 1, 1], [3.5, 0.25, 0.25]
    s = bgk.Solver(3, ne, lo, hi, 1, nv, tuple(-x for x in v), v, 0.02, body_force=FORCE)
    o = orc.Problem(3, small, lo, shi, 1, nv, tuple(-x for x in v), v, 0.02, force=FORCE)
    x = s.points()

    def prim(x):
        P = np.zeros((len(x), 5))
        a = 2 * np.pi * x[:, 0] / 3.5
        P[:, 0], P[:, 1], P[:, 2], P[:, 4] = 1 + 0.1 * np.sin(a), 0.1 * np.cos(a), 0.05, 1 + 0.05 * np.cos(a)
        return P

    s.set_state(prim(x))
    o.set_state(prim(o.points()))
    dt = o.dt(0.1)
    s.step(dt, 2)
    o.step(dt, 2)
    Q = s.moments().reshape(8, 8, 14, 8, 5)
    Qo = o.moments().reshape(14, 8, 5)
    # a tenth of the method's own bound of the FP32-split form, 1e-5 of the largest moment
    assert np.abs(Q - Qo[None, None]).max() <= 1e-6 * np.abs(Qo).max()
