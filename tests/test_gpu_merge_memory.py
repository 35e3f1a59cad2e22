"""Small problems keep two full stage buffers. All contexts together hold at most 1 GiB for that beyond the rotating
chunk slots: past it a context steps chunk by chunk on the slots, with the same results, and a closed context
gives its share back."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


def make(**opts):
    from paper_2308_06196_gb300 import bgk

    return bgk.Solver(3, [5, 4, 4], [0.0] * 3, [1.0] * 3, 3, (14, 14, 14), (-5.0,) * 3, (5.0,) * 3, 0.02, **opts)


def run(s):
    s.set_state(W.smooth_prim(s.points(), 3, seed=5, amp=0.1))
    s.step(1e-3, 2)
    return s.moments(), s.equilibrium(), s.get_f()


def test_many_small_contexts():
    _build.build()
    by_slots = make(chunks=8)  # one chunk per octant, launched in turn
    want, slots = run(by_slots), by_slots.device_bytes
    ss = [make() for _ in range(60)]
    extra = [s.device_bytes - slots for s in ss]
    assert 0 < extra[0] < 1 << 26 and sum(extra) <= 1 << 30
    assert extra[-1] == 0 and sum(extra) > (1 << 30) - 2 * extra[0]
    for s in (ss[0], ss[-1]):
        for a, b in zip(run(s), want):
            assert np.array_equal(a, b)
    for s in ss[:2]:
        s.close()
    again = [make() for _ in range(3)]
    assert [s.device_bytes - slots for s in again] == [extra[0], extra[0], 0]
