"""The autotuner's cache tells a small problem's merged launches from the same problem launched chunk by chunk
(opts.chunks = 8): the second form is timed for itself, and only a repeat is answered from the cache."""
import time

import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [0, 8])
def test_each_launch_form_is_tuned(first):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    def tuned(chunks):
        s = bgk.Solver(3, [5, 4, 3 + first], [0.0] * 3, [1.0] * 3, 2, (11, 12, 10), (-5.0,) * 3, (5.0,) * 3, 0.02,
                       chunks=chunks)
        s.set_state(W.smooth_prim(s.points(), 3, seed=5, amp=0.1))
        s.synchronize()
        t = time.perf_counter()
        s.autotune()
        return time.perf_counter() - t

    tuned(first)
    other, repeat = tuned(8 - first), min(tuned(first) for _ in range(4))
    # some ten lengths, three stage passes of 20 us or more each, against a look into the cache
    assert other > 3e-4 and other > 5 * repeat, (other, repeat)
