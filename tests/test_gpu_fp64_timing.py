"""Launch timing of the all-FP64 form: the stage time holds everything that a stage computes, the tabulation of
the Maxwellian's factors too, so that stage and Newton times together are the step's time. On two axes of two nodes
the table is a large part of the stage (4,100 exponentials a point beside 16,384 values)."""
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunks", [0, 1])
def test_stage_and_newton_times_are_the_step(chunks):
    _build.build()
    import torch
    from paper_2308_06196_gb300 import bgk

    s = bgk.Solver(1, [4096], [0.0], [1.0], 1, (4096, 2, 2), (-6.0, -1.0, -1.0), (6.0, 1.0, 1.0), 0.02,
                   precision=bgk.FP64, chunks=chunks)
    st = torch.cuda.Stream()
    s.set_stream(st.cuda_stream)
    P = W.smooth_prim(s.points(), 1, seed=2, amp=0.1)
    P[:, 2:4] = 0.0
    s.set_state(P)
    s.set_timing(True)
    share = []
    for _ in range(6):
        s.step(1e-6, 1)
        s.synchronize()
        s.set_timing(True)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(st)
        s.step(1e-6, 1)
        b.record(st)
        t = s.timing()
        share.append((t["stage_ms"] + t["newton_ms"]) / a.elapsed_time(b))
        assert t["stage_launches"] == 3 * (8 if chunks == 0 else 1) and t["newton_launches"] == 3
    # (what is left are the gaps between launches, some microseconds each of a step of several milliseconds)
    assert max(share) > 0.95, share
