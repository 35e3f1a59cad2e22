"""The all-FP64 form where the table of the Maxwellian's factors does not fit beside f and the stage buffers: the table
holds some of the elements at a time, with the same results, and the context is not refused for it."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

FLOW = dict(bc=[[0, 0], [2, 2], [0, 0]], bc_state=[[[0] * 5] * 2, [[0, 0.1, 0, 0, 1.0], [0, 0, 0, 0, 1.1]], [[0] * 5] * 2],
            body_force=(0.01, 0, 0))


# room: what is free beyond everything but the table, in tables
@pytest.mark.parametrize("dim, ne, p, nv, opts, curved, room", [
    (1, [1024], 1, (4096, 2, 2), {}, False, 0.4), (2, [101, 103], 2, (65, 3, 1), dict(limiter=True), False, 0.5),
    (3, [15, 14, 13], 1, (65, 3, 3), FLOW, False, 1.2), (3, [15, 14, 13], 1, (65, 3, 3), FLOW, True, 1.2)])
def test_table_in_blocks(dim, ne, p, nv, opts, curved, room):
    _build.build()
    import torch
    from paper_2308_06196_gb300 import bgk

    def make():
        return bgk.Solver(dim, ne, [0.0] * 3, [1.0] * 3, p, nv, (-6.0, -2.0, -2.0), (6.0, 2.0, 2.0), 0.02,
                          precision=bgk.FP64, chunks=8, **opts)

    def run(s):
        x = s.points()
        if curved:
            x = W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.05, "sine")
            s.set_geometry(x)
        P = W.smooth_prim(x, dim, seed=5, amp=0.05)
        P[:, 2:4] = 0.0
        s.set_state(P)
        s.step(1e-6, 2)
        out = s.moments(), s.equilibrium(), s.get_f()
        s.close()
        return out

    s = make()
    all_bytes, table = s.device_bytes, s.npts * sum(nv) * 8
    want = run(s)
    torch.cuda.empty_cache()
    left = (all_bytes - table + room * table) / 0.97
    fill = torch.empty(int(torch.cuda.mem_get_info()[0] - left), dtype=torch.uint8, device="cuda")
    try:
        s = make()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert s.device_bytes < all_bytes - table / 4
    got = run(s)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
