"""Launching the octants of a stage one by one (opts.chunks = 8; what every problem beyond 64 MB of f does: the octants'
own kernels, the rotating slots, the halo sources of later chunks) against the merged launch of a small problem
(chunks = 0), which the oracle comparisons run. The moment groups are the same, so the results must agree bit for
bit, for every kernel and form and for given and automatic group lengths; device_bytes shows that the two routes
were taken."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

D = [[1, 1], [0, 0], [0, 0]]
DS = [[[1.0, 0.1, 0, 0, 1.0], [0.8, 0, 0, 0, 1.1]], [[0] * 5] * 2, [[0] * 5] * 2]
WALL = [[0, 0], [2, 2], [0, 0]]
WS = [[[0] * 5] * 2, [[0, 0.1, 0, 0, 1.0], [0, 0, 0, 0, 1.1]], [[0] * 5] * 2]
DIR = dict(bc=D, bc_state=DS)
FLOW = dict(bc=WALL, bc_state=WS, body_force=(0.01, 0, 0))
GAS = dict(mu_ref=0.02, mu_omega=0.8, limiter=True)
LINES = [(1, [19], p, nv, o, "") for p in (1, 2, 3, 4, 5) for nv, o in (((9, 8, 11), DIR), ((10, 10, 1), GAS))]
QUADS = [(2, [3, 5], p, nv, o, "") for p in (1, 2, 3) for nv, o in (((9, 10, 8), {}), ((9, 9, 9), dict(DIR, **GAS)))]
HEXES = [(3, [2, 3, 2], p, (9, 9, 9), o, "") for p in (1, 2, 3) for o in ({}, GAS, dict(DIR, limiter=True), FLOW)]
CURVED = [(3, [3, 2, 3], p, (8, 9, 8), o, "curved") for p in (1, 2, 3) for o in ({}, dict(FLOW, limiter=True))]
OTHER = [(3, [3, 3, 3], p, (8, 9, 8), {}, "unstructured") for p in (1, 2, 3)]
OTHER += [(3, [2, 2, 3], 3, (8, 9, 8), dict(precision=1, **FLOW), c) for c in ("", "curved")]


def make(dim, ne, p, nv, opts, form, chunks, G):
    from paper_2308_06196_gb300 import bgk

    s = bgk.Solver(dim, ne, [0.0] * 3, [1.0] * 3, p, nv, (-5.0,) * 3, (5.0,) * 3, 0.02, chunks=chunks,
                   vtiles_per_task=G, **opts)
    x = s.points()
    if form:
        x = W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.1, "sine")
    if form == "unstructured":
        m = W.unstructured_box(ne, p, seed=11)
        x = x[m["node_map"]]
        s.set_connectivity(m["nbr"], m["nface"], m["orient"])
    if form:
        s.set_geometry(x)
    s.set_state(W.smooth_prim(x, dim, seed=5, amp=0.1))
    return s


@pytest.mark.parametrize("G", [0, 1, 3])
@pytest.mark.parametrize("dim, ne, p, nv, opts, form", LINES + QUADS + HEXES + CURVED + OTHER)
def test_octant_by_octant_equals_merged(dim, ne, p, nv, opts, form, G):
    _build.build()
    got, size = [], []
    for chunks in (0, 8):
        s = make(dim, ne, p, nv, opts, form, chunks, G)
        s.step(1e-3, 2)
        Q = s.moments()
        s.set_f(s.get_f())  # (the moments-only pass)
        s.step(1e-3, 1)
        got.append((Q, s.moments(), s.equilibrium(), s.get_f()))
        size.append(s.device_bytes)
    assert size[0] > size[1]
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("p, opts", [(1, {}), (2, {}), (2, GAS), (3, {}), (3, GAS)])
@pytest.mark.parametrize("chunks", [0, 8])
def test_exchange_faces_octant_by_octant(p, opts, chunks):
    """One subdomain that is its own neighbour across both exchange faces is the periodic box."""
    import torch

    _build.build()
    ne, nv, dt = [3, 2, 3], (9, 8, 9) if not opts else (9, 9, 9), 1e-3
    whole = make(3, ne, p, nv, opts, "", 8, 2)
    whole.step(dt, 2)
    s = make(3, ne, p, nv, dict(opts, bc=[[3, 3], [0, 0], [0, 0]]), "", chunks, 2)
    lo, hi = (torch.empty(s.halo_floats(), dtype=torch.float32, device="cuda") for _ in range(2))
    s.set_halo(0, hi)  # across the low face lies the layer next to the high one
    s.set_halo(1, lo)
    for _ in range(2):
        for st in range(3):
            s.halo_pack(st, lo, hi)
            s.stage(dt, st)
    s.synchronize()
    for a, b in ((whole.moments(), s.moments()), (whole.equilibrium(), s.equilibrium()), (whole.get_f(), s.get_f())):
        assert np.array_equal(a, b)
