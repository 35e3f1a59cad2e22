"""Tasks of several moment groups with a shorter last task, in every stage kernel that has them: the results must equal,
bit for bit, the same groups with one group per task. The launches of a captured stage show that the library's
choice holds several groups at these sizes."""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu

D = [[1, 1], [0, 0], [0, 0]]
DS = [[[1.0, 0.1, 0, 0, 1.0], [0.8, 0, 0, 0, 1.1]], [[0] * 5] * 2, [[0] * 5] * 2]
FLOW = dict(bc=[[0, 0], [2, 2], [0, 0]], bc_state=[[[0] * 5] * 2, [[0, 0.1, 0, 0, 1.0], [0, 0, 0, 0, 1.1]], [[0] * 5] * 2],
            body_force=(0.01, 0, 0))
GAS = dict(mu_ref=0.02, mu_omega=0.8, limiter=True)


def octant_tiles(nv):
    """32-velocity tiles of every sign octant of a grid on [-5, 5], in launch order (empty ones left out)."""
    # the middle one of an odd number of nodes is 0 but for the spacing's rounding
    low = [0 if n == 1 else sum(k * Fraction(10.0 / (n - 1)) < 5 for k in range(n)) for n in nv]
    out = []
    for o in range(8):
        n = 1
        for d in range(3):
            n *= nv[d] - low[d] if (o >> d) & 1 else low[d]
        if n:
            out.append(-(-n // 32))
    return out


class KernelParams(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def stage_grids(s, dt):
    """CTAs of the stage kernels that one stage of s launches (captured, not run)."""
    import torch

    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    s.synchronize()
    s.set_stream(st.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0
    s.stage(dt, 0)
    g, n, name, kind = C.c_void_p(), C.c_size_t(), C.c_char_p(), C.c_int()
    assert cu.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(g)) == 0
    s.set_stream(None)
    node, one = C.c_void_p(), C.c_size_t(1)  # a chain from its one root
    assert cu.cuGraphGetRootNodes(g, C.byref(node), C.byref(one)) == 0
    chain = []
    while one.value:
        chain.append(node.value)
        n.value = 1
        assert cu.cuGraphNodeGetDependentNodes(C.c_void_p(chain[-1]), C.byref(node), C.byref(n)) == 0
        one.value = n.value
    out = []
    for q in chain:
        q = C.c_void_p(q)
        assert cu.cuGraphNodeGetType(q, C.byref(kind)) == 0
        if kind.value != 0:  # not a kernel
            continue
        k = KernelParams()
        assert cu.cuGraphKernelNodeGetParams_v2(q, C.byref(k)) == 0
        if k.func:
            assert cu.cuFuncGetName(C.byref(name), C.c_void_p(k.func)) == 0
        else:
            assert cu.cuKernelGetName(C.byref(name), C.c_void_p(k.kern)) == 0
        if b"k_stage" in name.value:
            out.append(k.grid[0])
    assert cu.cuGraphDestroy(g) == 0
    return out


@pytest.mark.parametrize("dim, ne, p, nv, opts, curved", [
    (1, [69457], 1, (46, 46, 1), {}, False), (1, [44974], 2, (46, 46, 1), GAS, False),
    (1, [34796], 3, (46, 46, 1), dict(bc=D, bc_state=DS, limiter=True), False), (1, [679], 4, (14, 15, 14), {}, False),
    (1, [131], 5, (27, 27, 24), dict(bc=D, bc_state=DS, limiter=True), False),
    (2, [11, 11], 1, (28, 28, 25), {}, False), (2, [15, 16], 1, (18, 18, 18), GAS, False),
    (2, [28, 27], 3, (13, 13, 11), {}, False), (2, [27, 27], 3, (14, 15, 12), dict(bc=D, bc_state=DS, limiter=True), False),
    (3, [8, 9, 7], 1, (13, 13, 11), FLOW, False), (3, [7, 9, 8], 2, (12, 13, 9), FLOW, False),
    (3, [7, 8, 9], 2, (12, 14, 10), {}, False), (3, [4, 6, 6], 3, (13, 15, 13), {}, False),
    (3, [4, 5, 3], 3, (21, 21, 21), GAS, False), (3, [7, 6, 4], 3, (13, 13, 11), FLOW, False),
    (3, [10, 8, 9], 1, (12, 13, 9), {}, True), (3, [4, 5, 6], 1, (19, 19, 19), GAS, True),
    (3, [6, 5, 5], 2, (13, 15, 13), FLOW, True), (3, [5, 4, 5], 3, (13, 15, 13), {}, True)])
def test_ragged_tasks_of_several_groups(dim, ne, p, nv, opts, curved):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    tiles = octant_tiles(nv)
    G = max(1, min(8, max(tiles) * int(np.prod(ne)) // (152 * 32)))  # the library's moment group
    groups = [-(-n // G) for n in tiles]
    got, grids = [], []
    for o in ({}, dict(vtiles_per_task=G)):
        s = bgk.Solver(dim, ne, [0.0] * 3, [1.0] * 3, p, nv, (-5.0,) * 3, (5.0,) * 3, 0.02, chunks=8, **opts, **o)
        x = s.points()
        if curved:
            x = W.curved_nodes(x, [0.0] * 3, [1.0] * 3, ne, 0.1, "sine")
            s.set_geometry(x)
        P = W.smooth_prim(x, dim, seed=5, amp=0.1)
        s.set_state(P)
        grids.append(stage_grids(s, 1e-6))
        s.step(1e-6, 2)
        got.append((s.moments(), s.equilibrium()))
        s.close()
    assert len(grids[0]) == len(grids[1]) == len(tiles)
    tasks = [round(a * n / b) for a, b, n in zip(*grids, groups)]
    assert any(t > 1 and -(-n // t) >= 2 and n % -(-n // t) for t, n in zip(tasks, groups)), (groups, tasks)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
