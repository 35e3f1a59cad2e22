"""The p = 1 hexahedral kernel's periodic and Dirichlet-and-limiter forms keep 20 warps per SM: at 104 registers
instead of 96 it was 16, and up to 5 % slower."""
import ctypes as C

import numpy as np
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


class KernelParams(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


@pytest.mark.parametrize("chunks", [0, 8])
@pytest.mark.parametrize("opts", [{}, dict(bc=[[1, 1], [0, 0], [0, 0]], limiter=True, bc_state=[
    [[1.0, 0.1, 0, 0, 1.0], [0.8, 0, 0, 0, 1.1]], [[0] * 5] * 2, [[0] * 5] * 2])])
def test_twenty_warps(opts, chunks):
    import torch
    from paper_2308_06196_gb300 import bgk

    _build.build()
    s = bgk.Solver(3, [3, 2, 2], [0.0] * 3, [1.0] * 3, 1, (8, 8, 8), (-5.0,) * 3, (5.0,) * 3, 0.02, chunks=chunks, **opts)
    s.set_state(W.smooth_prim(s.points(), 3, seed=5, amp=0.1))
    s.synchronize()
    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    s.set_stream(st.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0
    s.stage(1e-3, 0)
    g, n, name, kind = C.c_void_p(), C.c_size_t(), C.c_char_p(), C.c_int()
    assert cu.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(g)) == 0
    assert cu.cuGraphGetNodes(g, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, C.byref(n)) == 0
    warps = []
    for q in nodes:
        k, ctas = KernelParams(), C.c_int()
        assert cu.cuGraphNodeGetType(C.c_void_p(q), C.byref(kind)) == 0
        if kind.value != 0:
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(q), C.byref(k)) == 0
        f = C.c_void_p(k.func)
        if not k.func:
            assert cu.cuKernelGetFunction(C.byref(f), C.c_void_p(k.kern)) == 0
        assert cu.cuFuncGetName(C.byref(name), f) == 0
        if b"k_stage3w" in name.value:
            assert cu.cuOccupancyMaxActiveBlocksPerMultiprocessor(C.byref(ctas), f, int(np.prod(k.block[:])),
                                                                  C.c_size_t(k.smem)) == 0
            warps.append(ctas.value * int(np.prod(k.block[:])) // 32)
    assert cu.cuGraphDestroy(g) == 0
    assert len(warps) == (1 if chunks == 0 else 8) and min(warps) >= 20, warps
