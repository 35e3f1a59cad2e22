"""The line stage's two forms at p <= 3, packed pairs of velocities and a lane per velocity, chosen by how much of the chip a
launch's tasks fill: the captured launch shows which ran on either side of the limit, and elements that are copies of
one another must give the same bits in both."""
import ctypes as C

import numpy as np
import pytest

from paper_2308_06196_gb300 import _build

pytestmark = pytest.mark.gpu


class KernelParams(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def stage_kernel(s):
    """Name of the stage kernel that one stage of s launches (captured, not run)."""
    import torch

    cu = C.CDLL("libcuda.so.1")
    st = torch.cuda.Stream()
    s.synchronize()
    s.set_stream(st.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(st.cuda_stream), 2) == 0
    s.stage(1e-3, 0)
    g, n, name, kind, out = C.c_void_p(), C.c_size_t(), C.c_char_p(), C.c_int(), set()
    assert cu.cuStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(g)) == 0
    s.set_stream(None)
    assert cu.cuGraphGetNodes(g, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, C.byref(n)) == 0
    for q in nodes:
        k = KernelParams()
        assert cu.cuGraphNodeGetType(C.c_void_p(q), C.byref(kind)) == 0
        if kind.value != 0:
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(q), C.byref(k)) == 0
        f = C.c_void_p(k.func)
        if not k.func:
            assert cu.cuKernelGetFunction(C.byref(f), C.c_void_p(k.kern)) == 0
        assert cu.cuFuncGetName(C.byref(name), f) == 0
        if b"k_stage" in name.value:
            out.add("pair" if b"pair" in name.value else "lane")
    assert cu.cuGraphDestroy(g) == 0
    assert len(out) == 1
    return out.pop()


@pytest.mark.parametrize("p, nv, opts", [
    (1, (8, 8, 8), dict(limiter=True)), (2, (8, 9, 10), {}), (3, (8, 8, 8), dict(mu_ref=0.02, mu_omega=0.8)), (3, (12, 11, 1), {})])
def test_forms_agree_bit_for_bit(p, nv, opts):
    _build.build()
    from paper_2308_06196_gb300 import bgk

    run, groups = 2 * (16 // (p + 1)), 0
    for o in range(8):
        n = [nv[d] - nv[d] // 2 if (o >> d) & 1 else nv[d] // 2 for d in range(3)]
        groups += -(-n[0] * n[1] * n[2] // 32)  # one tile each
    limit = -(-912 // groups) * run  # elements that give half a round of 1,824 tasks
    rng = np.random.default_rng(p)
    P = np.zeros((p + 1, 5))
    P[:, 0], P[:, 1:3], P[:, 4] = rng.uniform(0.8, 1.2, p + 1), rng.uniform(-0.3, 0.3, (p + 1, 2)), rng.uniform(0.9, 1.1, p + 1)
    got, forms = [], []
    for ne in (3, limit - run, limit):
        s = bgk.Solver(1, [ne], [0.0], [0.5 * ne], p, nv, (-6.0,) * 3, (6.0,) * 3, 1e-2, chunks=1, vtiles_per_task=1, **opts)
        s.set_state(np.tile(P, (ne, 1)))
        forms.append(stage_kernel(s))
        s.step(2e-3, 2)
        got.append([a.reshape(ne, -1) for a in (s.moments(), s.equilibrium(), s.get_f())])
    assert forms == ["lane", "lane", "pair"]
    for g in got[1:]:
        for a, b in zip(g, got[0]):
            assert np.array_equal(a, np.broadcast_to(b[0], a.shape))
