"""A small batch is not held up by long tasks: stepping a few members with the library's own task lengths takes no longer
than with one moment group per task."""
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members, seed", [(2, 2), (4, 3), (8, 3), (16, 2)])
def test_own_length_against_single_groups(members, seed):
    _build.build()
    import torch
    from paper_2308_06196_gb300.bgk import Batch, Solver

    ms = W.sod_members(members=members, seed=seed, degrees=(1, 3))
    runs = []
    for given in (False, True):
        ss = []
        for m in ms:
            c = W.mesh_kwargs(m)
            nvt = sum(-(-(a * b * d) // 32) for a in (c["nv"][0] // 2, -(-c["nv"][0] // 2))
                      for b in (c["nv"][1] // 2, -(-c["nv"][1] // 2)) for d in (c["nv"][2] // 2, -(-c["nv"][2] // 2)))
            G = max(1, min(8, nvt * c["nelem"][0] // (152 * 32)))  # the library's moment group
            s = Solver(c["dim"], c["nelem"], c["lo"], c["hi"], c["p"], c["nv"], c["vlo"], c["vhi"], c["tau"], bc=m["bc"],
                       bc_state=m["bc_state"], chunks=1, vtiles_per_task=G if given else 0)
            s.set_state(W.prim_sod(s.points(), m["left"], m["right"]))
            ss.append(s)
        b = Batch(ss)
        st = torch.cuda.Stream()
        b.set_stream(st.cuda_stream)
        runs.append((b, st, [s.dt(0.05) for s in ss], ss))
    best = [1e30, 1e30]
    for rep in range(70):  # the best of six, and of more where another job on the machine held some up
        if rep > 6 and best[0] <= 1.05 * best[1]:
            break
        for k, (b, st, dt, _) in enumerate(runs):
            x, y = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            x.record(st)
            b.step(dt, 4)
            y.record(st)
            b.synchronize()
            if rep:
                best[k] = min(best[k], x.elapsed_time(y))
    assert best[0] <= 1.05 * best[1], best
