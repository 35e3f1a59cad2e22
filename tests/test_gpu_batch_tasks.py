"""The task count that a batch reports is the one that its stage launches share out: runs of two half-warps'
elements (16 / (p + 1) each) times tasks of whole moment groups, whose length follows the degree's share of the chip unless it
was given or measured."""
import pytest

from paper_2308_06196_gb300 import _build, workloads as W

pytestmark = pytest.mark.gpu


def tiles(nv):
    """32-velocity tiles of a grid that is symmetric about 0: the octants are padded one by one."""
    n = 0
    for o in range(8):
        side = [k // 2 if not (o >> d) & 1 else k - k // 2 for d, k in enumerate(nv)]
        n += -(-side[0] * side[1] * side[2] // 32)
    return n


def runs(m):
    return -(-m["nelem"][0] // (2 * (16 // (m["p"] + 1))))


def count(m, G, ms):
    """Tasks of member m of ms with groups of G tiles; G = 0: the library's own groups and task length."""
    nvt, E = tiles(m["nv"]), m["nelem"][0]
    R = 1
    if G == 0:
        G = max(1, min(8, nvt * E // (152 * 32)))
        work = sum(runs(q) * tiles(q["nv"]) for q in ms if q["p"] == m["p"])
        R = max(1, max(1, min(16, work // (7 * 152 * 12))) // G)
    return runs(m) * -(-(-(-nvt // G)) // R)


@pytest.mark.parametrize("G, members", [(0, 7), (0, 96), (1, 7), (3, 7), (32, 7)])
def test_reported_tasks(G, members):
    _build.build()
    from paper_2308_06196_gb300.bgk import Batch, Solver

    ms = W.sod_members(members=members, seed=3, elements=(5, 400), degrees=(1, 3), nvs=(12, 15, 24))
    k = [W.mesh_kwargs(m) for m in ms]
    ss = [Solver(c["dim"], c["nelem"], c["lo"], c["hi"], c["p"], c["nv"], c["vlo"], c["vhi"], c["tau"], bc=m["bc"],
                 bc_state=m["bc_state"], chunks=1, vtiles_per_task=G) for c, m in zip(k, ms)]
    for s, m in zip(ss, ms):
        s.set_state(W.prim_sod(s.points(), m["left"], m["right"]))
    b = Batch(ss)
    assert b.tasks == sum(count(c, G, k) for c in k)
    b.step([s.dt(0.1) for s in ss], 1)
    b.synchronize()
    one = Batch(ss[:1])
    one.autotune()  # a measured length: one group per task, of one of the candidates
    nvt = tiles(k[0]["nv"])
    cands = [2, 4, 8, 16, 32, 64] + [-(-nvt // q) for q in (1, 2, 3, 4, 6, 8, 12, 16)]
    assert one.tasks in {count(k[0], g, k) for g in cands if 2 <= g <= 64}


@pytest.mark.parametrize("G, members", [(0, 9), (0, 60), (1, 9), (5, 9)])
def test_batch_equals_members_alone_bit_for_bit(G, members):
    """The batch shares the same moment groups out in tasks of its own length."""
    import numpy as np

    _build.build()
    from paper_2308_06196_gb300.bgk import Batch, Solver

    ms = W.sod_members(members=members, seed=8, elements=(5, 90), degrees=(1, 3), nvs=(12, 15, 24))

    def make():
        out = []
        for m in ms:
            c = W.mesh_kwargs(m)
            s = Solver(c["dim"], c["nelem"], c["lo"], c["hi"], c["p"], c["nv"], c["vlo"], c["vhi"], c["tau"], bc=m["bc"],
                       bc_state=m["bc_state"], chunks=1, vtiles_per_task=G)
            s.set_state(W.prim_sod(s.points(), m["left"], m["right"]))
            out.append(s)
        return out

    alone, members = make(), make()
    dt = [s.dt(0.1) for s in alone]
    b = Batch(members)
    b.step(dt, 3)
    b.synchronize()
    for s, t, h in zip(alone, members, dt):
        s.step(h, 3)
        for x, y in ((s.moments(), t.moments()), (s.equilibrium(), t.equilibrium()), (s.get_f(), t.get_f())):
            assert np.array_equal(x, y)
