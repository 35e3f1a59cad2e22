"""The Newton solve's integer conversions between FP32 and FP64 hand numbers outside their range (moments below
2^-60) to the hardware's: f times a power of two must give the same moments times it, exactly, and the same
perturbed state, in both forms of the solve, with velocities that are exactly zero among the inputs."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build

pytestmark = pytest.mark.gpu


def solve(f, nv, L):
    import torch
    from paper_2308_06196_gb300 import bgk

    f_dev = torch.from_numpy(f).cuda()
    Q = torch.full((len(f), 5), float("nan"), dtype=torch.float64, device="cuda")
    P = torch.full_like(Q, float("nan"))
    assert bgk.equilibrium_noalloc(f_dev, nv, (-L,) * 3, (L,) * 3, Q, P) == 0
    return Q.cpu().numpy(), P.cpu().numpy()


@pytest.mark.parametrize("npts", [50, 9729])
@pytest.mark.parametrize("nv", [(11, 12, 10), (13, 12, 1)])
def test_power_of_two_scaling(npts, nv):
    _build.build()
    L, m = 6.0, 2 if nv[2] == 1 else 3
    rng = np.random.default_rng(len(nv) + nv[2])
    v1 = [np.linspace(-L, L, n) if n > 1 else np.zeros(1) for n in nv]
    vz, vy, vx = np.meshgrid(v1[2], v1[1], v1[0], indexing="ij")
    v = np.stack([vx.ravel(), vy.ravel(), vz.ravel()], 1)
    u = rng.uniform(-0.3, 0.3, (50, 3))
    u[::3, :2] = 0.0
    th = rng.uniform(3.0, 4.0, 50)
    e = sum((v[None, :, d] - u[:, d, None]) ** 2 for d in range(m))
    f = np.exp(-e / (2 * th[:, None])) * np.where(np.arange(50) % 3 == 0, 1.0, 1.1)[:, None]
    f = np.resize(f.astype(np.float32), (npts, f.shape[1]))
    Q0, P0 = solve(f, nv, L)
    for k in (-70, 30):  # the smallest f, 2^-30, stays a normal number
        Q, P = solve(np.ldexp(f, k), nv, L)
        assert np.array_equal(Q, np.ldexp(Q0, k))
        P[:, 0] = np.ldexp(P[:, 0], -k)
        # alpha_0, at most 60 in size, is a double-float number: 60 2^-47 = 4e-13 in the residual of either
        # solve, times at most 30 for the 5 x 5 system
        assert np.all(np.abs(P - P0) <= 2 * 30 * 4.3e-13 * np.abs(P0).max(axis=0))
