"""The moments pass of bgk_equilibrium_noalloc at the sizes where its tiling can go wrong: velocity counts
below one thread's share, an exact multiple of the 2048-velocity group, one velocity
past it, point counts around its batches of six, an f that starts off a 16-byte boundary."""
import numpy as np
import pytest

from paper_2308_06196_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv, npts, shift", [
    ((5, 7, 9), 1, 0), ((5, 7, 9), 13, 0), ((16, 16, 8), 6, 0), ((16, 16, 8), 7, 1), ((13, 13, 13), 5, 0),
    ((12, 12, 12), 3000, 0), ((32, 32, 1), 11, 0), ((9, 9, 1), 2, 3), ((24, 24, 24), 12, 2)])
def test_moments_match_plain_sums(nv, npts, shift):
    import torch

    _build.build()
    from paper_2308_06196_gb300 import bgk

    L, m = 6.0, 2 if nv[2] == 1 else 3
    rng = np.random.default_rng(npts)
    v1 = [np.linspace(-L, L, n) if n > 1 else np.zeros(1) for n in nv]
    w1 = [np.r_[0.5, np.ones(n - 2), 0.5] * 2 * L / (n - 1) if n > 1 else np.ones(1) for n in nv]
    vz, vy, vx = np.meshgrid(v1[2], v1[1], v1[0], indexing="ij")
    w = (w1[2][:, None, None] * w1[1][None, :, None] * w1[0]).ravel()
    v = np.stack([vx.ravel(), vy.ravel(), vz.ravel()], 1)
    u = rng.uniform(-0.3, 0.3, (npts, 3))
    th = rng.uniform(3.0, 4.0, npts)  # wide enough for the coarsest grid here
    e = sum((v[None, :, d] - u[:, d, None]) ** 2 for d in range(m))
    f = (np.exp(-e / (2 * th[:, None])) * rng.uniform(0.9, 1.1, (npts, len(w)))).astype(np.float32)
    buf = torch.zeros(f.size + 8, dtype=torch.float32, device="cuda")
    f_dev = buf[shift:shift + f.size].view(npts, len(w))
    f_dev.copy_(torch.from_numpy(f))
    Q = torch.full((npts, 5), float("nan"), dtype=torch.float64, device="cuda")
    P = torch.full_like(Q, float("nan"))
    assert bgk.equilibrium_noalloc(f_dev, nv, (-L,) * 3, (L,) * 3, Q, P) == 0
    psi = np.concatenate([np.ones((len(w), 1)), v, 0.5 * (v**2).sum(1, keepdims=True)], 1)
    ref, size = f.astype(float) @ (w[:, None] * psi), f.astype(float) @ (w[:, None] * np.abs(psi))
    # 8 FMAs per thread, 5 + 8 adds across the warp and the CTA, each at most half an ulp of a sum that is
    # bounded by sum w |psi| f; the same for the index-basis sums that mix into a component (a factor 2)
    assert np.all(np.abs(Q.cpu().numpy() - ref) <= 2 * 21 * 2.0**-24 * size)
