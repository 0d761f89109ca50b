"""HEALPix grids whose longest ring does not fit an SM's shared memory as two sequences of field pairs
(4 nside above 7200): one field an element.  A field of few orders on rings of the exact ring geometry is
its own expected value up to the sums over latitude, which are formed here in FP64; the bar is the FP32
transforms' 1e-5 relative to the largest value.  Nside 1024 runs the pairs on the same field (rings past
the 1024 points up to which twiddles are copied into shared memory)."""
import numpy as np
import pytest

from oracle.healpix import ring_geometry
from oracle.legendre import pbar

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402

ORDERS = (0, 1, 2, 40)


def _field(z, npx, phi0, g, dev):
    """sum_m g[m](ring) cos(m phi) on the pixels, FP64."""
    n = torch.from_numpy(npx).to(dev)
    ring = torch.repeat_interleave(torch.arange(len(z), device=dev), n)
    first = torch.cumsum(n, 0) - n
    j = torch.arange(int(npx.sum()), device=dev) - first[ring]
    phi = torch.from_numpy(phi0).to(dev)[ring] + 2 * np.pi * j / n[ring]
    return sum(torch.from_numpy(g[m]).to(dev)[ring] * torch.cos(m * phi) for m in ORDERS)


@pytest.mark.parametrize("nside,nf", [(1024, 2), (2048, 1), (2048, 2)])
def test_heat_and_transforms_of_few_orders(nside, nf):
    lmax, t = 64, 1e-4
    z, npx, phi0 = ring_geometry(nside)
    st = np.sqrt(1.0 - z * z)
    g = {0: 1.0 + 0.5 * z, 1: 0.3 * st * z, 2: 0.2 * st ** 2, 40: st ** 40}
    P = pbar(lmax, z)
    area = 4 * np.pi / (12.0 * nside ** 2)
    want, coef = {}, {}
    for m in ORDERS:
        # F_m = n g_m / 2 for m > 0 (n g_0 for m = 0); the field is g_0 + 2 Re sum G_m e^{i m phi}
        coef[m] = P[m] @ (area * npx * g[m]) * (1.0 if m == 0 else 0.5)
        l = np.arange(m, lmax + 1)
        want[m] = (np.exp(-t * l * (l + 1)) * coef[m]) @ P[m] * (1.0 if m == 0 else 2.0)
    grid = shot.shot_grid_init_healpix(nside, lmax)
    try:
        f = _field(z, npx, phi0, g, "cuda").float()
        w = _field(z, npx, phi0, want, "cuda")
        scale = 1.0 + torch.arange(nf, device="cuda")
        x = (scale[:, None] * f[None]).contiguous()
        out = torch.empty_like(x)
        shot.shot_heat_apply(grid, t, x, out)
        for i in range(nf):
            assert float((out[i].double() - (1 + i) * w).abs().max() / w.abs().max()) <= 1e-5 * (1 + i)
        c = torch.empty((nf, lmax + 1, lmax + 1, 2), device="cuda")
        shot.shot_sht_analysis(grid, x, c)
        ref = np.zeros((lmax + 1, lmax + 1))
        for m in ORDERS:
            ref[m:, m] = coef[m]
        got = c.double().cpu().numpy()
        for i in range(nf):
            assert np.max(np.abs(got[i, :, :, 0] - (1 + i) * ref)) <= 1e-5 * (1 + i) * np.max(np.abs(ref))
            assert np.max(np.abs(got[i, :, :, 1])) <= 1e-5 * (1 + i) * np.max(np.abs(ref))
        # the plain synthesis of damped coefficients is the heat convolution
        l = torch.arange(lmax + 1, device="cuda", dtype=torch.float64)
        c *= torch.exp(-t * l * (l + 1)).float()[None, :, None, None]
        shot.shot_sht_synthesis(grid, c, out)
        assert float((out[0].double() - w).abs().max() / w.abs().max()) <= 1e-5
    finally:
        shot.shot_grid_free(grid)


def test_solve_at_nside_2048():
    """One field an element through the update, the check and the final pass: on constant measures of
    unit mass the plan has mass 1, and u (K v) = p at every node."""
    nside = 2048
    grid = shot.shot_grid_init_healpix(nside, 32)
    try:
        p = torch.full((1, 12 * nside ** 2), 1 / (4 * np.pi), device="cuda")
        rc, r = shot.shot_sinkhorn(grid, p, p, 0.1, max_iter=4, tol=0.0, check_every=2)
        assert rc == 0 and r["status"][0] == 0
        assert abs(r["mass_pi"][0] - 1.0) <= 1e-5 and r["err"][0] <= 1e-5
    finally:
        shot.shot_grid_free(grid)


def test_longer_rings_are_refused():
    nside = 3700
    grid = shot.shot_grid_init_healpix(nside, 1)
    try:
        x = torch.ones((1, 12 * nside ** 2), device="cuda")
        with pytest.raises(shot.ShotError) as e:
            shot.shot_heat_apply(grid, 1e-3, x, torch.empty_like(x))
        assert e.value.code == shot.SHOT_ERR_UNSUPPORTED
    finally:
        shot.shot_grid_free(grid)
