"""Rings of 1440 and 1024 longitudes run plans compiled for them (four CTAs an SM; the persistent update
kernel): heat applications with odd field counts and a band limit far below the ring's, and solves, on few
rings with and without an equator ring, against the oracle at the FP32 bars (1e-5)."""
import math

import numpy as np
import pytest

from oracle.grid import Grid as OGrid
from oracle import sht as osht
from oracle import sinkhorn as sk
from paper_2605_18389_gb300 import inputs
from tests.gpu_util import f32, potentials_err, rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


@pytest.mark.parametrize("nlat,nlon,nf", [(17, 1440, 1), (17, 1440, 3), (16, 1024, 5), (33, 1024, 2)])
def test_heat_matches_oracle(nlat, nlon, nf):
    og = OGrid(nlat, nlon)
    x, x64 = f32(np.random.default_rng([nlat, nlon, nf]).normal(size=(nf, nlat, nlon)) + 1.0)
    g = shot.shot_grid_init(nlat, nlon)
    try:
        inp = torch.from_numpy(x).cuda()
        out = torch.empty_like(inp)
        shot.shot_heat_apply(g, 1e-3, inp, out)
        got = out.cpu().numpy()
    finally:
        shot.shot_grid_free(g)
    for f in range(nf):
        assert rel_max(got[f], osht.heat_apply(og, x64[f], 1e-3)) <= 1e-5


@pytest.mark.parametrize("nlat,nlon,n", [(17, 1440, 3), (16, 1024, 2), (17, 1024, 1)])
@pytest.mark.parametrize("tau", [math.inf, 1.0])
def test_solve_matches_oracle(nlat, nlon, n, tau):
    eps, T = 0.4, 20
    og = OGrid(nlat, nlon)
    p, q = inputs.pairs("paper_uniform", 70 + n, n, og.x, og.nlon, og.a_ring, masses=not math.isinf(tau))
    (p32, p64), (q32, q64) = f32(p), f32(q)
    g = shot.shot_grid_init(nlat, nlon)
    try:
        rc, r = shot.shot_sinkhorn(g, torch.from_numpy(p32).cuda(), torch.from_numpy(q32).cuda(), eps, tau,
                                   max_iter=T, tol=0.0, check_every=10)
        ref = sk.sinkhorn(og, p64, q64, eps, tau, T=T, delta=0.0, C=10)
        assert rc == 0 and np.all(r["status"] == 0)
        u, v = r["u"].cpu().numpy(), r["v"].cpu().numpy()
        if math.isinf(tau):
            assert potentials_err(og, eps, u, v, ref["phi"], ref["psi"]) < 1e-5
        else:
            assert rel_max(eps * np.log(u), ref["phi"]) < 1e-5 and rel_max(eps * np.log(v), ref["psi"]) < 1e-5
        np.testing.assert_allclose(r["ot"], ref["ot"], rtol=1e-5)
        np.testing.assert_allclose(r["mass_pi"], ref["mass_pi"], rtol=1e-5)
        np.testing.assert_allclose(r["err"], ref["err"], rtol=1e-2, atol=1e-6)
    finally:
        shot.shot_grid_free(g)
