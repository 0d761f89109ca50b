"""Solves around the line between one field and two fields an element of the ring transforms, against the
oracle: one problem, the last count whose CTAs of one field are all resident (33 ring pairs, 13 problems) and the
first beyond it, rings on both sides of 3583 longitudes, the longest of which two CTAs of pairs share an SM,
and rings with a prime factor that a generic stage takes.  Balanced and unbalanced, an equator ring, a
marginal check."""
import math

import numpy as np
import pytest

from oracle.grid import Grid as OGrid
from oracle import sinkhorn as sk
from paper_2605_18389_gb300 import inputs
from tests.gpu_util import f32, potentials_err, rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402

TOL = 1e-5   # potentials, transport cost and mass of an FP32 solve against the oracle


@pytest.mark.parametrize("nlat,nlon,lmax,n,eps,fields", [
    (65, 135, 64, 1, 0.05, 1), (65, 135, 64, 13, 0.05, 1), (65, 135, 64, 14, 0.05, 2),
    (65, 130, 64, 1, 0.05, 1), (65, 130, 64, 13, 0.05, 2), (20, 802, 19, 1, 0.2, 2),
    (305, 3575, 20, 3, 0.5, 2), (305, 3584, 20, 3, 0.5, 1), (12, 6400, 11, 2, 0.5, 1),
])
@pytest.mark.parametrize("tau", [math.inf, 1.0])
def test_solve_matches_oracle(nlat, nlon, lmax, n, eps, fields, tau):
    T = 20
    og = OGrid(nlat, nlon, lmax)
    p, q = inputs.pairs("paper_uniform", 100 + n, n, og.x, og.nlon, og.a_ring, masses=not math.isinf(tau))
    (p32, p64), (q32, q64) = f32(p), f32(q)
    g = shot.shot_grid_init(nlat, nlon, lmax)
    try:
        assert shot.shot_grid_autotune(g, n)["idft_fg"] == fields
        rc, r = shot.shot_sinkhorn(g, torch.from_numpy(p32).cuda(), torch.from_numpy(q32).cuda(), eps, tau,
                                   max_iter=T, tol=0.0, check_every=10)
        assert rc == 0 and np.all(r["status"] == 0)
        k = [0, n - 1]
        ref = sk.sinkhorn(og, p64[k], q64[k], eps, tau, T=T, delta=0.0, C=10)
        u, v = r["u"].cpu().numpy()[k], r["v"].cpu().numpy()[k]
        if math.isinf(tau):
            assert potentials_err(og, eps, u, v, ref["phi"], ref["psi"]) < TOL
        else:
            assert rel_max(eps * np.log(u), ref["phi"]) < TOL and rel_max(eps * np.log(v), ref["psi"]) < TOL
        np.testing.assert_allclose(r["ot"][k], ref["ot"], rtol=TOL)
        np.testing.assert_allclose(r["mass_pi"][k], ref["mass_pi"], rtol=TOL)
        np.testing.assert_allclose(r["err"][k], ref["err"], rtol=1e-2, atol=1e-6)
    finally:
        shot.shot_grid_free(g)
