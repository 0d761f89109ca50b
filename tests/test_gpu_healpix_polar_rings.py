"""Plain synthesis on HEALPix grids with random coefficients of every order up to the highest band limit
(4 nside - 2): on the short rings near the poles many orders share a residue, and several threads share
the orders of a residue.  Against the oracle's direct sums; the bar is the FP32 transforms' 1e-5 relative
to the largest value.  Sizes: rings of 4 points only (nside 1), a longest ring below, at and above the CTA's
128 threads, one field and an odd last pair."""
import numpy as np
import pytest

from oracle.healpix import HealpixGrid
from tests.gpu_util import f32, rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


@pytest.mark.parametrize("nside,lmax,nf", [(1, 2, 1), (2, 6, 3), (3, 10, 2), (16, 62, 1), (31, 122, 3), (32, 126, 2),
                                           (40, 158, 1), (64, 40, 2)])
def test_synthesis_of_all_orders_matches_oracle(nside, lmax, nf):
    og = HealpixGrid(nside, lmax)
    L = lmax + 1
    c, c64 = f32(np.random.default_rng([nside, lmax]).normal(size=(nf, L, L, 2)) * np.tri(L)[None, :, :, None])
    c[:, :, 0, 1] = c64[:, :, 0, 1] = 0.0
    g = shot.shot_grid_init_healpix(nside, lmax)
    try:
        out = torch.empty((nf, og.npix), device="cuda")
        shot.shot_sht_synthesis(g, torch.from_numpy(c).cuda(), out)
        got = out.cpu().numpy()
    finally:
        shot.shot_grid_free(g)
    ref = og.synthesis(c64[..., 0] + 1j * c64[..., 1])[:, 0]
    for f in range(nf):
        assert rel_max(got[f], ref[f]) <= 1e-5
