"""Edges of the FP32 Legendre kernel's tiles against the oracle: nodes and rows around one 64-row
CTA and one 32-row warp, terms around one chunk of 16, column counts around each tile width
(16, 32, 48, 64 columns, two a field) and past one column tile.  The bar is the FP32 transforms'
1e-5 relative to the largest value (App. B's quadrature sums of at most 140 terms: each rounds to
6e-8 of the partial sum)."""
import numpy as np
import pytest

from oracle.grid import Grid as OGrid
from oracle import sht as osht
from tests.gpu_util import f32, rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


@pytest.mark.parametrize("nlat,nlon,lmax,nf", [
    (2, 4, 1, 1), (30, 60, 29, 8), (32, 64, 31, 9), (33, 70, 32, 16), (34, 68, 20, 17), (62, 124, 61, 24),
    (66, 132, 65, 25), (127, 254, 126, 3), (130, 260, 129, 32), (140, 280, 139, 33),
])
def test_fp32_heat_at_tile_edges(nlat, nlon, lmax, nf):
    og = OGrid(nlat, nlon, lmax)
    x, x64 = f32(np.random.default_rng([nlat, nf]).normal(size=(nf, nlat, nlon)) + 1.0)
    g = shot.shot_grid_init(nlat, nlon, lmax)
    try:
        inp = torch.from_numpy(x).cuda()
        out = torch.empty_like(inp)
        shot.shot_heat_apply(g, 1e-3, inp, out)
        got = out.cpu().numpy()
    finally:
        shot.shot_grid_free(g)
    for f in {0, nf // 2, nf - 1}:
        assert rel_max(got[f], osht.heat_apply(og, x64[f], 1e-3)) <= 1e-5
