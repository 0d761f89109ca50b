"""The ring transforms take two fields an element and 1, 2, 3 or 6 pairs of fields a CTA, with the
twiddles in shared memory up to 768 longitudes and the persistent update kernel beyond.  Heat
convolutions against the oracle where each choice begins and ends, with odd field counts (a last pair
with one field) and an equator ring; the bar is the FP32 transforms' 1e-5 relative to the largest
value.  And the persistent kernel against the one item per CTA on a ring whose plan is not a
compiled one, bit for bit (the same sums in the same order), a frozen partner included."""
import math
import os

import numpy as np
import pytest

from oracle.grid import Grid as OGrid
from oracle import sht as osht
from paper_2605_18389_gb300 import inputs
from tests.gpu_util import f32, rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


@pytest.mark.parametrize("nlat,nlon,nf", [
    (3, 5, 1), (9, 17, 2), (24, 48, 121), (48, 96, 120), (96, 256, 61), (101, 307, 49), (129, 512, 29),
    (65, 768, 5), (65, 770, 5), (64, 1536, 3), (17, 4099, 2), (4, 6400, 3),
])
def test_heat_at_field_and_ring_edges(nlat, nlon, nf):
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
    for f in {0, nf // 2, nf - 1}:
        assert rel_max(got[f], osht.heat_apply(og, x64[f], 1e-3)) <= 1e-5


@pytest.mark.parametrize("pairs,tau", [(2, math.inf), (3, 1.0)])
def test_persistent_update_on_a_runtime_plan(pairs, tau):
    nlat = 391   # an equator ring; 782 longitudes = 2 * 17 * 23, generic stages
    og = OGrid(nlat)
    p, q = inputs.pairs("paper_uniform", 5100 + pairs, pairs, og.x, og.nlon, og.a_ring, masses=not math.isinf(tau))
    q[0, 5, 7] = np.nan   # the first pair stops as non-finite and stays frozen beside its neighbour
    pt, qt = (torch.from_numpy(a.astype(np.float32)).cuda() for a in (p, q))
    res = []
    for flag in ("1", "0"):
        os.environ["SHOT_IDFT_PERSISTENT"] = flag
        try:
            g = shot.shot_grid_init(nlat)
        finally:
            del os.environ["SHOT_IDFT_PERSISTENT"]
        try:
            u3 = torch.empty((3 * pairs, og.nlat, og.nlon), device="cuda")
            v3 = torch.empty_like(u3)
            _, r = shot.shot_divergence(g, pt, qt, 0.05, tau, max_iter=20, tol=0.0, check_every=10, u3=u3, v3=v3)
            res.append((u3.cpu().numpy(), v3.cpu().numpy(), np.array(r["S"]), np.array(r["status"])))
        finally:
            shot.shot_grid_free(g)
    assert res[0][3][0] < 0 and np.all(res[0][3][1:] >= 0)
    for a, b in zip(res[0], res[1]):
        np.testing.assert_array_equal(a, b)
