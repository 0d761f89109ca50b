"""The sums that the solver's epilogue takes over a ring pair (Alg. 1's gauge and translation-invariant
sums, the marginal error): FP32 terms in short chains, joined in FP64 from at least eight partial sums,
whatever the number of threads that share a field.

The gauge makes the returned u sum to 1 over the nodes, so the FP64 sum of u shows the rounding of the
device's own sum.  The marginal below is 1.01 on the longitudes a thread meets first and 0.99 * 2^-23 on
the others: one plain FP32 chain a thread loses every later term (each is below half a unit in the last
place of 2.02), 8e-7 of the sum for eight longitudes a thread.  The bar is ten roundings of 2^-24: the factor
of u, its product with the buffer, and eight additions, the most that a term passes on rings of up to 768
longitudes and on HEALPix rings of 1024 points (13 on rings of 1440)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402


@pytest.mark.parametrize("kind,n,nlon,lmax,nf,width", [
    ("gl", 128, 256, -1, 45, 32),     # six pairs of fields a CTA
    ("gl", 129, 256, 100, 45, 32),    # the same with an equator ring (field by field)
    ("gl", 256, 512, -1, 25, 64),     # three
    ("gl", 128, 768, 100, 17, 96),    # two
    ("gl", 720, 1440, 100, 3, 192),   # one, persistent kernel
    ("gl", 720, 1440, 100, 1, 192),
    ("hp", 256, 0, 64, 3, 128),
])
def test_gauge_sum_keeps_small_terms(kind, n, nlon, lmax, nf, width):
    if kind == "hp":
        g = shot.shot_grid_init_healpix(n, lmax)
    else:
        g = shot.shot_grid_init(n, nlon, lmax)
    try:
        small = 0.99 * 2.0 ** -23
        if kind == "hp":
            ln, off, _ = shot.shot_grid_rings(g)
            p = np.full((nf, 12 * n * n), small, np.float32)
            for a, b in zip(off, ln):
                p[:, a:a + min(width, b)] = 1.01
        else:
            p = np.full((nf, n, nlon), small, np.float32)
            p[:, :, :width] = 1.01
        pt = torch.from_numpy(p).cuda()
        q = torch.ones_like(pt)
        rc, r = shot.shot_sinkhorn(g, pt, q, 4.0, max_iter=1, tol=0.0, check_every=0)
        assert rc == 0 and np.all(r["status"] == 0)
        s = r["u"].double().reshape(nf, -1).sum(1).cpu().numpy()
        assert np.max(np.abs(s - 1.0)) <= 10 * 2.0 ** -24, s
    finally:
        shot.shot_grid_free(g)
