"""Heat convolutions leave out the Legendre terms below 2^-100 (near the poles, high orders), the
spectra rows only such terms meet, and the order range of a ring's transform.  The plain transforms
keep every term, so analysis, e^{-t l(l+1)} and synthesis through them is the same operator with
nothing left out: the two agree to the rounding of the precision.  Sizes: no cut at all (33 rings), cuts
inside one chunk and past it (128, 200 with a narrow band limit, 321), a grid with both poles and a
HEALPix grid; odd field counts.  The bars are those of the transforms (1e-5, 1e-4 BF16x3, relative to
the largest value), since both sides round their sums."""
import numpy as np
import pytest

from tests.gpu_util import rel_max

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2605_18389_gb300 import shot  # noqa: E402

BAR = {shot.SHOT_FP32: 1e-5, shot.SHOT_TF32X3: 1e-5, shot.SHOT_BF16X3: 1e-4}


def _grid(kind, n, lmax, prec, mode):
    if kind == "cc":
        return shot.shot_grid_init_quad(shot.SHOT_QUAD_CLENSHAW_CURTIS, n, 2 * n, lmax, prec, mode)
    if kind == "hp":
        return shot.shot_grid_init_healpix(n, lmax, prec, mode)
    return shot.shot_grid_init(n, 2 * n, lmax, prec, mode)


@pytest.mark.parametrize("kind,n,lmax,nf", [("gl", 33, -1, 3), ("gl", 128, -1, 2), ("gl", 200, 90, 5),
                                            ("gl", 321, -1, 7), ("cc", 129, -1, 4), ("hp", 40, -1, 3)])
@pytest.mark.parametrize("prec,mode", [("FP32", "TABLE"), ("BF16X3", "TABLE"), ("TF32X3", "TABLE"),
                                       ("TF32X3", "RECURRENCE")])
def test_heat_with_polar_cut_matches_full_transforms(kind, n, lmax, nf, prec, mode):
    prec, mode = getattr(shot, "SHOT_" + prec), getattr(shot, "SHOT_" + mode)
    g = _grid(kind, n, lmax, prec, mode)
    try:
        L = shot.shot_grid_info(g)["lmax"] + 1
        npix = 12 * n * n if kind == "hp" else n * 2 * n
        shape = (nf, npix) if kind == "hp" else (nf, n, 2 * n)
        f = torch.from_numpy(np.random.default_rng([n, nf]).normal(size=shape).astype(np.float32)).cuda() + 1.0
        t = 2.0 / L ** 2   # the highest degrees keep a weight of e^-2
        # stale spectra of a call with nothing left out must not reach the heat convolution
        shot.shot_sht_analysis(g, torch.full_like(f, float("nan")), torch.empty((nf, L, L, 2), device="cuda"))
        out = torch.empty_like(f)
        shot.shot_heat_apply(g, t, f, out)
        c = torch.empty((nf, L, L, 2), device="cuda")
        shot.shot_sht_analysis(g, f, c)
        l = torch.arange(L, device="cuda", dtype=torch.float64)
        c *= torch.exp(-t * l * (l + 1)).float()[None, :, None, None]
        ref = torch.empty_like(f)
        shot.shot_sht_synthesis(g, c, ref)
        assert rel_max(out.cpu().numpy(), ref.cpu().numpy().astype(np.float64)) <= BAR[prec]
    finally:
        shot.shot_grid_free(g)


def test_plain_transforms_keep_every_term():
    """A field on the northernmost ring only: its coefficients of high order are tiny, not zero, where
    FP32 can hold them, and NaN in one ring reaches every coefficient and every node."""
    n = 128
    g = shot.shot_grid_init(n, 2 * n, -1, shot.SHOT_FP32)
    try:
        f = torch.zeros((1, n, 2 * n), device="cuda")
        f[0, 0, 0] = 1.0
        c = torch.empty((1, n, n, 2), device="cuda")
        shot.shot_sht_analysis(g, f, c)
        a = c[0, n - 1, :, 0].abs().cpu().numpy()
        assert np.all(a[:15] > 0) and a[14] < 1e-6 * a.max()
        f[0, 0, 0] = float("nan")
        shot.shot_sht_analysis(g, f, c)
        low = torch.tril(torch.ones((n, n), dtype=torch.bool, device="cuda"))
        assert bool(torch.isnan(c[0, :, :, 0][low]).all())
        out = torch.empty_like(f)
        shot.shot_heat_apply(g, 1e-3, f, out)
        assert bool(torch.isnan(out).all())
    finally:
        shot.shot_grid_free(g)
