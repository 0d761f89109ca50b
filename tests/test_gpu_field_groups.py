"""The solver's epilogue where several pairs of fields share a CTA (2, 3 or 6 pairs, a partial last group,
an equator ring), where the two fields of an element end differently, and where the persistent update
kernel takes several items a CTA on the compiled plans."""
import math
import os

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


def _cuda(a):
    return torch.from_numpy(a).cuda()


def _against_oracle(og, eps, tau, r, k, p, q, T, potentials=False):
    """Problem k of the solve r against the oracle's solve of the same pair."""
    ref = sk.sinkhorn(og, p[k:k + 1], q[k:k + 1], eps, tau, T=T, delta=0.0, C=10)
    assert ref["status"][0] == 0 and r["status"][k] == 0 and r["iters"][k] == T
    u, v = r["u"][k:k + 1].cpu().numpy(), r["v"][k:k + 1].cpu().numpy()
    if potentials:
        assert rel_max(u, ref["phi"]) < TOL and rel_max(v, ref["psi"]) < TOL
    elif math.isinf(tau):
        assert potentials_err(og, eps, u, v, ref["phi"], ref["psi"]) < TOL
    else:
        assert rel_max(eps * np.log(u), ref["phi"]) < TOL and rel_max(eps * np.log(v), ref["psi"]) < TOL
    np.testing.assert_allclose(r["ot"][k], ref["ot"][0], rtol=TOL)
    np.testing.assert_allclose(r["err"][k], ref["err"][0], rtol=1e-2, atol=1e-6)
    if not potentials:
        np.testing.assert_allclose(r["mass_pi"][k], ref["mass_pi"][0], rtol=TOL)


# 33 ring pairs of 130 longitudes: 29, 55 and 81 problems are the first odd counts of 2, 3 and 6 pairs a
# CTA; tau / eps = 1000 amplifies the rounding of the translation-invariant sum
@pytest.mark.parametrize("n,eps,tau", [(29, 0.05, math.inf), (55, 0.05, 1.0), (81, 0.05, math.inf), (81, 0.05, 1.0),
                                       (81, 0.01, 10.0)])
def test_several_pairs_a_cta_match_oracle(n, eps, tau):
    nlat, T = 65, 20
    og = OGrid(nlat)
    p, q = inputs.pairs("paper_uniform", 9000 + n, n, og.x, og.nlon, og.a_ring, masses=not math.isinf(tau))
    (p32, p64), (q32, q64) = f32(p), f32(q)
    pot = tau / eps > 100
    g = shot.shot_grid_init(nlat)
    try:
        rc, r = shot.shot_sinkhorn(g, _cuda(p32), _cuda(q32), eps, tau, max_iter=T, tol=0.0, check_every=10,
                                   flags=shot.SHOT_FLAG_POTENTIALS if pot else 0)
        assert rc == 0
        for k in (0, 1, n // 2, n - 2, n - 1):
            _against_oracle(og, eps, tau, r, k, p64, q64, T, pot)
    finally:
        shot.shot_grid_free(g)


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("how", ["nonpositive", "overflow"])
def test_partner_of_a_problem_that_stops(first, how):
    """Two problems share every element (30 problems on 16 ring pairs: pairs of fields); one stops, at the
    iteration at which the oracle stops it or because one value of u overflows, and the other gives what
    the oracle gives it alone."""
    nlat, T, n = 32, 20, 30
    eps = 4e-2 if how == "nonpositive" else 0.1
    og = OGrid(nlat)
    p, q = inputs.pairs("paper_uniform", 4711, n, og.x, og.nlon, og.a_ring)
    bad, good = first, 1 - first
    if how == "nonpositive":
        pv, qv = inputs.pairs("vmf3", 1001, 1, og.x, og.nlon, og.a_ring)
        p[bad], q[bad] = pv[0], qv[0]
    (p32, p64), (q32, q64) = f32(p), f32(q)
    g = shot.shot_grid_init(nlat)
    try:
        if how == "overflow":   # K v = 0.01 and p = 1e38 at one node
            p32[bad, 7, 11] = 1e38
            u, v = torch.ones((n, nlat, og.nlon), device="cuda"), torch.ones((n, nlat, og.nlon), device="cuda")
            v[bad] = 0.01
            rc, r = shot.shot_sinkhorn(g, _cuda(p32), _cuda(q32), eps, max_iter=T, tol=0.0, check_every=10,
                                       flags=shot.SHOT_FLAG_WARM_START, u=u, v=v)
            assert r["status"][bad] == shot.SHOT_ERR_NONFINITE and r["iters"][bad] == 1
        else:
            rc, r = shot.shot_sinkhorn(g, _cuda(p32), _cuda(q32), eps, max_iter=T, tol=0.0, check_every=10)
            ref = sk.sinkhorn(og, p64[bad:bad + 1], q64[bad:bad + 1], eps, T=T, delta=0.0, C=10)
            assert ref["status"][0] == sk.NONPOSITIVE
            assert r["status"][bad] == shot.SHOT_ERR_NONPOSITIVE and r["iters"][bad] == ref["iters"][0]
        assert rc < 0 and np.isnan(r["ot"][bad])
        _against_oracle(og, eps, math.inf, r, good, p64, q64, T)
    finally:
        shot.shot_grid_free(g)


# three and more items a CTA on 3 x 152 CTAs, an odd problem count (a half-empty last pair in the
# prefetch); 1440 and 1024 longitudes run compiled plans, 1000 the runtime one
@pytest.mark.parametrize("nlat,nlon,n,tau", [(720, 1440, 7, math.inf), (720, 1440, 7, 1.0), (512, 1024, 11, math.inf),
                                             (500, 1000, 11, 1.0)])
def test_persistent_update_with_several_items_a_cta(nlat, nlon, n, tau):
    """Bit for bit what one item a CTA gives (SHOT_IDFT_PERSISTENT=0), and the kernels that ran."""
    from torch.profiler import ProfilerActivity, profile
    og = OGrid(nlat, nlon)
    p, q = inputs.pairs("paper_uniform", 600 + n, n, og.x, og.nlon, og.a_ring, masses=not math.isinf(tau))
    pt, qt = _cuda(p.astype(np.float32)), _cuda(q.astype(np.float32))
    res = []
    for flag in ("1", "0"):
        os.environ["SHOT_IDFT_PERSISTENT"] = flag
        try:
            g = shot.shot_grid_init(nlat, nlon, 63)
        finally:
            del os.environ["SHOT_IDFT_PERSISTENT"]
        try:
            with profile(activities=[ProfilerActivity.CUDA]) as prof:
                rc, r = shot.shot_sinkhorn(g, pt, qt, 0.1, tau, max_iter=20, tol=0.0, check_every=10)
                torch.cuda.synchronize()
            assert rc == 0
            names = [e.key for e in prof.key_averages()]
            if any("k_reduce" in s for s in names):   # the profiler reports kernels here
                assert any("k_idft_p" in s for s in names) == (flag == "1"), names
            res.append([r["u"].cpu().numpy(), r["v"].cpu().numpy()] + [r[k] for k in ("ot", "ot_dual", "mass_pi", "err")])
        finally:
            shot.shot_grid_free(g)
    for a, b in zip(*res):
        np.testing.assert_array_equal(a, b)
