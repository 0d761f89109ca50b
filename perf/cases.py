"""Workloads that stand for what users of this package run, with their inputs, one pass through the
public entry points, the work that a pass cannot do without, and its result in 64 bits.

A case is a dict of plain values:
  kind     "heat" (shot_heat_apply), "sht" (shot_sht_analysis and shot_sht_synthesis), "sinkhorn"
           (shot_sinkhorn), "divergence" (shot_divergence), "multi" (shot_divergence_multi) or
           "grad" (shot_divergence_grad)
  grid     "gl" (Gauss-Legendre), "cc" (Clenshaw-Curtis) or "healpix"; nlat (nside on HEALPix), nlon
  prec     "fp32", "bf16x3" or "tf32x3";  mode "table" or "recurrence"
  nf       fields of a transform, or pairs of measures of a solve
  t        heat time (a solve's eps is 4 t);  tau the marginal penalty (0: balanced)
  T        iterations;  season: amplitude of the fields' zonal modulation;  ck: checkpoint interval
"""
import math

import numpy as np
import torch

from paper_2605_18389_gb300 import shot

PREC = {"fp32": shot.SHOT_FP32, "bf16x3": shot.SHOT_BF16X3, "tf32x3": shot.SHOT_TF32X3}
MODE = {"table": shot.SHOT_TABLE, "recurrence": shot.SHOT_RECURRENCE}
CHECK_EVERY = 10          # marginal check interval of the solves, as in the package's benchmark
MULTI_GRIDS = (64, 96, 128, 180)
MULTI_TAUS = (0.1, 1.0, 10.0)
MASSES = (0.5, 2.0)       # range of the masses of unbalanced problems


def _heat(name, grid, nlat, nlon, prec, nf, t, mode="table"):
    return {"name": name, "kind": "heat", "grid": grid, "nlat": nlat, "nlon": nlon, "prec": prec, "mode": mode,
            "nf": nf, "t": t}


def _solve(name, kind, grid, nlat, nlon, prec, nf, t, tau, T, season, ck=0):
    return {"name": name, "kind": kind, "grid": grid, "nlat": nlat, "nlon": nlon, "prec": prec, "mode": "table",
            "nf": nf, "t": t, "tau": tau, "T": T, "season": season, "ck": ck}


def listed():
    return [
        # smoothing one small map: nothing but launches and latency
        _heat("heat_32_one", "gl", 32, 64, "fp32", 1, 1e-2),
        # a ragged grid (a prime ring length, an odd number of rings and of fields)
        _heat("heat_97_ragged", "gl", 97, 202, "bf16x3", 7, 2e-3),
        # the operator of the gradient workload, in plain FP32
        _heat("heat_256_fp32", "gl", 256, 512, "fp32", 32, 1e-3),
        # the operator of the benchmark's headline: 24 problems on the large grid
        _heat("heat_720_tf32x3", "gl", 720, 1440, "tf32x3", 24, 1e-4),
        # the same without a table, for programs that keep memory small
        _heat("heat_720_recurrence", "gl", 720, 1440, "tf32x3", 24, 1e-4, "recurrence"),
        # spectral analysis and synthesis of maps on the equiangular grid of the runtime experiment
        {"name": "sht_cc512", "kind": "sht", "grid": "cc", "nlat": 512, "nlon": 1024, "prec": "fp32",
         "mode": "table", "nf": 8},
        # one balanced transport problem on the smallest grid that is solved in earnest
        _solve("sinkhorn_32", "sinkhorn", "gl", 32, 64, "fp32", 1, 4e-2, 0.0, 60, 0.05),
        # climate maps: unbalanced transport on HEALPix nside 64, eps = 0.01, tau = 100
        _solve("sinkhorn_healpix64", "sinkhorn", "healpix", 64, 0, "fp32", 8, 2.5e-3, 100.0, 50, 0.1),
        # the benchmark's headline solve (8 pairs, 24 problems), shortened, in the accurate split form
        _solve("divergence_720_tf32x3", "divergence", "gl", 720, 1440, "tf32x3", 8, 1e-4, 0.0, 40, 0.02),
        # the same solve unbalanced in plain FP32, the form that the split ones are compared with
        _solve("divergence_720_fp32", "divergence", "gl", 720, 1440, "fp32", 8, 1e-4, 1.0, 30, 0.02),
        # many pairs on uneven grids in one solve: 4 grids x 3 penalties x 8 pairs
        _solve("multi_64_180", "multi", "gl", 0, 0, "fp32", 8, 2.5e-3, 0.0, 40, 0.1),
        # the gradient through the unrolled iterations, 16 pairs of unequal mass as in the regional
        # attribution of climate maps (eps = 0.01), checkpoints every 20
        _solve("grad_256", "grad", "gl", 256, 512, "fp32", 16, 2.5e-3, 1.0, 60, 0.05, 20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["heat", "heat", "heat", "sht", "sinkhorn", "divergence", "grad"])
        grid = rng.choice(["gl", "gl", "gl", "cc", "healpix"])
        if grid == "healpix":
            nlat, nlon = _log_int(rng, 6, 128), 0
            lmax = 3 * nlat - 1
        else:
            nlat = _log_int(rng, 16, 720)
            nlon = 2 * nlat + rng.choice([0, 0, 0, rng.randint(0, 32)])
            lmax = nlat - 1
        # 40 = t lmax^2: the band limit resolves the kernel, as at the listed sizes
        c = {"kind": kind, "grid": grid, "nlat": nlat, "nlon": nlon, "prec": rng.choice(sorted(PREC)),
             "mode": "recurrence" if kind == "heat" and rng.random() < 0.2 else "table",
             "nf": _log_int(rng, 1, 48 if kind == "heat" else 8)}
        if kind != "sht":
            c["t"] = 40.0 / max(lmax, 15) ** 2
        if kind in ("sinkhorn", "divergence", "grad"):
            c["tau"] = rng.choice([0.0, 0.0, 1.0])
            c["T"] = rng.choice([10, 20, 35])
            # a modulation whose potentials stay within the FP32 range of the scalings
            c["season"] = min(0.05, 50.0 * c["t"])
            c["ck"] = 10
            if kind == "grad":   # FP32, as in the gradient workload
                c["prec"], c["tau"], c["t"] = "fp32", 1.0, max(c["t"], 2.5e-3)
        if work(c)["flops"] <= top:
            return c


# ---- geometry, inputs -------------------------------------------------------------------

_geometry = {}   # node positions and weights, by grid and size


def geometry(grid, nlat, nlon):
    """Rings in order from north: x = cos(theta), length, longitude of the first node, area weight
    of a node (FP64), band limit."""
    key = (grid, nlat, nlon)
    if key in _geometry:
        return _geometry[key]
    if grid == "healpix":
        nside, nr = nlat, 4 * nlat - 1
        k = np.minimum(np.arange(1, nr + 1), nr + 1 - np.arange(1, nr + 1))
        cap = k < nside
        z = np.where(cap, 1.0 - k * k / (3.0 * nside * nside), 4.0 / 3.0 - 2.0 * k / (3.0 * nside))
        x = np.where(np.arange(1, nr + 1) <= 2 * nside, z, -z)
        x[2 * nside - 1] = 0.0
        length = np.where(cap, 4 * k, 4 * nside)
        phi0 = np.where(cap, np.pi / (4.0 * k), np.pi * (2 - (k - nside + 1) % 2) / (4.0 * nside))
        a = np.full(nr, 4.0 * np.pi / (12 * nside * nside))
        g = (x, length, phi0, a, 3 * nside - 1)
    else:
        if grid == "gl":
            # Newton's method on the Legendre polynomial of degree nlat
            x = np.cos(np.pi * (np.arange(1, nlat + 1) - 0.25) / (nlat + 0.5))
            for _ in range(8):
                p0, p1 = np.ones_like(x), x.copy()
                for l in range(2, nlat + 1):
                    p0, p1 = p1, ((2 * l - 1) * x * p1 - (l - 1) * p0) / l
                dp = nlat * (p0 - x * p1) / (1.0 - x * x)
                x = x - p1 / dp
            w = 2.0 / ((1.0 - x * x) * dp * dp)
        else:
            n = nlat - 1
            j = np.arange(nlat)
            x = np.cos(np.pi * j / n)
            w = np.ones(nlat)
            for k in range(1, n // 2 + 1):
                b = 1.0 if 2 * k == n else 2.0
                w -= b * np.cos(2.0 * np.pi * ((k * j) % n) / n) / (4.0 * k * k - 1.0)
            w *= np.where((j == 0) | (j == n), 1.0, 2.0) / n
        g = (x, np.full(nlat, nlon), np.zeros(nlat), w * 2.0 * np.pi / nlon, nlat - 1)
    _geometry[key] = g
    return g


def _node_maps(case, nlat=None, nlon=None):
    """Area weight and latitude of every node of a field, FP64 on the GPU."""
    x, length, _, a, _ = geometry(case["grid"], nlat or case["nlat"], nlon or case["nlon"])
    rep = torch.from_numpy(length.astype(np.int64)).cuda()
    return (torch.from_numpy(a).cuda().repeat_interleave(rep),
            torch.from_numpy(np.arcsin(np.clip(x, -1.0, 1.0))).cuda().repeat_interleave(rep))


def _shape(case, nlat=None, nlon=None):
    return (-1,) if case["grid"] == "healpix" else (nlat or case["nlat"], nlon or case["nlon"])


def _measures(case, gen, count, nlat=None, nlon=None, masses=None):
    """`count` positive fields: U(0, 1) per node (the runtime experiment's) on a background, times a
    seasonal zonal modulation 1 + season cos(lat - lat0), normalised to unit mass (times U[masses])."""
    a, lat = _node_maps(case, nlat, nlon)
    f = torch.rand(count, a.numel(), generator=gen, device="cuda", dtype=torch.float32).double()
    f = 0.05 + 0.95 * f
    if case.get("season"):
        lat0 = (torch.rand(count, 1, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * math.radians(23.5)
        f = f * (1.0 + case["season"] * torch.cos(lat - lat0))
    f = f / (f * a).sum(1, keepdim=True)
    if masses:
        lo, hi = masses
        f = f * (lo + (hi - lo) * torch.rand(count, 1, generator=gen, device="cuda", dtype=torch.float64))
    return f.float().reshape(count, *_shape(case, nlat, nlon)).contiguous()


def inputs(case, seed):
    """The tensors a program has in hand before the call."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, nf = case["kind"], case["nf"]
    if kind == "heat":
        # maps of both signs with a mean, as anomalies and scalings have
        n = _node_maps(case)[0].numel()
        f = torch.randn(nf, n, generator=gen, device="cuda") * 0.5 + 1.0
        return {"f": f.reshape(nf, *_shape(case)).contiguous()}
    if kind == "sht":
        n = _node_maps(case)[0].numel()
        lmax = geometry(case["grid"], case["nlat"], case["nlon"])[4]
        f = torch.randn(nf, n, generator=gen, device="cuda").reshape(nf, *_shape(case)).contiguous()
        l = torch.arange(lmax + 1, device="cuda")
        c = torch.randn(nf, lmax + 1, lmax + 1, 2, generator=gen, device="cuda")
        c = c * (l[:, None] >= l[None, :])[None, :, :, None]   # entries [l][m], m <= l
        c = c / (1.0 + l.float())[None, :, None, None]         # a falling spectrum
        c[:, :, 0, 1] = 0.0
        return {"f": f, "c": c.contiguous()}
    if kind == "multi":
        return {"sets": [{"nlat": n, "tau": tau, "p": _measures(case, gen, nf, n, 2 * n, MASSES),
                          "q": _measures(case, gen, nf, n, 2 * n, MASSES)} for n in MULTI_GRIDS for tau in MULTI_TAUS]}
    # unequal masses under a marginal penalty; the gradient keeps its scalings in FP32, which bounds
    # how far apart they may be
    mp = mq = MASSES if case["tau"] else None
    if kind == "grad":
        mp, mq = (1.05, 1.2), (0.8, 0.95)
    return {"p": _measures(case, gen, nf, masses=mp), "q": _measures(case, gen, nf, masses=mq)}


class Handle:
    """A grid handle that is released with its owner."""

    def __init__(self, case, nlat=None, nlon=None):
        nlat, nlon = nlat or case["nlat"], nlon or case["nlon"]
        p, m = PREC[case["prec"]], MODE[case["mode"]]
        if case["grid"] == "healpix":
            self.h = shot.shot_grid_init_healpix(nlat, -1, p, m)
        elif case["grid"] == "cc":
            self.h = shot.shot_grid_init_quad(shot.SHOT_QUAD_CLENSHAW_CURTIS, nlat, nlon, -1, p, m)
        else:
            self.h = shot.shot_grid_init(nlat, nlon, -1, p, m)

    def __del__(self):
        h, self.h = getattr(self, "h", None), None
        if h is not None:
            shot.shot_grid_free(h)


def prepare(case, seed):
    s = inputs(case, seed)
    s["case"] = case
    if case["kind"] == "multi":
        s["handles"] = {n: Handle(case, n, 2 * n) for n in MULTI_GRIDS}
        for st in s["sets"]:
            st["grid"] = s["handles"][st["nlat"]].h
            st["eps"] = 4.0 * case["t"]
        return s
    s["g"] = Handle(case)
    if case["kind"] == "heat":
        s["out"] = torch.empty_like(s["f"])
    elif case["kind"] == "sht":
        s["coef_out"], s["field_out"] = torch.empty_like(s["c"]), torch.empty_like(s["f"])
    elif case["kind"] == "sinkhorn":
        s["u"], s["v"] = torch.empty_like(s["p"]), torch.empty_like(s["p"])
    elif case["kind"] == "divergence":
        shape = (3 * case["nf"],) + tuple(s["p"].shape[1:])
        s["u"], s["v"] = torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")
    return s


def _scalars(*arrays):
    """The solve's scalars in one FP32 array: they come from FP32 fields."""
    return np.stack([np.asarray(a) for a in arrays]).astype(np.float32)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "heat":
        shot.shot_heat_apply(s["g"].h, case["t"], s["f"], s["out"])
        return s["out"]
    if kind == "sht":
        shot.shot_sht_analysis(s["g"].h, s["f"], s["coef_out"])
        shot.shot_sht_synthesis(s["g"].h, s["c"], s["field_out"])
        return {"coeffs": s["coef_out"], "fields": s["field_out"]}
    if kind == "multi":
        _, outs = shot.shot_divergence_multi(s["sets"], max_iter=case["T"], tol=0.0, check_every=CHECK_EVERY)
        return {"S": _scalars(*[x for o in outs for x in (o["S"], o["S_dual"])]),
                "status": np.stack([o["status"] for o in outs])}
    eps, tau = 4.0 * case["t"], case["tau"] or math.inf
    if kind == "grad":
        _, r = shot.shot_divergence_grad(s["g"].h, s["p"], s["q"], eps, tau, case["T"], case["ck"])
        return {"grad": r["grad"], "S": _scalars(r["S"]), "status": r["status"]}
    if kind == "sinkhorn":
        _, r = shot.shot_sinkhorn(s["g"].h, s["p"], s["q"], eps, tau, case["T"], 0.0, CHECK_EVERY,
                                  shot.SHOT_FLAG_POTENTIALS, s["u"], s["v"])
        return {"phi": r["u"], "psi": r["v"], "scalars": _scalars(r["ot"], r["ot_dual"], r["mass_pi"]),
                "status": r["status"], "iters": r["iters"]}
    _, r = shot.shot_divergence(s["g"].h, s["p"], s["q"], eps, tau, case["T"], 0.0, CHECK_EVERY,
                                shot.SHOT_FLAG_POTENTIALS, s["u"], s["v"])
    ot = r["ot3"].reshape(3, -1)
    return {"phi": s["u"], "psi": s["v"], "scalars": _scalars(*ot, r["S"], r["S_dual"]), "status": r["status"],
            "iters": r["iters3"]}


# ---- the work of a pass --------------------------------------------------------------------

def _operator_flops(grid, nlat, nlon, nf):
    """One heat convolution of nf fields: both Legendre contractions over the folded hemisphere and
    the ring transforms (2.5 n log2 n a real transform)."""
    x, length, _, _, lmax = geometry(grid, nlat, nlon)
    rows, nh = (lmax + 1) * (lmax + 2) // 2, (len(x) + 1) // 2
    fft = float(np.sum(2.5 * length * np.log2(np.maximum(length, 2))))
    return 2.0 * (2.0 * rows * nh * 2 * nf) + 2.0 * fft * nf, int(length.sum())


def work(case):
    kind, nf = case["kind"], case["nf"]
    if kind == "multi":
        f = b = 0.0
        for n in MULTI_GRIDS:
            fl, npix = _operator_flops("gl", n, 2 * n, 3 * nf * len(MULTI_TAUS))
            f += fl * 2 * case["T"]
            b += 8.0 * nf * len(MULTI_TAUS) * npix
        return {"bytes": b, "flops": f}
    if kind in ("heat", "sht"):
        fl, npix = _operator_flops(case["grid"], case["nlat"], case["nlon"], nf)
        lmax = geometry(case["grid"], case["nlat"], case["nlon"])[4]
        return {"bytes": 8.0 * nf * npix + (16.0 * nf * (lmax + 1) ** 2 if kind == "sht" else 0.0), "flops": fl}
    probs = {"sinkhorn": 1, "divergence": 3, "grad": 3}[kind] * nf
    fl, npix = _operator_flops(case["grid"], case["nlat"], case["nlon"], probs)
    steps = 2.0 * case["T"]
    if kind == "grad":   # two problems a pair are differentiated: one adjoint convolution for each
        steps += 2.0 * case["T"] * 2.0 / 3.0
        return {"bytes": 12.0 * nf * npix, "flops": fl * steps}
    return {"bytes": (8.0 * nf + 8.0 * probs) * npix, "flops": fl * steps}


# ---- the results in 64 bits ---------------------------------------------------------------

class Operator:
    """The transforms and the heat convolution of a grid in FP64 (torch), straight from their
    definitions: ring Fourier sums, orthonormal associated Legendre functions, quadrature."""

    def __init__(self, grid, nlat, nlon):
        x, length, phi0, a, lmax = geometry(grid, nlat, nlon)
        self.L, self.nr = lmax + 1, len(x)
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.a = torch.from_numpy(a).to(dev)
        self.rep = torch.from_numpy(length.astype(np.int64)).to(dev)
        self.area = self.a.repeat_interleave(self.rep)
        self.nlon = None if grid == "healpix" else nlon
        xs = torch.from_numpy(x).to(dev)
        st = torch.sqrt((1.0 - xs) * (1.0 + xs))
        m = torch.arange(self.L, device=dev, dtype=torch.float64)[:, None]
        pmm = torch.full((self.L, self.nr), 1.0 / math.sqrt(4.0 * math.pi), device=dev, dtype=torch.float64)
        for k in range(1, self.L):
            pmm[k] = -math.sqrt((2.0 * k + 1.0) / (2.0 * k)) * st * pmm[k - 1]
        self.P = torch.zeros(self.L, self.L, self.nr, device=dev, dtype=torch.float64)   # [m][l][ring]
        p2, p1 = torch.zeros_like(pmm), torch.zeros_like(pmm)
        for l in range(self.L):
            lm = m[:l + 1]
            new = torch.zeros_like(pmm)
            if l > 0:
                al = torch.sqrt((4.0 * l * l - 1.0) / (l * l - lm[:l] ** 2))
                be = (torch.sqrt(((l - 1.0) ** 2 - lm[:l] ** 2).clamp_min(0.0) / (4.0 * (l - 1.0) ** 2 - 1.0))
                      if l > 1 else 0.0)
                new[:l] = al * (xs * p1[:l] - be * p2[:l])
            new[l] = pmm[l]
            self.P[:, l] = new
            p2, p1 = p1, new
        if self.nlon is None:   # rings of their own length and first longitude: padded Fourier matrices
            nmax = int(length.max())
            k = torch.arange(nmax, device=dev, dtype=torch.float64)[None]
            lon = torch.from_numpy(phi0).to(dev)[:, None] + 2.0 * math.pi * k / self.rep.double()[:, None]
            self.keep = (k < self.rep[:, None])
            e = torch.polar(torch.ones((), device=dev, dtype=torch.float64).expand(self.nr, nmax, self.L),
                            lon[:, :, None] * m.T[None])
            self.E = e * self.keep[:, :, None]

    def fourier(self, f):
        """[nf, nodes] -> [ring, nf, m], sum over the ring of f e^{-i m phi}"""
        if self.nlon is not None:
            return torch.fft.rfft(f.reshape(f.shape[0], self.nr, self.nlon))[..., :self.L].transpose(0, 1)
        pad = torch.zeros(f.shape[0], *self.keep.shape, device=f.device, dtype=f.dtype)
        pad = pad.masked_scatter(self.keep.expand_as(pad), f)
        return torch.bmm(pad.transpose(0, 1).to(self.E.dtype), self.E.conj())

    def fields(self, G):
        """[ring, nf, m] -> [nf, nodes], Re G_0 + 2 Re sum G_m e^{i m phi}"""
        if self.nlon is not None:
            f = torch.fft.irfft(G.transpose(0, 1), n=self.nlon, norm="forward")
            return f.reshape(f.shape[0], -1)
        w = torch.full((self.L,), 2.0, device=G.device, dtype=torch.float64)
        w[0] = 1.0
        f = torch.bmm(G * w, self.E.transpose(1, 2)).real.transpose(0, 1)
        return f[self.keep.expand_as(f)].reshape(G.shape[1], -1)

    def analysis(self, f):
        """[nf, nodes] -> [m, l, 2 nf] (real parts, then imaginary ones)"""
        F = (self.fourier(f) * self.a[:, None, None]).permute(2, 0, 1)
        return torch.bmm(self.P, torch.cat([F.real, F.imag], 2))

    def synthesis(self, c):
        G = torch.bmm(self.P.transpose(1, 2), c)
        nf = c.shape[2] // 2
        return self.fields(torch.complex(G[..., :nf], G[..., nf:]).permute(1, 2, 0))

    def heat(self, f, t):
        l = torch.arange(self.L, device=f.device, dtype=torch.float64)
        return self.synthesis(self.analysis(f) * torch.exp(-t * l * (l + 1.0))[None, :, None])


def _sinkhorn64(op, p, q, eps, tau, T):
    """Potentials after T iterations, and each problem's cost, cost - eps mass, and mass."""
    # u = e^la u', v = e^lb v' with u', v' of mean 1: unbalanced scalings outgrow even FP64
    t, a = eps / 4.0, op.area
    u, v = torch.ones_like(p), torch.ones_like(q)
    bal = torch.isinf(tau)
    gamma = torch.where(bal, torch.ones_like(tau), tau / (tau + eps))
    et = torch.where(bal, torch.zeros_like(tau), eps / tau)
    tf = torch.where(bal, torch.ones_like(tau), tau)
    la, lb = torch.zeros_like(tau), torch.zeros_like(tau)
    total = lambda x: x.sum(1, keepdim=True)   # noqa: E731

    def half(m, x, lx):
        w = (m / op.heat(x, t)) ** gamma
        mean = w.mean(1, keepdim=True)
        return w / mean, torch.log(mean) - gamma * lx

    for _ in range(T):
        u, la = half(p, v, lb)
        v, lb = half(q, u, la)
        c = torch.where(bal, -(la + torch.log(total(u))),
                        0.5 * tf / eps * (torch.log(total(a * p * u ** -et)) - et * la
                                          - torch.log(total(a * q * v ** -et)) + et * lb))
        la, lb = la + c, lb - c
    phi, psi = eps * (la + torch.log(u)), eps * (lb + torch.log(v))
    tp = torch.where(bal, phi, -tf * torch.expm1(-phi / tf))
    tq = torch.where(bal, psi, -tf * torch.expm1(-psi / tf))
    ot = (a * (tp * p + tq * q)).sum(1)
    mass = (a * torch.exp(la + lb) * u * op.heat(v, t)).sum(1)
    return phi, psi, ot, ot - eps * mass, mass


def _divergence64(op, p, q, eps, tau, T):
    """(phi, psi) of the three problems of every pair, their costs, S and S_dual"""
    B = p.shape[0]
    phi, psi, ot, od, _ = _sinkhorn64(op, torch.cat([p, p, q]), torch.cat([q, p, q]), eps, tau.repeat(3, 1), T)
    dm = (op.area * (p - q)).sum(1)
    S = ot[:B] - 0.5 * (ot[B:2 * B] + ot[2 * B:]) + 0.5 * eps * dm * dm
    return phi, psi, ot, S, od[:B] - 0.5 * (od[B:2 * B] + od[2 * B:])


def exact(case, seed):
    x = inputs(case, seed)
    kind = case["kind"]
    flat = lambda f: f.double().reshape(f.shape[0], -1)   # noqa: E731
    if work(case)["flops"] > 5e12:
        return None   # too long in 64 bits
    if kind == "multi":
        S = []
        for n in MULTI_GRIDS:
            op = Operator("gl", n, 2 * n)
            mine = [s for s in x["sets"] if s["nlat"] == n]
            p, q = (torch.cat([flat(s[k]) for s in mine]) for k in ("p", "q"))
            tau = torch.cat([torch.full((case["nf"], 1), s["tau"], device=p.device, dtype=torch.float64) for s in mine])
            _, _, _, s, sd = _divergence64(op, p, q, 4.0 * case["t"], tau, case["T"])
            for i in range(len(mine)):
                S += [v[i * case["nf"]:(i + 1) * case["nf"]].cpu().numpy() for v in (s, sd)]
        return {"S": np.stack(S), "status": None}
    op = Operator(case["grid"], case["nlat"], case["nlon"])
    if kind == "heat":
        return op.heat(flat(x["f"]), case["t"]).reshape(x["f"].shape)
    if kind == "sht":
        c = op.analysis(flat(x["f"]))   # [m, l, 2 nf]
        nf = case["nf"]
        coef = torch.stack([c[..., :nf], c[..., nf:]], -1).permute(2, 1, 0, 3).contiguous()   # [nf, l, m, 2]
        cin = x["c"].double().permute(2, 1, 0, 3)   # [m, l, nf, 2]
        out = op.synthesis(torch.cat([cin[..., 0], cin[..., 1]], 2)).reshape(x["f"].shape)
        return {"coeffs": coef, "fields": out}
    p, q, eps = flat(x["p"]), flat(x["q"]), 4.0 * case["t"]
    tau = torch.full((case["nf"], 1), case["tau"] or math.inf, device=p.device, dtype=torch.float64)
    shape = x["p"].shape[1:]
    if kind == "grad":
        p = p.requires_grad_(True)
        S = _divergence64(op, p, q, eps, tau, case["T"])[3]
        g, = torch.autograd.grad(S.sum(), p)
        return {"grad": g.reshape(x["p"].shape), "S": S.detach().cpu().numpy()[None], "status": None}
    if kind == "sinkhorn":
        phi, psi, ot, od, mass = _sinkhorn64(op, p, q, eps, tau, case["T"])
        sc = [ot, od, mass]
    else:
        phi, psi, ot, S, Sd = _divergence64(op, p, q, eps, tau, case["T"])
        sc = [*ot.reshape(3, -1), S, Sd]
    return {"phi": phi.reshape(-1, *shape), "psi": psi.reshape(-1, *shape),
            "scalars": np.stack([s.cpu().numpy() for s in sc]), "status": None, "iters": None}
