"""The calls whose speed matters to a user of this library, as cases that can be
timed and checked: photometry of a catalogue, log L with its gradient for an
outside sampler, a new galaxy set, and the batched sampler itself.

Each case names an operation, an SSP grid, a filter set and sizes.  The grids
and filter sets are those of the repository's workloads: a 50 x 6 x 2000 grid
with six top-hats, and the 107 x 12 x 5994 production grid with 6, 12 or 20
Gaussian bands (or six tabulated throughput curves).  Parameters are uniform
in the inner 98% of their prior ranges, redshifts uniform, every galaxy with
its own data and band mask.

The second half of the file is the model in plain torch: in 64 bits it gives
the values that `exact` returns, in 32 bits the magnitudes that stand for the
observed ones.  Every tensor is made from the seed alone.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2506_19919_gb300 as sps

# Prior ranges of the 12 parameters (lgM, tau, alpha, beta, F_burst, lgT_peak,
# dlgT, lgZ, sigma_lgZ, A_V, delta, F_floor).
LO = np.array([-1.5, 0.5, 0.1, 0.1, 0.0, 6.0, 0.05, -2.0, 0.05, 0.0, -1.0, 0.0])
HI = np.array([2.5, 12.0, 5.0, 5.0, 0.2, 8.5, 1.5, 0.2, 0.5, 3.0, 0.4, 0.5])
TOPHAT, GAUSS, TABLE = 0, 1, 2


def _case(name, op, bands, gal, chains=1, mode="exact", prec="fp32", masked=False, mdf=False, samples=0):
    return {"name": name, "op": op, "bands": bands, "gal": gal, "chains": chains, "mode": mode, "prec": prec,
            "masked": masked, "mdf": mdf, "samples": samples}


def listed():
    return [
        # a few galaxies checked interactively against exact photometry at the default precision
        _case("phot_exact_fp32_few", "photometry", "tophat6", 64),
        # one step of an outside sampler with a handful of galaxies: launches and latency count
        _case("like_approx_few", "loglike_grad", "gauss12", 16, 4, "approx", masked=True),
        # a handful of galaxies on the exact path, the gradient for an optimiser
        _case("like_exact_bf16_few", "loglike_grad", "gauss6", 100, 1, "exact", "bf16"),
        # reference-precision photometry (the default arguments) of a mid-sized sample
        _case("phot_exact_fp32", "photometry", "gauss6", 20011),
        # reference-precision log L and gradient, e.g. to judge the faster modes
        _case("like_exact_fp32", "loglike_grad", "gauss6", 8192),
        # production photometry of a catalogue on the tensor cores, and with the approximation
        _case("phot_exact_bf16", "photometry", "gauss6", 100000, 1, "exact", "bf16"),
        _case("phot_approx", "photometry", "gauss6", 100000, 1, "approx"),
        # 100,000 (galaxy, chain) pairs: log L and the adjoint, both paths
        _case("like_exact_bf16", "loglike_grad", "gauss6", 100000, 1, "exact", "bf16"),
        _case("like_approx", "loglike_grad", "gauss6", 100000, 1, "approx"),
        # every chain's gradient at FP32-grade accuracy on the tensor cores, uneven band masks
        _case("like_exact_tf32x3", "loglike_grad", "gauss12", 4096, 4, "exact", "tf32x3", masked=True),
        # a new catalogue: per-galaxy tables at the galaxies' redshifts, then their magnitudes
        _case("catalogue", "catalogue", "gauss12", 4001, 1, "approx"),
        # the batched sampler, 3-12 observed bands per galaxy
        _case("hmc", "hmc", "gauss12", 4096, 4, "approx", masked=True, samples=2),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    count = {"gauss6": 6, "gauss12": 12, "gauss20": 20, "table6": 6, "tophat6": 6}
    op = rng.choice(["photometry", "photometry", "loglike_grad", "loglike_grad", "loglike_grad", "loglike_grad_z",
                     "catalogue", "hmc"])
    if op == "catalogue":
        bands = rng.choice(["gauss6", "gauss12", "gauss20", "table6"])
        return _drawn(op, bands, size(20, 48000 // count[bands]), 1, "approx")
    if op == "hmc":
        return _drawn(op, rng.choice(["gauss6", "gauss12"]), size(30, 4096), rng.choice([1, 2, 3, 4]), "approx",
                      masked=True, samples=2)
    mode = rng.choice(["exact", "exact", "approx"])
    prec = "fp32" if mode == "approx" else rng.choice(["fp32", "bf16", "bf16", "tf32x3"])
    bands = rng.choice(["gauss6", "gauss12", "gauss20", "table6"] + (["tophat6"] if op != "loglike_grad_z" else []))
    nb = count[bands]
    grad = op != "photometry"
    rows = {"approx": 600000 // nb, "fp32": 8192 if grad else 20011, "tf32x3": 16384 * 6 // nb,
            "bf16": 600000 // nb // (2 if nb == 20 else 1)}[mode if mode == "approx" else prec]
    if op == "loglike_grad_z":
        rows //= 4
    chains = 1 if op == "photometry" else rng.choice([1, 2, 4])
    mdf = rng.random() < 0.15
    return _drawn(op, bands, max(1, size(1, rows) // chains), chains, mode, prec,
                  masked=grad and rng.random() < 0.7, mdf=mdf)


def _drawn(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _tables(bands, mdf):
    """Grids, a synthetic SSP table (positive, smooth; a floor and 8 Gaussians in
    ln lambda that fade with age) and the filter set."""
    rng = np.random.default_rng(1906)
    A, Z, N, lo, hi = (50, 6, 2000, 1000.0, 12000.0) if bands == "tophat6" else (107, 12, 5994, 91.0, 25000.0)
    age = np.logspace(6.0, math.log10(1.4e10), A)
    lgz = np.linspace(-2.0, 0.2, Z)
    lam = np.geomspace(lo, hi, N)
    ln = np.log(lam)
    mu, s = rng.uniform(ln[0], ln[-1], 8), rng.uniform(0.05, 0.5, 8)
    amp = rng.uniform(0.2, 1.0, (8, Z)) * (1.0 + 0.1 * np.arange(Z))
    gyr = age / 1e9
    fade = np.where(mu < math.log(4000.0), gyr[:, None] ** -0.5, 1.0)
    shape = np.exp(-0.5 * ((ln - mu[:, None]) / s[:, None]) ** 2)
    coef = (fade[:, None, :] * amp.T[None, :, :]).reshape(A * Z, 8)
    ssp = (1e-15 * gyr ** -0.7)[:, None, None] * (0.02 + (coef @ shape).reshape(A, Z, N))
    tab_n = tab_T = None
    if bands == "tophat6":
        e = np.array([3200.0, 4000.0, 5500.0, 7000.0, 8200.0, 9200.0, 10600.0])
        kind, p0, p1 = np.full(6, TOPHAT), e[:-1], e[1:]
    elif bands == "table6":
        e = np.array([3200.0, 4000.0, 5500.0, 7000.0, 8200.0, 9200.0, 10600.0])
        p0, ns, Ts = [], [], []
        for a, b in zip(e[:-1], e[1:]):
            w = 0.01 * (a + b)
            x0 = 10.0 * math.floor((a - 8 * w) / 10.0)
            x = x0 + 10.0 * np.arange(int(math.ceil((b + 8 * w - x0) / 10.0)) + 1)
            T = 0.7 / (1 + np.exp(-(x - a) / w)) / (1 + np.exp((x - b) / w)) * (1 + 0.03 * np.sin(x / 60.0))
            T[0] = T[-1] = 0.0
            p0.append(x0)
            ns.append(len(x))
            Ts.append(T)
        kind, p0, p1 = np.full(6, TABLE), np.array(p0), np.full(6, 10.0)
        tab_n, tab_T = np.array(ns, np.int32), np.concatenate(Ts)
    else:
        p0 = {"gauss6": np.linspace(3600.0, 9700.0, 6), "gauss12": np.geomspace(3000.0, 24000.0, 12),
              "gauss20": np.geomspace(3000.0, 24000.0, 20)}[bands]
        kind, p1 = np.full(len(p0), GAUSS), p0 / np.geomspace(3.4, 25.5, len(p0))
    off = -0.25 * np.log10(1.0 + gyr) if mdf else None
    return SimpleNamespace(age_yr=age, lgZ=lgz, lam_ang=lam, ssp=ssp, band_kind=kind.astype(np.int32),
                           band_p0=p0.astype(np.float64), band_p1=p1.astype(np.float64), band_tab_n=tab_n,
                           band_tab_T=tab_T, mdf_offset=off, n_band=len(kind), K=A * Z)


def _theta(rng, n):
    u = rng.uniform(size=(n, 12))
    return (LO + 0.01 * (HI - LO) + 0.98 * u * (HI - LO)).astype(np.float32)


def _inputs(case, seed):
    """Host arrays and device tensors of a case, all float32 (masks int32)."""
    T = _tables(case["bands"], case["mdf"])
    rng = np.random.default_rng(seed)
    G, C, B = case["gal"], case["chains"], T.n_band
    z = rng.uniform(0.05, 1.0 if case["bands"] == "tophat6" else 3.0, G).astype(np.float32)
    truth = _theta(rng, G)
    d = SimpleNamespace(T=T, z=z, obs=None, sigma=None, mask=None, idx=None)
    d.theta = torch.as_tensor(truth if case["op"] in ("photometry", "catalogue") else _theta(rng, G * C)).cuda()
    if case["op"] in ("photometry", "catalogue"):
        return d
    lo = B // 4 if case["masked"] else B
    k = rng.integers(lo, B + 1, G)
    rank = np.argsort(np.argsort(rng.uniform(size=(G, B)), axis=1), axis=1)
    bits = ((rank < k[:, None]).astype(np.uint32) << np.arange(B, dtype=np.uint32)).sum(1, dtype=np.uint32)
    d.mask = torch.as_tensor(bits.view(np.int32)).cuda()
    err = 0.2 if case["op"] == "hmc" else 0.05
    d.sigma = torch.full((G, B), err, dtype=torch.float32, device="cuda")
    noise = torch.as_tensor(rng.normal(0.0, err, (G, B)).astype(np.float32)).cuda()
    with torch.no_grad():
        m = [_mags(T, t, zz, case["mode"]) for t, zz in _chunks(torch.as_tensor(truth).cuda(), torch.as_tensor(z).cuda())]
    d.obs = torch.cat(m) + noise
    if C > 1:
        d.idx = torch.arange(G, dtype=torch.int32, device="cuda").repeat_interleave(C)
    if case["op"] == "hmc":                     # chains start in the posterior, in unbounded space
        s = (truth.astype(np.float64) - LO) / (HI - LO)
        d.theta = torch.as_tensor(np.log(s / (1 - s)).astype(np.float32)).cuda().repeat_interleave(C, 0)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    ctx = sps.Context(d.T)
    if case["op"] != "catalogue":
        ctx.set_galaxies(d.z, build_approx=case["mode"] == "approx")
    return SimpleNamespace(case=case, ctx=ctx, d=d, seed=seed)


# ---------------------------------------------------------------- one pass
def run(state):
    c, ctx, d = state.case, state.ctx, state.d
    if c["op"] == "photometry":
        return {"mag": ctx.photometry(d.theta, mode=c["mode"], prec=c["prec"])}
    if c["op"] == "catalogue":
        ctx.set_galaxies(d.z, build_approx=True)
        return {"mag": ctx.photometry(d.theta, mode="approx")}
    if c["op"] == "hmc":
        # sampling goes on from a known step size
        out = ctx.hmc_run(d.theta, d.obs, d.sigma, d.mask, chains_per_gal=c["chains"], n_warm=0, n_samp=c["samples"],
                          L_min=8, L_max=64, eps0=2e-3, seed=state.seed)
        return {k: out[k] for k in ("samples", "accept_prob", "step_size", "divergences", "grad_evals")}
    call = ctx.loglike_grad if c["op"] == "loglike_grad" else ctx.loglike_grad_z
    ll, grad = call(d.theta, d.obs, d.sigma, d.mask, gal_idx=d.idx, mode=c["mode"], prec=c["prec"])
    return {"ll": ll, "grad": grad}


# ---------------------------------------------------------------- work of one pass
def _support(T):
    """Grid points inside each band and inside their union, averaged over redshift."""
    per, union = np.zeros(T.n_band), 0.0
    zs = np.linspace(0.1, 1.0 if T.band_kind[0] == TOPHAT else 2.95, 16)
    for z in zs:
        lo, hi = T.band_p0, T.band_p1
        if T.band_kind[0] == GAUSS:
            half = 6 * T.band_p1 / (2 * math.sqrt(2 * math.log(2)))
            lo, hi = T.band_p0 - half, T.band_p0 + half
        elif T.band_kind[0] == TABLE:
            lo, hi = T.band_p0, T.band_p0 + T.band_p1 * (T.band_tab_n - 1)
        x = (1 + z) * T.lam_ang
        inside = (x >= lo[:, None]) & (x < hi[:, None])
        per += inside.sum(1) / len(zs)
        union += inside.any(0).sum() / len(zs)
    return per, union


def work(case):
    T = _tables(case["bands"], case["mdf"])
    G, B, K = case["gal"], T.n_band, T.K
    rows = G * case["chains"]
    per, union = _support(T)
    nb = (B // 4 + B) / 2 if case["masked"] else B              # observed bands
    table = 4 * K * union * (0.5 if case["prec"] == "bf16" else 1)
    cssp = 4.0 * G * K * B
    if case["op"] == "catalogue":
        return {"bytes": 4 * K * len(T.lam_ang) + cssp + 4 * G * (13 + B), "flops": 2 * K * per.sum() * G + 2.0 * K * B * G}
    if case["op"] == "hmc":
        evals = rows * (1 + case["samples"] * 36.0)
        return {"bytes": cssp * nb / B + 4 * rows * 12 * (1 + case["samples"]) + 8 * G * B, "flops": 4.0 * nb * K * evals}
    grad = case["op"] != "photometry"
    io = 4 * rows * (12 + (14 if grad else B)) + (8 * G * B if grad else 0)
    if case["mode"] == "approx":
        z = 2 if case["op"] == "loglike_grad_z" else 1          # d c_SSP / dz too
        return {"bytes": io + cssp * nb / B * z, "flops": (4.0 if grad else 2.0) * nb * K * rows}
    return {"bytes": io + table, "flops": (4.0 if grad else 2.0) * K * union * rows}


# ---------------------------------------------------------------- the model in plain torch
def _chunks(*tensors, rows=2048):
    for i in range(0, tensors[0].shape[0], rows):
        yield tuple(None if t is None else t[i:i + rows] for t in tensors)


@functools.lru_cache(maxsize=None)
def _double_exponential(h=1.0 / 16.0, umax=3.2):
    """Nodes (distance to the nearer end, and which end) and weights of the tanh-sinh rule on [0, 1]."""
    u = h * np.arange(0, int(round(umax / h)) + 1)
    a = 0.5 * math.pi * np.sinh(u)
    d = 1.0 / (1.0 + np.exp(2.0 * a))
    w = h * 0.25 * math.pi * np.cosh(u) / np.cosh(a) ** 2
    return (np.concatenate([d, d[1:]]), np.concatenate([w, w[1:]]),
            np.concatenate([np.ones(len(u), bool), np.zeros(len(u) - 1, bool)]))


def _dust_curve(lam):
    """Calzetti et al. (2000) k'(lambda) with R_V = 4.05 and the unit Drude bump at 0.2175 um."""
    x = lam * 1e-4
    k = torch.where(x < 0.63, 2.659 * (-2.156 + 1.509 / x - 0.198 / x ** 2 + 0.011 / x ** 3),
                    2.659 * (-1.857 + 1.040 / x)) + 4.05
    b = (x * 0.035) ** 2
    return k.clamp(min=0.0), b / ((x ** 2 - 0.2175 ** 2) ** 2 + b)


def _attenuation(lam, th):
    k, bump = _dust_curve(lam)
    AV, dl, ff = (th[:, i:i + 1] for i in (9, 10, 11))
    A = AV / 4.05 * (k * torch.exp(dl * torch.log(lam / 5500.0)) + (0.85 - 1.9 * dl).clamp(min=0.0) * bump)
    return ff + (1 - ff) * torch.exp(-0.4 * math.log(10.0) * A)


def _weights(T, th, t_obs):
    """SSP weights [N, A, Zn] of the double power law, the triweight burst and the metallicity Gaussian."""
    new = functools.partial(torch.as_tensor, dtype=th.dtype, device=th.device)
    tau, al, be = (th[:, i, None, None] for i in (1, 2, 3))
    mid = np.sqrt(T.age_yr[1:] * T.age_yr[:-1])
    edge = new(np.concatenate([[0.0], mid / 1e9, [1e30]]))
    To = t_obs[:, None]
    e = torch.minimum(edge, To)
    width = e[:, 1:] - e[:, :-1]
    live = width > 0
    width = torch.where(live, width, torch.ones_like(width))
    hi = To - e[:, :-1]
    lo = torch.where(live, To - e[:, 1:], torch.zeros_like(hi))
    hi = torch.where(live, hi, torch.ones_like(hi))
    dist, wq, left = _double_exponential()
    dist, wq, left = new(dist), new(wq), torch.as_tensor(left, device=th.device)
    t = torch.where(left, lo[..., None] + width[..., None] * dist, hi[..., None] - width[..., None] * dist)
    lu = torch.log(t) - torch.log(tau)
    f = torch.exp(be * lu - torch.nn.functional.softplus((al + be) * lu, threshold=1e9))
    m = torch.where(live, width * (f * wq).sum(-1), torch.zeros_like(width))
    M = m.sum(1, keepdim=True)
    le = torch.minimum(new(np.concatenate([[-100.0], np.log10(mid), [100.0]])), torch.log10(To * 1e9))
    u = ((le - th[:, 5:6]) / th[:, 6:7]).clamp(-1.0, 1.0)
    cdf = 0.5 + 35.0 / 32.0 * (u - u ** 3 + 0.6 * u ** 5 - u ** 7 / 7.0)
    burst = (cdf[:, 1:] - cdf[:, :-1]) / cdf[:, -1:]
    w = (1 - th[:, 4:5]) * m + th[:, 4:5] * burst * M
    mean = th[:, 7:8, None] + (new(T.mdf_offset)[None, :, None] if T.mdf_offset is not None else 0.0)
    y = (new(0.5 * (T.lgZ[1:] + T.lgZ[:-1])) - mean) / th[:, 8:9, None]
    below, above = torch.special.ndtr(y), torch.special.ndtr(-y)
    inner = torch.where(y[..., 1:] > 0, above[..., :-1] - above[..., 1:], below[..., 1:] - below[..., :-1])
    q = torch.cat([below[..., :1], inner, above[..., -1:]], -1)
    return 10.0 ** (th[:, 0, None, None]) * 1e9 * w[:, :, None] * q


def _mags(T, th, z, mode):
    """AB magnitudes [N, B] in the type of `th`, differentiable in th and z."""
    new = functools.partial(torch.as_tensor, dtype=th.dtype, device=th.device)
    opz = 1 + z[:, None]
    Om, OL, H0 = 0.3, 0.7, 70.0
    hubble = 3.0856775814913673e19 / H0 / 3.15576e16
    t_obs = 2 / (3 * math.sqrt(OL)) * hubble * torch.asinh(math.sqrt(OL / Om) * opz[:, 0] ** -1.5)
    x, wx = np.polynomial.legendre.leggauss(48)
    x, wx = new(0.5 * (x + 1)), new(0.5 * wx)
    dc = (wx / torch.sqrt(Om * (1 + z[:, None] * x) ** 3 + OL)).sum(1) * z * 299792.458 / H0
    lam = new(T.lam_ang)
    step = np.diff(T.lam_ang)                           # trapezoid rule
    q = new(0.5 * (np.append(step, 0.0) + np.append(0.0, step)))
    scale = 1e15                                        # keeps the 32-bit sums in range
    S = _weights(T, th, t_obs).flatten(1) @ new(T.ssp.reshape(T.K, -1) * scale)
    if mode == "exact":
        F = _attenuation(lam[None, :], th)
    xo = opz * lam
    mags, off = [], 0
    for b in range(T.n_band):
        p0, p1 = float(T.band_p0[b]), float(T.band_p1[b])
        if T.band_kind[b] == TOPHAT:
            t = ((xo >= p0) & (xo < p1)).to(th.dtype)
        elif T.band_kind[b] == GAUSS:
            u = (xo - p0) * (2 * math.sqrt(2 * math.log(2)) / p1)
            t = torch.where(u.abs() < 6.0, torch.exp(-0.5 * u * u), torch.zeros_like(u))
        else:
            n = int(T.band_tab_n[b])
            tab = new(T.band_tab_T[off:off + n])
            off += n
            u = (xo - p0) / p1
            m = u.detach().floor().clamp(0, n - 2).long()
            t = torch.where((u >= 0) & (u <= n - 1), tab[m] + (u - m) * (tab[m + 1] - tab[m]), torch.zeros_like(u))
        tq = t * q
        wb = tq / lam
        if mode == "exact":
            c = (wb * F * S).sum(1)
        else:
            eff = (tq * lam).sum(1) / tq.sum(1)
            c = _attenuation(eff[:, None], th)[:, 0] * (wb * S).sum(1)
        # m = -2.5 log10((1 + z) L_sun c / (4 pi d_L^2 3631 Jy N_b)), logarithms taken apart
        lum = math.log10(3.828e33 / (4 * math.pi * 3631e-23)) - 2 * math.log10(3.0856775814913673e24) - math.log10(scale)
        mags.append(-2.5 * (torch.log10(c) - torch.log10(wb.sum(1)) - torch.log10(opz[:, 0]) - 2 * torch.log10(dc) + lum))
    return torch.stack(mags, 1)


def exact(case, seed):
    if case["op"] == "hmc":                # a trajectory in 64 bits takes minutes
        return None
    d = _inputs(case, seed)
    z = torch.as_tensor(d.z).cuda().double()
    if case["op"] in ("photometry", "catalogue"):
        with torch.no_grad():
            return {"mag": torch.cat([_mags(d.T, t.double(), zz, case["mode"]) for t, zz in _chunks(d.theta, z)])}
    idx = torch.arange(len(d.theta), device="cuda") if d.idx is None else d.idx.long()
    lls, grads = [], []
    for th, i in _chunks(d.theta, idx):
        th = th.double().requires_grad_()
        zz = z[i].requires_grad_()
        seen = (d.mask[i].long()[:, None] >> torch.arange(d.T.n_band, device="cuda")) & 1
        r = (_mags(d.T, th, zz, case["mode"]) - d.obs[i].double()) / d.sigma[i].double()
        ll = -0.5 * (seen * r * r).sum(1)
        g, gz = torch.autograd.grad(ll.sum(), (th, zz))
        lls.append(ll.detach())
        grads.append(torch.cat([g, gz[:, None]], 1) if case["op"] == "loglike_grad_z" else g)
    return {"ll": torch.cat(lls), "grad": torch.cat(grads)}
