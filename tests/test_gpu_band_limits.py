"""Where a band ends: a Gaussian is integrated over |l - p0| < 6 s and no
further, whatever other rows share a tensor-core tile, also where steep dust
makes the spectrum rise by orders of magnitude past that limit; and bands
anywhere on a grid of more than 65,536 wavelengths; and magnitudes where dust
leaves less than 2^-126 of the flux.

Bars: 3xTF32 and FP32 1e-4 mag and BF16 5e-3 mag against the FP64 oracle (an
exponent of ~60 carries ~1e-5 relative rounding); the same row alone 2e-5 mag
(another order of FP32 sums of such exponentials); gradients 1e-3 (BF16 3e-2) of the row's
largest component."""
import numpy as np
import pytest
import torch

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


def _flat(n_band, n_lam=1501):
    """A table without spectral features, of order one (attenuated by 35 mag and
    more, fluxes stay normal numbers), bands whose tails reach the far UV."""
    rng = np.random.default_rng(3)
    bands = W._gauss_bands(np.geomspace(3000.0, 9000.0, n_band))
    t = W.make_tables(rng, 19, 7, n_lam, 91.0, 12000.0, bands)
    t.ssp = np.repeat(t.ssp.mean(-1, keepdims=True), n_lam, -1) / t.ssp.mean()
    return t


def _cut_gaussians(monkeypatch):
    """The oracle's Gaussians go on past 6 s; the library's end there."""
    full = O.transmission

    def cut(tables, lam_obs):
        T = full(tables, lam_obs)
        for b in np.flatnonzero(np.asarray(tables.band_kind) == W.BAND_GAUSS):
            s = tables.band_p1[b] / (2.0 * np.sqrt(2.0 * np.log(2.0)))
            T[..., b, :] *= ((lam_obs - tables.band_p0[b]).abs() < 6.0 * s).to(T.dtype)
        return T

    monkeypatch.setattr(O, "transmission", cut)


@pytest.mark.parametrize("n_band", [2, 6, 8, 9, 17])
def test_gaussian_support_under_steep_dust(n_band, monkeypatch):
    import paper_2506_19919_gb300 as pkg
    _cut_gaussians(monkeypatch)
    t = _flat(n_band)
    n = 64
    z = np.linspace(0.3, 2.9, n).astype(np.float32).astype(np.float64)
    th = W.prior_draw(np.random.default_rng(4), n)
    th[:, 9], th[:, 10], th[:, 11] = 3.0, -1.0, 0.0              # A_V, delta, F_floor
    ctx = pkg.Context(t)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z, t, "exact").numpy()
    obs = (ref - 1.0).astype(np.float32).astype(np.float64)
    sigma, mask = np.full(obs.shape, 0.05), np.full(n, (1 << n_band) - 1, np.uint32)
    _, gr, _ = O.loglike_and_grad(th, z, t, obs, sigma, mask, "exact", wrt_z=True)
    gr = gr.numpy()
    scale = np.abs(gr).max(1, keepdims=True)
    for prec, mtol, gtol in (("fp32", 1e-4, 1e-3), ("tf32x3", 1e-4, 1e-3), ("bf16", 5e-3, 3e-2)):
        m = ctx.photometry(th, mode="exact", prec=prec).cpu().numpy()
        assert np.abs(m - ref).max() < mtol, prec
        for i in (0, 31, n - 1):
            alone = ctx.photometry(th[i:i + 1], gal_idx=np.array([i], np.int32), mode="exact", prec=prec).cpu().numpy()
            assert np.abs(alone - m[i]).max() < 2e-5, prec
        ll, g = (x.cpu().numpy() for x in ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec=prec))
        lz, gz = (x.cpu().numpy() for x in ctx.loglike_grad_z(th, obs, sigma, mask, mode="exact", prec=prec))
        assert (np.abs(g - gr[:, :12]) / scale).max() < gtol, prec
        assert (np.abs(g - gz[:, :12]) / scale).max() < 1e-3, prec
        np.testing.assert_allclose(ll, lz, rtol=1e-3)
    ctx.close()


@pytest.mark.parametrize("kind", ["gauss", "table", "tophat"])
def test_more_wavelengths_than_16_bits(kind):
    """Bands on both sides of grid index 65,536 and across it."""
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(5)
    centres = np.array([6000.0, 10200.0, 11000.0]) * 1.05
    bands = {"gauss": (np.full(3, W.BAND_GAUSS, np.int32), centres, centres / 60.0),
             "tophat": (np.full(3, W.BAND_TOPHAT, np.int32), centres - 300.0, centres + 300.0)}.get(kind)
    t = W.make_tables(rng, 6, 3, 70001, 900.0, 12000.0, bands or W._gauss_bands([5000.0]))
    if kind == "table":
        k, p0, p1, tn, tT = W.tabulated_bands(rng, [600.0, 1000.0, 1110.0, 1150.0])
        t = W.with_bands(t, k, p0, p1, tn, tT)
    n = 9
    z = rng.uniform(0.03, 0.07, n).astype(np.float32).astype(np.float64)
    th = W.prior_draw(rng, n)
    ctx = pkg.Context(t)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z, t, "exact").numpy()
    obs = (ref - 1.0).astype(np.float32).astype(np.float64)
    sigma, mask = np.full(obs.shape, 0.05), np.full(n, 7, np.uint32)
    _, gr, _ = O.loglike_and_grad(th, z, t, obs, sigma, mask, "exact")
    gr = gr.numpy()
    for prec, mtol, gtol in (("fp32", 2e-5, 1e-4), ("tf32x3", 1e-4, 1e-3), ("bf16", 5e-3, 3e-2)):
        assert np.abs(ctx.photometry(th, mode="exact", prec=prec).cpu().numpy() - ref).max() < mtol, prec
        _, g = ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec=prec)
        assert (np.abs(g.cpu().numpy() - gr).max(1) / np.abs(gr).max(1)).max() < gtol, prec
        if kind != "tophat":
            _, gz = ctx.loglike_grad_z(th, obs, sigma, mask, mode="exact", prec=prec)
            assert (np.abs(gz.cpu().numpy()[:, :12] - gr).max(1) / np.abs(gr).max(1)).max() < gtol, prec
    ctx.close()


@pytest.mark.parametrize("mode,prec", [("approx", "fp32"), ("exact", "fp32"), ("exact", "bf16"), ("exact", "tf32x3")])
def test_deep_attenuation_stays_finite(mode, prec):
    """A band attenuated by 97-108 mag with F_floor = 0: 10^(-0.4 A) is a
    denormal FP32 number of nine bits or more (1e-3 relative), not zero."""
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(3)
    bands = (np.full(2, W.BAND_TOPHAT, np.int32), np.array([1940.0, 5000.0]), np.array([1960.0, 6000.0]))
    t = W.make_tables(rng, 19, 7, 4001, 91.0, 12000.0, bands)
    t.ssp = np.repeat(t.ssp.mean(-1, keepdims=True), 4001, -1) * (1e15 / t.ssp.mean())   # fluxes stay normal numbers
    n = 140
    z = np.full(n, 2.9, np.float32).astype(np.float64)
    th = W.prior_draw(rng, n)
    th[:, 10], th[:, 11] = -0.2, 0.0
    rest = 1950.0 / 3.9 * 1e-4
    k = O.calzetti_k0(torch.tensor(rest)).item() * (rest / 0.55) ** -0.2
    k += O.bump_strength(torch.tensor(-0.2)).item() * O.drude_shape(torch.tensor(rest)).item()
    th[:, 9] = rng.uniform(99.0, 106.0, n) * 4.05 / k
    th = th.astype(np.float32).astype(np.float64)
    ctx = pkg.Context(t)
    ctx.set_galaxies(z, build_approx=True)
    ref = O.photometry(th, z, t, mode).numpy()
    m = ctx.photometry(th, mode=mode, prec=prec).cpu().numpy()
    assert np.abs(m - ref).max() < 5e-3
    if mode == "exact":            # all but F_floor, whose column is 10^40 and more
        obs = (ref - 1.0).astype(np.float32).astype(np.float64)
        sigma, mask = np.full(obs.shape, 0.05), np.full(n, 3, np.uint32)
        _, gr, _ = O.loglike_and_grad(th, z, t, obs, sigma, mask, mode)
        gr = gr.numpy()[:, :11]
        _, g = ctx.loglike_grad(th, obs, sigma, mask, mode=mode, prec=prec)
        assert (np.abs(g.cpu().numpy()[:, :11] - gr).max(1) / np.abs(gr).max(1)).max() < 3e-2
    ctx.close()
