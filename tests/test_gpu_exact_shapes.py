"""The exact path where its kernels change with the filter set or the table:
the band counts at which the tensor-core forward changes its tile and its
epilogue warps, the metallicity counts on both sides of the separable weight
gradient, and the row counts on both sides of the one-launch redshift order;
and a sampler run of few chains, whose launch shape differs from a long run's.

Bars: BF16 5e-3 mag and 3xTF32 1e-4 mag against FP32; FP32 magnitudes 2e-5 mag
and gradients 1e-4 of the row's largest component against the FP64 oracle
(residuals of 1 mag of one sign: no cancellation between bands); a row in
another batch 1e-5 mag; the same chains in another launch shape bit for bit."""
import os

import numpy as np
import pytest

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


def _context(n_age, n_met, n_band, n, seed=6):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(seed)
    bands = W._gauss_bands(np.geomspace(2500.0, 10000.0, n_band) if n_band > 1 else [5000.0])
    tabs = W.make_tables(rng, n_age, n_met, 601, 900.0, 12000.0, bands)
    z = rng.uniform(0.05, 1.0, n).astype(np.float32).astype(np.float64)
    return pkg.Context(tabs), tabs, z, W.prior_draw(rng, n)


@pytest.mark.parametrize("n_band", [1, 6, 7, 8, 9, 16, 17, 24, 25, 32])
def test_forward_shapes_match_fp32(n_band):
    n = 133
    ctx, tabs, z, th = _context(9, 5, n_band, n)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z, tabs, "exact").numpy()
    obs = np.repeat(ref.min(1, keepdims=True) - 1.0, n_band, 1)
    sigma, mask = np.full(obs.shape, 0.05), np.full(n, (1 << n_band) - 1, np.uint32)
    mask[::4] &= np.uint32(0x55555555)
    for prec, mtol in (("fp32", 2e-5), ("bf16", 5e-3), ("tf32x3", 1e-4)):
        assert np.abs(ctx.photometry(th, mode="exact", prec=prec).cpu().numpy() - ref).max() < mtol
    _, gr, _ = O.loglike_and_grad(th, z, tabs, obs.astype(np.float32).astype(np.float64), sigma, mask, "exact")
    gr = gr.numpy()
    for prec, gtol in (("fp32", 1e-4), ("tf32x3", 1e-3), ("bf16", 3e-2)):
        _, g = ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec=prec)
        g = g.cpu().numpy()
        assert (np.abs(g - gr).max(1) / np.maximum(np.abs(gr).max(1), 1e-30)).max() < gtol, prec
    ctx.close()


@pytest.mark.parametrize("n_age,n_met", [(2, 2), (31, 11), (33, 12), (109, 12), (100, 13), (128, 10), (40, 16)])
def test_weight_gradient_shapes_match_oracle(n_age, n_met):
    n = 37
    ctx, tabs, z, th = _context(n_age, n_met, 3, n)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z, tabs, "exact").numpy()
    obs = (np.repeat(ref.min(1, keepdims=True) - 1.0, 3, 1)).astype(np.float32).astype(np.float64)
    sigma, mask = np.full(obs.shape, 0.05), np.full(n, 7, np.uint32)
    _, gr, _ = O.loglike_and_grad(th, z, tabs, obs, sigma, mask, "exact")
    _, g = ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec="fp32")
    assert (np.abs(g.cpu().numpy() - gr.numpy()).max(1) / np.abs(gr.numpy()).max(1)).max() < 1e-4
    ctx.close()


@pytest.mark.parametrize("n", [1023, 1024, 1025])
def test_row_order_around_the_one_launch_limit(n):
    ctx, _, z, th = _context(9, 5, 3, 50)
    ctx.set_galaxies(z, build_approx=False)
    idx = np.random.default_rng(n).permutation(np.arange(n) % 50).astype(np.int32)   # many equal redshifts
    for prec in ("fp32", "bf16"):
        alone = ctx.photometry(th, mode="exact", prec=prec).cpu().numpy()
        m = ctx.photometry(th[idx], gal_idx=idx, mode="exact", prec=prec).cpu().numpy()
        assert np.abs(m - alone[idx]).max() < 1e-5
    ctx.close()


@pytest.mark.parametrize("n,chains", [(1, 1), (7, 2), (300, 4)])
def test_sampler_of_few_chains_in_every_shape(n, chains):
    ctx, tabs, z, th = _context(31, 5, 4, n)
    ctx.set_galaxies(z, build_approx=True)
    obs = O.photometry(th, z, tabs, "approx").numpy() + 0.02
    sigma, mask = np.full(obs.shape, 0.05), np.full(n, 15, np.uint32)
    x0 = np.random.default_rng(n).normal(0.0, 0.3, (n * chains, 12)).astype(np.float32)

    def run(shape):
        if shape:
            os.environ["SPS_HMC_SHAPE"] = shape
        try:
            o = ctx.hmc_run(x0, obs, sigma, mask, chains_per_gal=chains, n_warm=2, n_samp=3, seed=5)
            return o["samples"].cpu().numpy()
        finally:
            os.environ.pop("SPS_HMC_SHAPE", None)

    ref = run(None)
    assert np.isfinite(ref).all()
    for shape in ("1,1", "1,8", "2,4") if chains > 1 else ("1,1", "1,8"):
        assert np.array_equal(run(shape), ref), shape
    ctx.close()
