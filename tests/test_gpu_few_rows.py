"""Approximate photometry and log L + gradient of few rows (one block per row)
against the general one-row-per-warp path and the FP64 oracle: one row, odd
counts, the largest count that takes this route and the first that does not;
the fewest and the most age bins (2 and 128), odd metallicity counts up to the
12 it accepts, one band and 32, masks with no, one and all bands; a row that is
not finite.

Bars: magnitudes 1e-5 mag, gradients 1e-4 of the row's largest component
(residuals of 1 mag, all of one sign: no cancellation between bands)."""
import os

import numpy as np
import pytest
import torch

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


def _general(f):
    os.environ["SPS_LIKE_ROWS"] = "1"
    try:
        return f()
    finally:
        os.environ.pop("SPS_LIKE_ROWS", None)


@pytest.mark.parametrize("n_age,n_met,n_band", [(2, 2, 1), (31, 5, 3), (107, 12, 6), (128, 10, 32)])
@pytest.mark.parametrize("n", [1, 7, 760, 761])
def test_few_rows_match_general_path_and_oracle(n_age, n_met, n_band, n):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(n + n_age)
    bands = W._gauss_bands(np.geomspace(3000.0, 9000.0, n_band) if n_band > 1 else [5000.0])
    tabs = W.make_tables(rng, n_age, n_met, 500, 900.0, 12000.0, bands)
    G = 23
    z = rng.uniform(0.05, 1.0, G).astype(np.float32).astype(np.float64)
    idx = rng.integers(0, G, n).astype(np.int32)
    th = W.prior_draw(rng, n)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=True)
    ref = O.photometry(th, z[idx], tabs, "approx").numpy()
    m = ctx.photometry(th, gal_idx=idx, mode="approx").cpu().numpy()
    assert np.abs(m - ref).max() < 1e-5
    mg = _general(lambda: ctx.photometry(th, gal_idx=idx, mode="approx").cpu().numpy())
    assert np.abs(m - mg).max() < 1e-5
    # data per galaxy 1 mag brighter than the first row that refers to it; other rows differ more
    sigma = np.full((G, n_band), 0.05)
    obs = np.full((G, n_band), ref.min() - 1.0)          # brighter than every row in every band
    mask = rng.integers(0, 1 << n_band, G, dtype=np.uint64).astype(np.uint32)
    mask[0], mask[1], mask[2] = 0, 1, (1 << n_band) - 1
    call = lambda: ctx.loglike_grad(th, obs, sigma, mask, gal_idx=idx, mode="approx")   # noqa: E731
    ll, g = (x.cpu().numpy().astype(np.float64) for x in call())
    llg, gg = (x.cpu().numpy().astype(np.float64) for x in _general(call))
    scale = np.maximum(np.abs(gg).max(1, keepdims=True), 1e-30)
    assert (np.abs(g - gg) / scale).max() < 1e-4
    np.testing.assert_allclose(ll, llg, rtol=1e-5)
    assert (ll[mask[idx] == 0] == 0).all() and (g[mask[idx] == 0] == 0).all()
    k = min(n, 60)
    obs32 = obs.astype(np.float32).astype(np.float64)
    llr, gr, _ = O.loglike_and_grad(th[:k], z[idx[:k]], tabs, obs32[idx[:k]], sigma[idx[:k]], mask[idx[:k]], "approx")
    scale = np.maximum(np.abs(gr.numpy()).max(1, keepdims=True), 1e-30)
    assert (np.abs(g[:k] - gr.numpy()) / scale).max() < 1e-4
    np.testing.assert_allclose(ll[:k], llr.numpy(), rtol=1e-5)
    # a row that is not finite is NaN and flagged; the others stand
    bad = torch.as_tensor(th, dtype=torch.float32, device="cuda")
    bad[0, 3] = float("nan")
    out = torch.zeros((n, n_band), device="cuda")
    with pytest.raises(pkg.SpsError):
        ctx.photometry(bad, gal_idx=idx, mode="approx", out=out)
    out = out.cpu().numpy()
    assert np.isnan(out[0]).all() and (n == 1 or np.array_equal(out[1:], m[1:]))
    ctx.close()


@pytest.mark.parametrize("n_age,n_met", [(33, 10), (70, 12), (107, 12)])
def test_few_rows_after_other_kernels(n_age, n_met):
    """The block-per-row kernel reads no quadrature bookkeeping that another
    kernel left in shared memory: log L + gradient of the same rows before and
    after calls that integrate other rows with other layouts."""
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(n_age)
    tabs = W.make_tables(rng, n_age, n_met, 401, 900.0, 12000.0, W._gauss_bands([3600.0, 5200.0, 7600.0]))
    G, n = 9, 760
    z = rng.uniform(0.05, 1.0, G).astype(np.float32).astype(np.float64)
    idx = rng.integers(0, G, n).astype(np.int32)
    th = W.prior_draw(rng, n)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=True)
    obs, sigma, mask = np.full((G, 3), 15.0), np.full((G, 3), 0.05), np.full(G, 7, np.uint32)
    call = lambda: [x.cpu().numpy() for x in ctx.loglike_grad(th, obs, sigma, mask, gal_idx=idx)]   # noqa: E731
    ll, g = _general(call)
    other = W.prior_draw(rng, 2000)
    oi = rng.integers(0, G, 2000).astype(np.int32)
    for mode in ("exact", "approx"):
        for _ in range(3):
            ctx.photometry(other, gal_idx=oi, mode=mode)
            ctx.loglike_grad(other, obs, sigma, mask, gal_idx=oi, mode=mode)
            l1, g1 = call()
            assert (np.abs(g1 - g).max(1) / np.abs(g).max(1)).max() < 1e-4
            np.testing.assert_allclose(l1, ll, rtol=1e-5)
    ctx.close()
