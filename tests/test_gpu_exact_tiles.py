"""The exact path at the sizes where its tiling changes: rows around the 64-
and 128-row tiles and the switch between them, several row tiles in scrambled
redshift order, wavelength and reduction splits, an odd number of (age, Z)
columns, a ragged wavelength grid, and filter sets that cover a part of it,
or nearly all of it; FP32 against the FP64 oracle, the other
precisions against the FP32 path (magnitudes) and every precision against
itself on the same rows in other batches.

Bars: FP32 magnitudes 2e-5 mag (fast exponentials of arguments up to ~10 add
~5e-6 relative to the FP32 sums' 1e-6), its gradient 1e-4 of the row's largest
component; BF16 5e-3 mag and 3xTF32 1e-4 mag.  A row in another batch changes
by the order of FP32 sums: 1e-5 mag, and 1e-3 of its largest gradient component
(through the residual, and through BF16 roundings of v that flip)."""
import numpy as np
import pytest
import torch

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


def _bands(which):
    if which == "part":
        return W._gauss_bands([3600.0, 5500.0])
    if which == "all":
        return W._gauss_bands(np.geomspace(2000.0, 11000.0, 9))
    return W._tophat_bands([320, 400, 550])


def _case(which, n, seed=4):
    rng = np.random.default_rng(seed)
    tabs = W.make_tables(rng, 19, 7, 901, 900.0, 12000.0, _bands(which))      # 133 columns
    z = rng.uniform(0.05, 1.2, n).astype(np.float32).astype(np.float64)
    return tabs, z, W.prior_draw(rng, n)


def _rel(g, ref):
    g, ref = np.asarray(g, np.float64), np.asarray(ref, np.float64)
    return (np.abs(g - ref).max(1) / np.abs(ref).max(1)).max()


@pytest.mark.parametrize("which", ["part", "all", "tophat"])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 128, 129, 300])
def test_exact_tiles_match_oracle(which, n):
    import paper_2506_19919_gb300 as pkg
    tabs, z, th = _case(which, n)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=False)
    B = tabs.n_band
    # residuals of 1 mag, all of one sign: near the data, or where bands pull
    # against each other, the gradient is a difference of rounding errors
    mr = O.photometry(th, z, tabs, "exact").numpy()
    obs = (mr - 1.0).astype(np.float32).astype(np.float64)
    sigma = np.full((n, B), 0.05)
    mask = np.full(n, (1 << B) - 1, np.uint32)
    mask[1::3] &= ~np.uint32(1)
    llr, gr, _ = O.loglike_and_grad(th, z, tabs, obs, sigma, mask, "exact")
    m32 = ctx.photometry(th, mode="exact").cpu().numpy()
    assert np.abs(m32 - mr).max() < 2e-5
    ll, g = ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec="fp32")
    assert _rel(g.cpu().numpy(), gr.numpy()) < 1e-4
    np.testing.assert_allclose(ll.cpu().numpy(), llr.numpy(), rtol=1e-4)
    # the other precisions: magnitudes against FP32, and every row in its tile,
    # order and split against the row in calls of its own few
    for prec, mtol in (("fp32", 1e-7), ("bf16", 5e-3), ("tf32x3", 1e-4)):
        m = ctx.photometry(th, mode="exact", prec=prec).cpu().numpy()
        assert np.abs(m - m32).max() < mtol
        _, g = ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec=prec)
        g = g.cpu().numpy()
        for i in (np.array([0]), np.arange(n)[::-1][:5], np.arange(0, n, 7)):
            idx = i.astype(np.int32)
            mi = ctx.photometry(th[i], gal_idx=idx, mode="exact", prec=prec).cpu().numpy()
            assert np.abs(mi - m[i]).max() < 1e-5
            _, gi = ctx.loglike_grad(th[i], obs, sigma, mask, gal_idx=idx, mode="exact", prec=prec)
            assert _rel(gi.cpu().numpy(), g[i]) < 1e-3
    ctx.close()


@pytest.mark.parametrize("n", [40, 20000])
def test_exact_large_tile_and_row_order(n):
    """Enough rows for the 128-row tile; rows repeat a few galaxies in random
    order (gal_idx), so rows of one galaxy land in different tiles and must
    agree with the rows evaluated alone."""
    import paper_2506_19919_gb300 as pkg
    tabs, z, th = _case("part", 40)
    rng = np.random.default_rng(1)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z, tabs, "exact").numpy()
    obs = (ref - 1.0).astype(np.float32)
    sigma, mask = np.full(obs.shape, 0.05), np.full(40, 3, np.uint32)
    idx = rng.permutation(np.arange(n) % 40).astype(np.int32)
    _, gref, _ = O.loglike_and_grad(th, z, tabs, obs.astype(np.float64), sigma, mask, "exact")
    for prec, mtol, gtol in (("fp32", 2e-5, 1e-4), ("bf16", 5e-3, None), ("tf32x3", 1e-4, None)):
        m = ctx.photometry(th[idx], gal_idx=idx, mode="exact", prec=prec).cpu().numpy()
        assert np.abs(m - ref[idx]).max() < mtol
        ll, g = ctx.loglike_grad(th[idx], obs, sigma, mask, gal_idx=idx, mode="exact", prec=prec)
        g = g.cpu().numpy()
        if gtol:
            assert _rel(g, gref.numpy()[idx]) < gtol
        first = np.unique(idx, return_index=True)[1]         # a galaxy's rows, wherever they landed
        assert _rel(g, g[first][idx]) < 1e-3
    ctx.close()
