"""The one-row-per-warp kernel of the approximate path (photometry with an
age-dependent MDF, and log L with the redshift column) against the FP64
oracle: row counts around the switches from one to two and to the most warps
per block, with idle warps in the last block; tables of 4 columns, of an odd
number of columns, of the most columns, and of more metallicities than half a
warp; one band and several, masks with no, one and all bands.

Bars: magnitudes 1e-5 mag, gradients 1e-4 of the row's largest component
(residuals of at least 1 mag, all of one sign: no cancellation between bands)."""
import numpy as np
import pytest

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_age,n_met,n_band", [(2, 2, 1), (31, 5, 3), (109, 12, 6), (25, 20, 4)])
@pytest.mark.parametrize("n", [1, 152, 153, 912, 1217])
def test_row_kernel_matches_oracle(n_age, n_met, n_band, n):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(n + n_age)
    bands = W._gauss_bands(np.geomspace(3000.0, 9000.0, n_band) if n_band > 1 else [5000.0])
    tabs = W.make_tables(rng, n_age, n_met, 500, 900.0, 12000.0, bands)
    G = 9
    z = rng.uniform(0.05, 1.0, G).astype(np.float32).astype(np.float64)
    idx = rng.integers(0, G, n).astype(np.int32)
    th = W.prior_draw(rng, n)
    some = np.unique(np.r_[0, n - 1, rng.integers(0, n, 30)])          # rows the oracle evaluates
    sigma = np.full((G, n_band), 0.05)
    mask = rng.integers(0, 1 << n_band, G, dtype=np.uint64).astype(np.uint32)
    mask[0], mask[1], mask[2] = 0, 1, (1 << n_band) - 1
    for mdf in (False, True):
        t = W.with_mdf_offset(tabs, W.mzr_offsets(tabs.age_yr, 0.4)) if mdf else tabs
        ctx = pkg.Context(t)
        ctx.set_galaxies(z, build_approx=True)
        ref = O.photometry(th[some], z[idx[some]], t, "approx").numpy()
        m = ctx.photometry(th, gal_idx=idx, mode="approx").cpu().numpy()
        assert np.abs(m[some] - ref).max() < 1e-5
        obs = np.full((G, n_band), m.min() - 1.0).astype(np.float32).astype(np.float64)
        ll, g = (x.cpu().numpy().astype(np.float64)
                 for x in ctx.loglike_grad_z(th, obs, sigma, mask, gal_idx=idx, mode="approx"))
        assert np.isfinite(ll).all() and np.isfinite(g).all()
        i = idx[some]
        llr, gr, _ = O.loglike_and_grad(th[some], z[i], t, obs[i], sigma[i], mask[i], "approx", wrt_z=True)
        gr = gr.numpy()
        scale = np.maximum(np.abs(gr).max(1, keepdims=True), 1e-30)
        assert (np.abs(g[some] - gr) / scale).max() < 1e-4
        np.testing.assert_allclose(ll[some], llr.numpy(), rtol=1e-5)
        ctx.close()
