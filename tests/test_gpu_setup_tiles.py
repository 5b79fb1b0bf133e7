"""The per-galaxy set-up (zero points, supports, lambda_eff, c_SSP and its
redshift derivative) at the sizes where its tiling changes: one galaxy, around
the 4- and 16-galaxy blocks and the switch between them, an odd number of
(age, Z) columns, bands that leave the wavelength grid, and Gaussian, top-hat
and tabulated bands side by side; against the FP64 oracle.

Bars: magnitudes 1e-5 mag (FP32 sums of positive terms, ~1e-6 relative, and the
FP32 output's 1e-6 mag at |m| ~ 25); the 13-column gradient 1e-4 of the row's
largest component (the FP32 bar)."""
import numpy as np
import pytest
import torch

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


def _tables(tophat):
    rng = np.random.default_rng(8)
    kind, p0, p1 = W._gauss_bands([3000.0, 4500.0, 11000.0])
    tk, t0, t1, tn, tT = W.tabulated_bands(rng, [500.0, 640.0])
    parts = [(kind, p0, p1, np.zeros(3, np.int32)), (tk, t0, t1, tn)]
    if tophat:
        parts.append((np.array([W.BAND_TOPHAT], np.int32), np.array([7000.0]), np.array([8200.0]),
                      np.zeros(1, np.int32)))
    base = W.make_tables(rng, 5, 3, 401, 900.0, 12000.0, (kind, p0, p1))      # 15 columns
    kind, p0, p1, tn = (np.concatenate([p[i] for p in parts]) for i in range(4))
    return W.with_bands(base, kind, p0, p1, tn.astype(np.int32), tT)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 17, 319, 320, 511, 512, 529])
def test_setup_tiles_match_oracle(n):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(100 + n)
    z = rng.uniform(0.05, 3.0, n).astype(np.float32).astype(np.float64)
    th = W.prior_draw(rng, n)
    tabs = _tables(True)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=True)
    for mode in ("approx", "exact"):
        m = ctx.photometry(th, mode=mode).cpu().numpy()
        assert np.abs(m - O.photometry(th, z, tabs, mode).numpy()).max() < 1e-5
    ctx.close()
    tabs = _tables(False)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=True)
    truth = O.photometry(W.prior_draw(rng, n), z, tabs, "approx").numpy()
    sigma = np.full(truth.shape, 0.05)
    mask = np.full(n, 0b1111, np.uint32)
    _, g = ctx.loglike_grad_z(th, truth, sigma, mask, mode="approx")
    _, ref, _ = O.loglike_and_grad(th, z, tabs, truth.astype(np.float32).astype(np.float64), sigma, mask, "approx",
                                   wrt_z=True)
    g, ref = g.cpu().numpy().astype(np.float64), ref.numpy()
    assert (np.abs(g - ref).max(1) / np.abs(ref).max(1)).max() < 1e-4
    ctx.close()
