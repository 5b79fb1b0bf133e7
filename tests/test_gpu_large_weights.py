"""Exact gradients of rows whose band weights gamma_b / c_b are near the largest
FP32 number (very faint rows, or data of very small errors): bands that overlap
must not overflow their sum.

Bar: 1e-3 of the row's largest component against the FP64 oracle for FP32, 3e-2
for BF16 (residuals of 1 mag of one sign: no cancellation)."""
import numpy as np
import pytest

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12, 1300])
def test_sum_over_bands_does_not_overflow(n):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(8)
    t = W.make_tables(rng, 19, 7, 901, 900.0, 12000.0, W._gauss_bands(np.linspace(5000.0, 5400.0, 6), 4.0, 4.0))
    z = np.full(n, 0.1, np.float32).astype(np.float64)
    th = W.prior_draw(rng, n)
    th[:, 0] = 0.0
    k = 12
    c = O.flux_exact(O._t(th[:k]), O._t(z[:k]), t)
    c = c[0].numpy() / 1e9                                      # per unit of 1e9 10^lgM
    ref = O.photometry(th[:k], z[:k], t, "exact").numpy()
    obs = np.tile(ref - 1.0, (n // k + 1, 1))[:n].astype(np.float32).astype(np.float64)
    # gamma_b / c_b of 2e38 in the faintest band: with six such bands the sum is 1e39
    sigma = np.full(obs.shape, np.sqrt(2.5 / np.log(10.0) / (2e38 * c.min())))
    idx = (np.arange(n) % k).astype(np.int32)
    mask = np.full(n, 63, np.uint32)
    ctx = pkg.Context(t)
    ctx.set_galaxies(z, build_approx=False)
    s32 = sigma.astype(np.float32).astype(np.float64)
    _, gr, _ = O.loglike_and_grad(th[:k], z[:k], t, obs[:k], s32[:k], mask[:k], "exact")
    gr = gr.numpy()
    for prec, tol in (("fp32", 1e-3), ("bf16", 3e-2)):
        _, g = ctx.loglike_grad(th[idx], obs, sigma, mask, gal_idx=np.arange(n, dtype=np.int32), mode="exact", prec=prec)
        g = g.cpu().numpy().astype(np.float64)
        assert (np.abs(g[:k] - gr).max(1) / np.abs(gr).max(1)).max() < tol, prec
        assert np.isfinite(g).all()
    ctx.close()
