"""Tabulated throughput curves in the per-galaxy set-up (double-float): the
segment of a sample coordinate that FP32 rounds up to the next sample.

Bars: magnitudes 1e-5 mag and the 13-column gradient 1e-4 of the row's largest
component against the FP64 oracle (the FP32 bars)."""
import numpy as np
import pytest

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("below", [5e-7, 2e-9, 0.3])
def test_wavelengths_just_below_the_samples(below):
    """Every redshifted wavelength `below` of a step under a sample of the curve:
    T and its slope are those of the segment that ends there."""
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(9)
    z = np.full(40, np.float32(0.37)).astype(np.float64)
    step, p0, n_tab = 25.0, 4000.0, 161
    nodes = (p0 + step * (np.arange(1, 300) - below)) / (1.0 + z[0])
    lam = np.concatenate([np.geomspace(900.0, nodes[0] - 5.0, 200), nodes])
    t = W.make_tables(rng, 9, 5, len(lam), 900.0, 9000.0, W._gauss_bands([5000.0]))
    t = W.with_bands(t, [W.BAND_TABLE], [p0], [step], [n_tab], rng.uniform(0.1, 1.0, n_tab))
    t.lam_ang = lam
    th = W.prior_draw(rng, 40)
    ctx = pkg.Context(t)
    ctx.set_galaxies(z, build_approx=True)
    ref = O.photometry(th, z, t, "approx").numpy()
    assert np.abs(ctx.photometry(th, mode="approx").cpu().numpy() - ref).max() < 1e-5
    obs = (ref - 1.0).astype(np.float32).astype(np.float64)
    sigma, mask = np.full(obs.shape, 0.05), np.full(40, 1, np.uint32)
    _, gr, _ = O.loglike_and_grad(th, z, t, obs, sigma, mask, "approx", wrt_z=True)
    gr = gr.numpy()
    _, g = ctx.loglike_grad_z(th, obs, sigma, mask, mode="approx")
    assert (np.abs(g.cpu().numpy() - gr).max(1) / np.abs(gr).max(1)).max() < 1e-4
    ctx.close()
