"""Star formation histories that peak long after t_obs (parameters outside the
prior, which the calls accept): the masses are denormal numbers, not zero.

Bar: 5e-3 mag against the FP64 oracle (a mass of 2^-138 keeps 11 bits)."""
import numpy as np
import pytest

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("z,tau,beta", [(12.0, 12.0, 24.0), (12.0, 40.0, 17.0), (19.5, 200.0, 12.0)])
def test_faint_histories(z, tau, beta):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(3)
    t = W.make_tables(rng, 31, 5, 1601, 91.0, 12000.0, W._gauss_bands([3600.0, 5500.0, 8000.0]))
    t.ssp = t.ssp * (1e18 / t.ssp.mean())                        # fluxes stay normal numbers
    zz = np.full(800, z, np.float32).astype(np.float64)
    th = W.prior_draw(rng, 800)
    th[:, 1], th[:, 3] = tau, beta
    th = th.astype(np.float32).astype(np.float64)
    ctx = pkg.Context(t)
    ctx.set_galaxies(zz, build_approx=True)
    k = 20                                                       # few rows, and as many as take the other kernels
    for mode, prec in (("approx", "fp32"), ("exact", "fp32"), ("exact", "bf16")):
        ref = O.photometry(th[:k], zz[:k], t, mode).numpy()
        for n in (k, 800):
            idx = np.arange(n, dtype=np.int32)
            m = ctx.photometry(th[:n], gal_idx=idx, mode=mode, prec=prec).cpu().numpy()
            assert np.abs(m[:k] - ref).max() < 5e-3, (mode, prec, n)
    ctx.close()
