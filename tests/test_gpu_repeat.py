"""The same call on the same inputs gives the same bits: column parts of the
tensor-core forward."""
import numpy as np
import pytest
import torch

import sps_workloads as W

pytestmark = pytest.mark.gpu


def _context(n_band, G, approx, seed=2, zmax=0.5):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(seed)
    t = W.make_tables(rng, 19, 7, 901, 900.0, 12000.0, W._gauss_bands(np.geomspace(3600.0, 9000.0, n_band)))
    ctx = pkg.Context(t)
    z = rng.uniform(0.45, zmax, G).astype(np.float32)            # some tens of redshift buckets
    ctx.set_galaxies(z, build_approx=approx)
    obs = torch.as_tensor(rng.normal(20.0, 1.0, (G, n_band)).astype(np.float32)).cuda()
    sigma = torch.full((G, n_band), 0.1, device="cuda")
    mask = torch.full((G,), (1 << n_band) - 1, dtype=torch.int32, device="cuda")
    return ctx, rng, z, obs, sigma, mask


def _same(calls):
    first = calls()
    for _ in range(5):
        for a, b in zip(first, calls()):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n_band", [2, 6, 8, 9])
@pytest.mark.parametrize("prec", ["bf16", "tf32x3"])
def test_column_parts_add_up_in_order(n_band, prec):
    ctx, rng, _, obs, sigma, mask = _context(n_band, 100, False)
    th = torch.as_tensor(W.prior_draw(rng, 100).astype(np.float32)).cuda()
    _same(lambda: [ctx.photometry(th, mode="exact", prec=prec),
                   *ctx.loglike_grad(th, obs, sigma, mask, mode="exact", prec=prec),
                   *ctx.loglike_grad_z(th, obs, sigma, mask, mode="exact", prec=prec)])
    ctx.close()
