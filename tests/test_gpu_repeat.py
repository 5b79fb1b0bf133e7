"""The same call on the same inputs gives the same bits: column parts of the
tensor-core forward, rows that share a redshift bucket, galaxy sets built
again, and seeded samplers on top of them."""
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


@pytest.mark.parametrize("n", [1025, 5000, 40001])
def test_rows_of_one_redshift_bucket_keep_their_order(n):
    G = 5000
    ctx, rng, _, obs, sigma, mask = _context(6, G, False)
    th = torch.as_tensor(W.prior_draw(rng, n).astype(np.float32)).cuda()
    idx = torch.as_tensor(rng.integers(0, G, n).astype(np.int32)).cuda()
    for prec in ("fp32", "bf16", "tf32x3"):
        _same(lambda: [ctx.photometry(th, gal_idx=idx, mode="exact", prec=prec),
                       *ctx.loglike_grad(th, obs, sigma, mask, gal_idx=idx, mode="exact", prec=prec)])
    ctx.close()


@pytest.mark.parametrize("zmax", [0.4501, 0.5, 3.0])
def test_redshift_order_of_many_rows(zmax):
    """One bucket for all rows, some tens, most of them: the row alone within
    1e-5 mag (another order of FP32 sums)."""
    G, n = 2500, 70001
    ctx, rng, _, _, _, _ = _context(2, G, False, zmax=zmax)
    th = W.prior_draw(rng, n).astype(np.float32)
    idx = rng.integers(0, G, n).astype(np.int32)
    m = ctx.photometry(torch.as_tensor(th).cuda(), gal_idx=torch.as_tensor(idx).cuda(), mode="exact").cpu().numpy()
    some = np.r_[np.arange(500), n - 1 - np.arange(500)]
    few = ctx.photometry(th[some], gal_idx=idx[some], mode="exact").cpu().numpy()
    assert np.isfinite(m).all() and np.abs(m[some] - few).max() < 1e-5
    ctx.close()


def test_galaxy_set_built_again():
    """The tables of a set are the same bits each time, and a galaxy's row of
    them does not depend on the others (sets of 16 and of 4 galaxies a block)."""
    ctx, rng, z, obs, sigma, mask = _context(4, 3000, True, zmax=3.0)
    th = torch.as_tensor(W.prior_draw(rng, 3000).astype(np.float32)).cuda()
    call = lambda: [ctx.photometry(th, mode="approx"),                                       # noqa: E731
                    *ctx.loglike_grad(th, obs, sigma, mask), *ctx.loglike_grad_z(th, obs, sigma, mask)]
    first = call()
    for _ in range(3):
        ctx.set_galaxies(z, build_approx=True)
        for a, b in zip(first, call()):
            assert torch.equal(a, b)
    for step in (2, 11):
        ctx.set_galaxies(z[1::step].copy(), build_approx=True)
        some = ctx.loglike_grad_z(th[1::step], obs[1::step], sigma[1::step], mask[1::step])
        for a, b in zip(first[3:], some):
            assert torch.equal(a[1::step], b)
    ctx.close()


@pytest.mark.parametrize("mode,prec", [("approx", "fp32"), ("exact", "bf16"), ("exact", "fp32")])
def test_seeded_chains(mode, prec):
    G = 1100
    runs = []
    for _ in range(3):
        ctx, rng, _, obs, sigma, mask = _context(4, G, mode == "approx")
        x0 = torch.as_tensor(rng.normal(0.0, 0.3, (G, 12)).astype(np.float32)).cuda()
        out = ctx.hmc_run(x0, obs, sigma, mask, chains_per_gal=1, n_warm=3, n_samp=3, L_min=2, L_max=6, eps0=0.01,
                          seed=7, mode=mode, prec=prec)
        torch.cuda.synchronize()
        runs.append(out["samples"].clone())
        ctx.close()
    for r in runs[1:]:
        assert torch.equal(r, runs[0])
