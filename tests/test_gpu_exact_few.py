"""The exact path's weights and their adjoint for few rows (a block per row)
against the kernels that take a warp per row, by evaluating the same rows in a
call of few rows and, repeated, in one of more; and against the FP64 oracle:
tables of the fewest and the most ages, odd and many metallicities (more than
12 take the few-row weights with the general gradient), every precision, with
and without the redshift column, one row and both sides of the limit; a row
that is not finite.

Bars: the same row in the other call 1e-5 mag (one order of FP32 sums against
another) and 1e-3 of its largest gradient component (through the residual, and
through BF16 roundings that flip); FP32 against the oracle 2e-5 mag and 1e-4 of
the largest component (residuals of 1 mag of one sign: no cancellation)."""
import numpy as np
import pytest
import torch

import sps_workloads as W
from oracle import sps as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_age,n_met", [(2, 2), (31, 5), (33, 13), (109, 12), (128, 10), (25, 20)])
@pytest.mark.parametrize("n", [1, 9, 1216])
def test_few_rows_match_many_and_oracle(n_age, n_met, n):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(n + n_age)
    tabs = W.make_tables(rng, n_age, n_met, 401, 900.0, 12000.0, W._gauss_bands([3600.0, 5200.0, 7600.0]))
    G = 9
    z = rng.uniform(0.05, 1.0, G).astype(np.float32).astype(np.float64)
    th = W.prior_draw(rng, n)
    idx = rng.integers(0, G, n).astype(np.int32)
    ctx = pkg.Context(tabs)
    ctx.set_galaxies(z, build_approx=False)
    ref = O.photometry(th, z[idx], tabs, "exact").numpy()
    obs = np.full((G, 3), ref.min() - 1.0).astype(np.float32).astype(np.float64)
    sigma, mask = np.full((G, 3), 0.05), np.full(G, 7, np.uint32)
    many = np.arange(1217) % n                                # the same rows in a call of 1,217
    k = min(n, 40)
    _, gr, _ = O.loglike_and_grad(th[:k], z[idx[:k]], tabs, obs[idx[:k]], sigma[idx[:k]], mask[idx[:k]], "exact",
                                  wrt_z=True)
    gr = gr.numpy()
    for prec in ("fp32", "bf16", "tf32x3"):
        m = ctx.photometry(th, gal_idx=idx, mode="exact", prec=prec).cpu().numpy()
        mm = ctx.photometry(th[many], gal_idx=idx[many], mode="exact", prec=prec).cpu().numpy()
        assert np.abs(m[many] - mm).max() < 1e-5
        if prec == "fp32":
            assert np.abs(m - ref).max() < 2e-5
        for call in (ctx.loglike_grad, ctx.loglike_grad_z):
            ll, g = (x.cpu().numpy() for x in call(th, obs, sigma, mask, gal_idx=idx, mode="exact", prec=prec))
            lm, gm = (x.cpu().numpy() for x in call(th[many], obs, sigma, mask, gal_idx=idx[many], mode="exact",
                                                    prec=prec))
            assert (np.abs(g[many] - gm).max(1) / np.abs(gm).max(1)).max() < 1e-3
            np.testing.assert_allclose(ll[many], lm, rtol=1e-4)
            if prec == "fp32":
                r = gr[:, :g.shape[1]]
                assert (np.abs(g[:k] - r).max(1) / np.abs(r).max(1)).max() < 1e-4
    bad = torch.as_tensor(th, dtype=torch.float32, device="cuda")
    bad[0, 3] = float("nan")
    out = torch.zeros((n, 3), device="cuda")
    with pytest.raises(pkg.SpsError):
        ctx.photometry(bad, gal_idx=idx, mode="exact", out=out)
    out = out.cpu().numpy()
    assert np.isnan(out[0]).all()
    if n > 1:
        m = ctx.photometry(th, gal_idx=idx, mode="exact").cpu().numpy()
        assert np.abs(out[1:] - m[1:]).max() < 1e-5
    ctx.close()
