"""A sampler run replayed from its captured graph after the galaxy tables have
moved: a larger set in between frees and reallocates them.  The chains are
those of a fresh context, bit for bit."""
import numpy as np
import pytest
import torch

import sps_workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sampler", ["hmc", "nuts"])
def test_graph_follows_the_galaxy_tables(sampler):
    import paper_2506_19919_gb300 as pkg
    rng = np.random.default_rng(12)
    t = W.make_tables(rng, 19, 7, 901, 900.0, 12000.0, W._gauss_bands([3600.0, 5500.0, 8000.0]))
    G, C = 40, 2
    z = rng.uniform(0.05, 1.0, 4000).astype(np.float32)
    x0 = torch.as_tensor(rng.normal(0.0, 0.3, (G * C, 12)).astype(np.float32)).cuda()
    obs = torch.as_tensor(rng.normal(20.0, 1.0, (G, 3)).astype(np.float32)).cuda()
    sigma, mask = torch.full((G, 3), 0.1, device="cuda"), torch.full((G,), 7, dtype=torch.int32, device="cuda")
    th = torch.as_tensor(W.prior_draw(rng, 4000).astype(np.float32)).cuda()

    def run(ctx):
        out = ctx.hmc_run(x0, obs, sigma, mask, chains_per_gal=C, n_warm=2, n_samp=3, L_min=2, L_max=6, max_depth=4,
                          sampler=sampler, seed=3)
        return out["samples"].cpu().numpy()

    fresh = pkg.Context(t)
    fresh.set_galaxies(z[:G])
    ref = run(fresh)
    fresh.close()
    ctx = pkg.Context(t)
    for _ in range(2):
        ctx.set_galaxies(z[:G])
        assert np.array_equal(run(ctx), ref)
        ctx.set_galaxies(z)
        ctx.photometry(th, mode="approx")
    ctx.close()
