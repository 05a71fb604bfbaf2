"""The cluster V-cycle of grids whose coarsest level has more cells than a block has threads (odd
levels of large grids, csrc/k_cluster.cu), against the tiled FP64 V-cycle of the same grid.

Tolerance: a V-cycle here is about 100 half-sweeps of at most six FP32 operations per cell, each
2^-24 relative, on an operator that does not amplify: below 100 * 6 * 6e-8 = 4e-5 of max |z|."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny", [(656, 400), (672, 400), (864, 432), (1008, 496), (1040, 496)])
def test_vcycle_with_a_wide_coarsest_level(nx, ny):
    rng = np.random.default_rng(nx)
    z = []
    for precision in (pkg.FP64_BATCHED, pkg.MIXED):
        cfg = pkg.default_config(nx, ny, n_members=1, n_steps=2, n_window=1, precision=precision)
        ens = pkg.Ensemble(cfg)
        if not z:
            x = cfg.x0 + (np.arange(nx) + 0.5) * (cfg.x1 - cfg.x0) / nx
            y = cfg.y0 + (np.arange(ny) + 0.5) * (cfg.y1 - cfg.y0) / ny
            fluid = (y[:, None] > 0) | ((x > 0) & (x < 1))[None, :]
            r = np.where(fluid, rng.standard_normal((ny, nx)).astype(np.float32), 0.0)
            r = np.where(fluid, (r - r[fluid].mean()).astype(np.float32), 0.0)
        z.append(ens.apply_preconditioner(r).cpu().numpy())
        ens.close()
    assert np.abs(z[1] - z[0]).max() <= 4e-5 * np.abs(z[0]).max()
