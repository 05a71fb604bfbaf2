"""The H^1 conjugate gradients on one to sixteen thread blocks per component, with ragged last blocks.

Tolerance: the conjugate gradients stop at 1e-13 of |b|, and the operator's smallest eigenvalue is 1, so |x - x*| is
at most 1e-13 |b|; the right-hand side is noise of unit variance, so 1e-11 of max |x| + 1e-9 is above it and rounding.
"""
import numpy as np
import pytest

import oracle
import paper_2605_23812_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny", [(32, 16), (64, 32), (80, 48), (96, 48), (176, 80), (240, 112), (1024, 512)])
def test_h1_smoothing_over_the_splits(nx, ny):
    cfg = pkg.default_config(nx, ny, n_members=1, n_steps=2, n_window=1, precision=pkg.FP64_BATCHED)
    ens = pkg.Ensemble(cfg)
    g = np.random.default_rng(nx).standard_normal(ens.n_ctrl)
    gs = ens.h1_smooth(g, 0.02).cpu().numpy()
    assert np.array_equal(gs, ens.h1_smooth(g, 0.02).cpu().numpy())
    ens.close()
    ref = oracle.h1_smooth(oracle.cavity_params(nx, ny, cfg.Re), g, 0.02)
    np.testing.assert_allclose(gs, ref, rtol=1e-9, atol=1e-11 * np.abs(ref).max())
