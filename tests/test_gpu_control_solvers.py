"""The solvers in control space at the sizes where their split changes: the H^1 conjugate gradients on one
to sixteen thread blocks per component, with ragged last blocks, and the kept eigenpairs of the Lanczos
projection, computed apart or, where they lie close, by diagonalising the whole projection.

Tolerances: the conjugate gradients stop at 1e-13 of |b|, and the operator's smallest eigenvalue is 1, so |x - x*| is
at most 1e-13 |b|; the right-hand side is noise of unit variance, so 1e-11 of max |x| + 1e-9 is above it and rounding.
A kept pair's residual is below 1e-12 of the largest eigenvalue by the convergence test, 1e-11 with rounding.  Vectors
computed apart mix by m eps over the least gap (1e-7), 1.6e-7 at order 144, and the correction squares that: 1e-12.
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


# distinct eigenvalues; 48 of a fast-decaying spectrum (close ones among the last); a square set (exactly degenerate pairs)
@pytest.mark.parametrize("nx,ny,N,region,a", [(96, 48, 4, None, 0.05), (176, 80, 31, None, 0.05), (96, 48, 96, None, 0.12),
                                              (128, 64, 12, (0.2, 0.8, -0.8, -0.2), 0.1)])
def test_eigenpairs_apart_and_close(nx, ny, N, region, a):
    kw = {} if region is None else {"region": region}
    cfg = pkg.default_config(nx, ny, n_members=N, n_steps=2, n_window=1, precision=pkg.FP64_BATCHED, corr_len=a, **kw)
    ens = pkg.Ensemble(cfg)
    lam = ens.use_eigen_ensemble()
    E = ens.get_ensemble().cpu().numpy()
    ens.close()
    P = oracle.cavity_params(nx, ny, cfg.Re)
    B = oracle.covariance_B(P, cfg.sigma, a, *(() if region is None else (region,)))
    n = B.shape[0]
    if region is None:
        ref = np.linalg.eigvalsh(B)[::-1]
        np.testing.assert_allclose(lam[::2], ref[:len(lam[::2])], rtol=0, atol=1e-11 * ref[0])
    for comp in (0, 1):
        V = E[comp * n:(comp + 1) * n, comp::2]
        V = V / np.linalg.norm(V, axis=0)
        assert np.linalg.norm(B @ V - V * lam[comp::2], axis=0).max() <= 1e-11 * lam[0]
        assert np.abs(V.T @ V - np.eye(V.shape[1])).max() <= 1e-12
