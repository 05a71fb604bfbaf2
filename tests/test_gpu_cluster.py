"""The cluster pressure solve (csrc/k_cluster.cu) at the sizes where its plan changes: one thread block
or several, 2 x 2 or 4 x 4 cells per thread, one to three gathered stages, an odd coarsest level, idle
threads, and grids that stay on the tiled kernels; trajectories against the FP64 oracle.

Tolerances: FP64 as in the parity tests, 1e-10 after 100 steps (here 6).  MIXED: a tendency is a sum of
terms of size u^2 / h rounded in FP32, so a step of dt = 0.3 h / U adds at most about 0.3 * 8 terms * 2^-24
= 1.4e-7 relative to U; six steps stay under 1e-6 of the velocity's norm.
"""
import numpy as np
import pytest

import oracle
import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


GRIDS = [(8, 4), (16, 8), (32, 16), (34, 18), (36, 20), (48, 16), (80, 48), (128, 80), (176, 80), (256, 128), (304, 144)]


@pytest.mark.parametrize("precision", [pkg.FP64_BATCHED, pkg.MIXED])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_trajectory_at_plan_edges(nx, ny, precision):
    N, steps = 1, 6
    P = oracle.cavity_params(nx, ny, 500.0)
    cfg = pkg.default_config(nx, ny, Re=500.0, n_steps=steps, n_window=2, n_members=N, precision=precision,
                             region=(-1.2, 2.5, -1.0, 1.0), corr_len=0.5, div_tol=1e-12 if precision != pkg.MIXED else 1e-11,
                             max_outer=40, max_inner=10)
    u0, v0 = synth.cavity_ic(nx, ny)
    ens = pkg.Ensemble(cfg)
    ens.set_initial_state(u0, v0)
    E = ens.get_ensemble().cpu().numpy()
    E[:] = 0.0                          # the flow without forcing: the oracle's control region is its default one
    ens.set_ensemble(E)
    ens.forward_ensemble(np.zeros(N))
    fu, fv = np.zeros((ny, nx + 1)), np.zeros((ny + 1, nx))
    ou, ov = oracle.trajectory(P, u0, v0, steps, fu, fv)[:2]
    assert (ens.member_status() == 0).all(), ens.diagnostics()
    tol = 1e-6 if precision == pkg.MIXED else 1e-10
    for m in range(N + 1):
        u, v, _ = (t.cpu().numpy() for t in ens.get_state(m))
        err = np.sqrt((((u - ou) ** 2).sum() + ((v - ov) ** 2).sum()) / ((ou**2).sum() + (ov**2).sum()))
        assert err <= tol, (m, err)
    ens.close()
