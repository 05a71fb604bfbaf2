"""The pressure solve in a thread-block cluster against the tiled kernels of the same method on the same grid: one
preconditioned step of the conjugate gradients, and whole runs.

Tolerances.  One step moves the pressure by alpha z, z the V-cycle of the right-hand side.  Mixed handles smooth with the tiled
kernels' operations in their order, and only the sums in alpha differ in order: at most one ulp of alpha, 2^-23 of max |p|.
FP64 ones differ by the rounding of a reciprocal and of sums: about 100 half-sweeps of six operations of 2^-53,
7e-14 of max |z|, and as much again for alpha.  Runs: both solves stop at div_tol; FP64 as in the parity tests, 1e-10 of the
velocity's norm; mixed: where alpha rounds differently a tendency does (2^-24 of U per term, 0.3 * 8 terms a
step): 1e-6 over six steps."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu

TILED_SOLVE = 1
SOLVERS = [{}, {"nu_pre": 3, "nu_post": 3, "coarse_sweeps": 1, "nu_coarse": 2}, {"nu_pre": 1, "nu_post": 2}]
FP64_GRIDS = [(32, 16), (64, 32), (128, 64), (176, 80), (256, 128)]
GRIDS = [(pkg.FP64_BATCHED, *g) for g in FP64_GRIDS] + [(pkg.MIXED, *g) for g in FP64_GRIDS + [(304, 144), (512, 256), (592, 240)]]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def both(cfg, w):
    ens = pkg.Ensemble(cfg)
    ens.set_initial_state(*synth.cavity_ic(cfg.nx, cfg.ny))
    out = []
    for tiled in (1, 0):
        ens.set_diagnostic(TILED_SOLVE, tiled)
        ens.forward_ensemble(w)
        out.append(([[t.cpu().numpy() for t in ens.get_state(m)] for m in range(cfg.n_members + 1)], ens.member_status(), ens.diagnostics()))
    ens.close()
    return out


@pytest.mark.parametrize("solver", [0, 1, 2])
@pytest.mark.parametrize("precision,nx,ny", GRIDS)
def test_one_preconditioned_step(precision, nx, ny, solver):
    cfg = pkg.default_config(nx, ny, n_members=1, n_steps=1, n_window=1, precision=precision, max_outer=1, max_inner=1, **SOLVERS[solver])
    a, b = both(cfg, np.array([0.5]))
    tol = 2.0**-23 if precision == pkg.MIXED else 1.4e-13
    for (_, _, p), (_, _, q) in zip(a[0], b[0]):
        assert np.abs(p).max() > 0
        assert np.abs(p - q).max() <= tol * np.abs(p).max()


@pytest.mark.parametrize("conditional", [0, 1])
@pytest.mark.parametrize("precision,nx,ny", GRIDS)
def test_run_by_both_paths(precision, nx, ny, conditional):
    cfg = pkg.default_config(nx, ny, n_members=2, n_steps=6, n_window=2, precision=precision, conditional_refinement=conditional,
                             div_tol=1e-11 if precision == pkg.MIXED else 1e-12, max_outer=40, max_inner=10)
    a, b = both(cfg, np.array([0.4, -0.3]))
    assert (a[1] == 0).all() and (b[1] == 0).all(), (a[2], b[2])
    tol = 1e-6 if precision == pkg.MIXED else 1e-10
    for s, t in zip(a[0], b[0]):
        s, t = (np.concatenate([x.ravel() for x in q[:2]]) for q in (s, t))
        assert np.linalg.norm(s - t) <= tol * np.linalg.norm(s)
