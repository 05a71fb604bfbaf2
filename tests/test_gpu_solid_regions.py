"""The level-0 kernels of the tiled solve skip regions without a fluid cell and count on zeros there:
a preconditioner application with a right-hand side that is nonzero in solid cells must leave nothing
behind, and a run before and after it must agree bit for bit (the same kernels on the same numbers).
Grids that do not run whole in a cluster, one to three sweep pairs."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,precision,nu", [(1024, 512, pkg.MIXED, 1), (1024, 512, pkg.MIXED, 3), (840, 424, pkg.MIXED, 2),
                                                (512, 256, pkg.FP64_BATCHED, 2)])
def test_runs_agree_around_a_preconditioner_call(nx, ny, precision, nu):
    import torch
    cfg = pkg.default_config(nx, ny, n_members=1, n_steps=4, n_window=2, precision=precision, nu_pre=nu, nu_post=nu)
    ens = pkg.Ensemble(cfg)
    ens.set_initial_state(*synth.cavity_ic(nx, ny))
    w = np.array([0.5])
    ens.forward_ensemble(w)
    J = ens.cost()[0].copy()
    s = [t.clone() for t in ens.get_state(1)]
    r = torch.from_numpy(np.random.default_rng(1).standard_normal((ny, nx))).cuda()
    ens.apply_preconditioner(r)
    ens.forward_ensemble(w)
    assert np.array_equal(J, ens.cost()[0]) and J.min() > 0
    for a, b in zip(s, ens.get_state(1)):
        assert torch.equal(a, b)
    ens.close()
