"""The blocks of a cluster pressure solve wait for one another a limited number of tries.  With a limit of
none, a solve whose data is still under way gives up: the member's status has to say so, whichever block gave up and in each form of
the kernel (whole solve, one launch per refinement, V-cycle from level 1 on), and the handle has to run afterwards
as a new one does, bit for bit."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu

WAIT_LIMIT = 0


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,precision,conditional", [(128, 64, pkg.FP64_BATCHED, 1), (256, 128, pkg.MIXED, 0), (512, 256, pkg.MIXED, 1),
                                                         (672, 400, pkg.MIXED, 1), (1024, 512, pkg.MIXED, 0)])
def test_a_wait_that_runs_out_is_reported(nx, ny, precision, conditional):
    cfg = pkg.default_config(nx, ny, n_members=2, n_steps=3, n_window=1, precision=precision, conditional_refinement=conditional, max_outer=40)

    def new():
        ens = pkg.Ensemble(cfg)
        ens.set_initial_state(*synth.cavity_ic(nx, ny))
        return ens

    def run(ens):
        ens.forward_ensemble(np.array([0.3, -0.2]))
        return ens.member_status(), [t.cpu().numpy() for t in ens.get_state(2)]

    ens = new()
    ens.set_diagnostic(WAIT_LIMIT, 0)
    assert (run(ens)[0] & pkg.ST_DIVERGENCE).all()
    ens.set_diagnostic(WAIT_LIMIT, -1)
    status, state = run(ens)
    ens.close()
    fresh = new()
    status0, state0 = run(fresh)
    fresh.close()
    assert (status == 0).all() and (status0 == 0).all()
    for a, b in zip(state, state0):
        assert np.array_equal(a, b)


def test_a_preconditioner_application_that_ran_out_is_refused():
    nx, ny = 1024, 512
    ens = pkg.Ensemble(pkg.default_config(nx, ny, n_members=1, n_steps=2, n_window=1, precision=pkg.MIXED))
    r = np.random.default_rng(0).standard_normal((ny, nx))
    r[:ny // 2] = 0.0                                        # the channel's cells alone: zero in solid cells
    z = ens.apply_preconditioner(r).cpu().numpy()
    ens.set_diagnostic(WAIT_LIMIT, 0)
    with pytest.raises(pkg.EnvarError):
        ens.apply_preconditioner(r)
    ens.set_diagnostic(WAIT_LIMIT, -1)
    assert np.array_equal(z, ens.apply_preconditioner(r).cpu().numpy())
    ens.close()
