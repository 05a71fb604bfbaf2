"""A preconditioner application to a right-hand side that is not finite must leave nothing behind: the
run after it has the bits of the run before it, on grids whose level-0 kernels skip regions without a fluid cell
and on grids that are solved whole in a cluster."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,precision,value", [(1024, 512, pkg.MIXED, np.nan), (1024, 512, pkg.MIXED, 1e300), (840, 424, pkg.MIXED, np.inf),
                                                   (512, 256, pkg.FP64_BATCHED, np.nan), (512, 256, pkg.MIXED, np.nan)])
def test_run_after_a_nonfinite_right_hand_side(nx, ny, precision, value):
    cfg = pkg.default_config(nx, ny, n_members=1, n_steps=3, n_window=1, precision=precision)
    ens = pkg.Ensemble(cfg)
    ens.set_initial_state(*synth.cavity_ic(nx, ny))

    def run():
        ens.forward_ensemble(np.array([0.5]))
        return ens.cost()[0].copy(), [t.cpu().numpy() for m in (0, 1) for t in ens.get_state(m)]

    J, state = run()
    assert np.isfinite(J).all()
    z = ens.apply_preconditioner(np.full((ny, nx), value)).cpu().numpy()
    assert not np.isfinite(z).all()
    J1, state1 = run()
    ens.close()
    assert np.array_equal(J, J1)
    for a, b in zip(state, state1):
        assert np.array_equal(a, b)
