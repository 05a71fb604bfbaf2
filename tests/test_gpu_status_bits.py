"""A member's status word holds every bit that a block of the correction sets: a run whose solve ends above div_tol and
whose velocity leaves the finite numbers or the CFL limit reports both, in each of many identical runs."""
import numpy as np
import pytest

import paper_2605_23812_gb300 as pkg
from paper_2605_23812_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,precision", [(384, 120, pkg.MIXED), (192, 128, pkg.FP64_BATCHED), (64, 32, pkg.FP64_PLAIN)])
def test_no_bit_is_lost(nx, ny, precision):
    cfg = pkg.default_config(nx, ny, n_members=1, n_steps=1, n_window=0, precision=precision, max_outer=1, max_inner=1, div_tol=1e-10)
    ens = pkg.Ensemble(cfg)
    u0, v0 = synth.cavity_ic(nx, ny)
    bad = np.array(u0)
    bad[-2, nx // 4::nx // 8] = np.inf
    ens.set_initial_state(bad, v0)
    seen = set()
    for _ in range(300):
        ens.forward_ensemble(np.array([0.3]))
        seen.update(int(s) for s in ens.member_status())
    ens.close()
    assert len(seen) == 1 and seen.pop() & (pkg.ST_NONFINITE | pkg.ST_DIVERGENCE) == pkg.ST_NONFINITE | pkg.ST_DIVERGENCE
