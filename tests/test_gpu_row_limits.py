"""Step forms that need rows of a multiple of four cells."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("tune", [False, True])
@pytest.mark.parametrize("n_core", [20, 19])     # nx = 42, 41
def test_warp_specialised_step_is_refused_off_rows_of_four(n_core, tune):
    from paper_2211_16665_gb300._capi import CsemError
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=n_core, npml=8, ratio=1.05, n_st=3, n_rec=2, n_freq=2, nt=64)
    eng = Engine.from_workload(wl, autotune=tune)
    assert eng.nx % 4 != 0
    with pytest.raises(CsemError):
        eng.set_launch(wspec=(8, 4, 3))
    eng.close()
