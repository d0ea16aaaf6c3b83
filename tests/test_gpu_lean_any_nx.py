"""Row lengths that are no multiple of four: the autotuner may pick the lean kernels there (their last pair of cells
may hold the entry nx of the row, and the high x slab starts on an even cell), so a tuned run is compared with the
scalar kernels of an untuned context, for the run of each kind."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402


def rel(a, b):
    return (a - b).norm().item() / b.norm().item()


@pytest.mark.parametrize("nx,npml", [(17, 6), (23, 5), (33, 1), (66, 7), (67, 8), (129, 10), (131, 3), (30, 0)])
@pytest.mark.parametrize("vti", [False, True])
def test_tuned_runs_match_scalar_kernels(nx, npml, vti):
    from paper_2211_16665_gb300.engine import Engine, misfit
    wl = W.small_box(n_core=nx - 2 * npml, n_core_y=14, n_core_z=15, npml=npml, n_freq=3, nt=320, n_rec=5)
    src = W.Points.make([[wl.src.x[0], 0.0, wl.src.z[0]], [wl.src.x[0] - 40.0, 90.0, wl.src.z[0]]], [0, 1])
    out = []
    for tune in (False, True):
        eng = Engine.from_workload(wl, max_src=2, autotune=tune, vti=vti)
        assert eng.nx == nx
        rho = eng.model_tensor(wl.rho_true if not vti else [wl.rho_true, wl.rho])
        if not tune:
            eng.set_launch(block=32)
        d, E = eng.fwd_model(rho, src, wl.rec, keep_volume=True)
        basis, _, _ = eng.estimate_adjoint_basis()
        r = misfit(2.0 * (out[0][0] if out else d), d)[1] if not out else misfit(2.0 * out[0][0], out[0][0])[1]
        V = eng.adjoint_model(rho, wl.rec, r, basis)
        t = eng.gradient_td(rho, src, wl.rec, r, segment=64)
        eng.check()
        pad = E[..., nx + 1:]
        assert not bool(torch.view_as_real(pad).any())
        out.append((d, E, V, t))
        eng.close()
    # FP32 rounding of 320 steps, measured between any two kernel families at 1e-7 .. 5e-7
    assert all(rel(b, a) <= 1e-5 for a, b in zip(*out))
