"""The FP64 step kernels against the oracle where their thread order has edges: no slabs, slabs wider than what is
between them, rows that fill whole warps and that do not, every plane blocking, and every frequency count of the
register flush."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fdtd  # noqa: E402
from paper_2211_16665_gb300 import workloads as W  # noqa: E402


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("cx,cy,cz,npml", [(13, 9, 8, 0), (3, 4, 5, 5), (18, 13, 11, 8), (26, 8, 9, 3), (45, 6, 7, 10)])
@pytest.mark.parametrize("n_freq", [1, 3])
def test_fp64_runs_match_the_oracle(cx, cy, cz, npml, n_freq):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=cx, n_core_y=cy, n_core_z=cz, npml=npml, n_freq=n_freq, nt=90, n_rec=4,
                     layered_model=False, ratio=1.1, n_st=1)
    rng = np.random.default_rng(5)
    wl.rho = wl.rho * rng.uniform(0.3, 1.0, wl.rho.shape)
    wl.precision, wl.kahan = 64, 0
    pb = fdtd.problem_from_workload(wl)
    d0, E0 = fdtd.forward(pb, wl.rho, wl.src, wl.rec, keep_volume=True)
    Bp, _ = fdtd.adjoint_basis(pb, 1e-6)
    V0 = fdtd.adjoint(pb, wl.rho, wl.rec, d0, Bp)
    eng = Engine.from_workload(wl, precision=64, kahan=0, autotune=False)
    rho = eng.model_tensor(wl.rho)
    for kz, mb in ((1, 4), (2, 8), (4, 6), (8, 4)):
        eng.set_launch(kz_h=kz, mb_h=mb, kz_e=kz, mb_e=mb, block=32)
        d, E = eng.fwd_model(rho, wl.src, wl.rec, keep_volume=True)
        V = eng.adjoint_model(rho, wl.rec, torch.as_tensor(d0, device="cuda"), torch.as_tensor(Bp, device="cuda"))
        eng.check()
        # 90 steps, each rounding a few 1e-16: far below 1e-12, far above any wrong coefficient
        assert rel(d.cpu().numpy(), d0) <= 1e-12
        nx = eng.nx + 1
        assert rel(E[..., :nx].cpu().numpy(), np.asarray(E0)[..., :nx]) <= 1e-12
        assert rel(V[..., :nx].cpu().numpy(), np.asarray(V0)[..., :nx]) <= 1e-12
    eng.close()
