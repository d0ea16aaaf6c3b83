"""Launches of a few waves: the planes of the last, partial wave go to blocks of one plane.  Runs whose launches end in
such blocks are compared with scalar kernels (which have none), plane by plane, so that a plane stepped twice or not
at all shows wherever it lies."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402


def waves(nz, per, kz, mb):
    return (nz + kz - 1) // kz * per / (152.0 * mb)


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("nz", [89, 90, 91])
@pytest.mark.parametrize("kz,mb", [(2, 4), (4, 4), (4, 6), (2, 8)])
def test_every_plane_is_stepped_once(order, nz, kz, mb):
    from paper_2211_16665_gb300.engine import Engine
    nx, ny, npml = 96, 88, 6
    if kz == 4 and mb == 6:                     # more rows, for a launch of more than 1.2 waves
        ny = 120
    assert 1.2 < waves(nz, 2 * (ny // 4), kz, mb) <= 8
    wl = W.small_box(n_core=nx - 2 * npml, n_core_y=ny - 2 * npml, n_core_z=nz - 2 * npml, npml=npml, n_freq=2,
                     nt=160, n_rec=4)
    src = W.Points.make([[wl.src.x[0], 0.0, wl.src.z[0]]], [0])
    out = []
    for lean in (0, 2):
        eng = Engine.from_workload(wl, max_src=1, autotune=False, order=order)
        if lean:
            eng.set_launch(kz_h=kz, mb_h=mb, lean_h=2, kz_e=kz, mb_e=mb, lean_e=2, block=32, flush_mode=1)
        d, E = eng.fwd_model(eng.model_tensor(wl.rho_true), src, wl.rec, keep_volume=True)
        eng.check()
        out.append((d, E))
        eng.close()
    # FP32 rounding of 160 steps, by plane: the fields of a plane come from planes around it, whose rounding errors
    # are some 1e-6 of them; a plane that missed a step or took one twice is off by a good part of itself
    a, b = out[1][1], out[0][1]
    z = b.dim() - 3
    for k in range(1, nz):
        x, y = a.select(z, k), b.select(z, k)
        assert (x - y).norm().item() <= 1e-3 * y.norm().item(), k
    assert (out[1][0] - out[0][0]).norm().item() <= 1e-5 * out[0][0].norm().item()
