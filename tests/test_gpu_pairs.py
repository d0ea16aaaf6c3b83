"""The FP32 kernels that carry sums and products as pairs (cell gradient, volume normalisation, coefficient set-up):
ragged sizes, values from subnormal to overflowing, infinities and NaN, and volumes that are not 16-byte aligned."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402


def engine(nx, ny, nz, n_src=1, n_freq=2, **kw):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=nx - 6, n_core_y=ny - 6, n_core_z=nz - 6, npml=3, n_freq=n_freq, nt=8)
    src = W.Points.make([[wl.src.x[0], 20.0 * s, wl.src.z[0]] for s in range(n_src)], 0)
    return wl, src, Engine.from_workload(wl, max_src=n_src, autotune=False, **kw)


def reference(eng, wl, rho, E, V, wrt):
    """The gradient in FP64 from FP32-rounded edge sums, and the bound of its FP32 rounding per cell."""
    p = -(E.to(torch.complex128) * V.to(torch.complex128)).real.sum(dim=(0, 2))[..., :eng.nx + 1]
    dV = [torch.as_tensor(np.diff(a), device="cuda") for a in (wl.zn, wl.yn, wl.xn)]
    vol = 0.25 * dV[0][:, None, None] * dV[1][None, :, None] * dV[2][None, None, :]

    def cells(q, comp):
        for a in {0: (0, 1), 1: (0, 2), 2: (1, 2)}[comp]:
            n = q.shape[a]
            q = q.narrow(a, 0, n - 1) + q.narrow(a, 1, n - 1)
        return q.narrow(2 - comp, 0, q.shape[2 - comp] - 1)
    out, mag = [], []
    for c in (0, 1, 2):
        out.append(vol * cells(p[c], c))
        mag.append(vol * cells(p[c].abs(), c))
    if eng.vti:
        g, m = torch.stack([out[0] + out[1], out[2]]), torch.stack([mag[0] + mag[1], mag[2]])
    else:
        g, m = out[0] + out[1] + out[2], mag[0] + mag[1] + mag[2]
    if wrt == "lnrho":
        g, m = -g / rho.double(), m / rho.double()
    # every edge sum and the result are rounded to FP32 once: 2^-24 of the magnitudes each
    return g, 2.0 ** -23 * m + 1e-44 * vol.max()


@pytest.mark.parametrize("nx,ny,nz,n_src,vti,scale", [(13, 14, 17, 1, False, 1.0), (22, 10, 9, 3, True, 1e-14),
                                                      (131, 11, 16, 2, False, 1e6), (129, 9, 10, 1, True, 1e-3)])
def test_cell_gradient_matches_fp64(nx, ny, nz, n_src, vti, scale):
    wl, src, eng = engine(nx, ny, nz, n_src, vti=vti)
    g = torch.Generator(device="cuda").manual_seed(7)
    vs = eng.volume_shape(n_src)
    E, V = (scale * torch.randn(vs, generator=g, device="cuda", dtype=torch.complex64) for _ in range(2))
    rho = torch.rand(eng.model_shape, generator=g, device="cuda") + 0.3
    for wrt in ("lnrho", "sigma"):
        got = eng.gradient(rho, E, V, wrt=wrt)
        ref, bound = reference(eng, wl, rho, E, V, wrt)
        assert bool(((got.double() - ref).abs() <= bound).all())
    # the same from buffers on an odd multiple of eight bytes
    for x in (E, V):
        buf = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")
        buf[1:] = x.reshape(-1)
        y = buf[1:].view(vs)
        assert y.data_ptr() % 16 == 8
        a, b = (y, V) if x is E else (E, y)
        got = eng.gradient(rho, a, b)
        ref, bound = reference(eng, wl, rho, E, V, "lnrho")
        assert bool(((got.double() - ref).abs() <= bound).all())
    eng.close()


def test_cell_gradient_of_large_and_non_finite_volumes():
    wl, src, eng = engine(20, 17, 15)
    g = torch.Generator(device="cuda").manual_seed(3)
    vs = eng.volume_shape(1)
    E, V = (torch.randn(vs, generator=g, device="cuda", dtype=torch.complex64) for _ in range(2))
    E[0, 0, 0, 5, 5, 5], V[0, 0, 0, 5, 5, 5] = 3e25, 2e12          # overflows scaled, not as it is
    E[0, 1, 1, 8, 6, 7], V[0, 1, 1, 8, 6, 7] = complex(2e30, 2e30), complex(1e10, 1e10)   # inf - inf in FP32, 0 in FP64
    E[0, 2, 0, 3, 9, 9] = float("inf")
    E[0, 2, 1, 11, 4, 4] = float("nan")
    rho = torch.ones(eng.model_shape, device="cuda")
    got = eng.gradient(rho, E, V, wrt="sigma").double()
    ref, bound = reference(eng, wl, rho, E, V, "sigma")
    small = ref.abs() < 3e38
    assert bool((torch.isnan(got) == torch.isnan(ref)).all())
    assert bool((torch.isinf(got) == (torch.isinf(ref) | (ref.abs() >= 3.5e38))).all())
    assert bool(((got - ref).abs() <= bound)[small & torch.isfinite(ref)].all())
    eng.close()


@pytest.mark.parametrize("vti", [False, True])
@pytest.mark.parametrize("nx,ny,nz", [(18, 17, 19), (131, 10, 9)])
def test_extreme_resistivities_step_as_in_fp64(nx, ny, nz, vti):
    """Cells outside the range of pairs take the general evaluation; volumes agree with an FP64 context."""
    wl, src, e32 = engine(nx, ny, nz, vti=vti, kahan=1)
    _, _, e64 = engine(nx, ny, nz, vti=vti, precision=64, kahan=0)
    rho = np.broadcast_to(wl.rho, e32.model_shape).copy()
    rho.reshape(-1)[[700, 801, 902]] = 1e-14, 1e-20, 5e-13
    out = []
    for e in (e32, e64):
        _, v = e.fwd_model(e.model_tensor(rho.astype(np.float32)), src, wl.rec, keep_volume=True)
        e.check()
        out.append(v[..., :nx + 1].to(torch.complex128))
        e.close()
    assert (out[0] - out[1]).norm() <= 1e-6 * out[1].norm()        # 8 FP32 steps


def test_bad_resistivity_is_reported():
    from paper_2211_16665_gb300 import _capi
    wl, src, eng = engine(18, 17, 19)
    for bad in (0.0, -1.0, float("inf"), float("nan")):
        rho = eng.model_tensor(wl.rho)
        rho[9, 8, 7] = bad
        eng.fwd_model(rho, src, wl.rec)
        with pytest.raises(_capi.CsemError):
            eng.check()
        eng.fwd_model(eng.model_tensor(wl.rho), src, wl.rec)
        eng.check()
    eng.close()
