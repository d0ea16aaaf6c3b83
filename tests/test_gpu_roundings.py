"""Roundings of the FP32 step kernels.  Gradients multiply a rounding difference by up to 10^4 (the adjoint basis is
ill-conditioned), so the kernels spell their roundings out: traces equal the stored ones of the same kernels compiled
from plain expressions, and every instance with the same planes per thread (in a tuned context: every instance) gives
the same bits."""
import json
import os

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "step_roundings.json")
CONFIGS = {"order 2, %d planes" % kz: dict(order=2, kz=kz, mb=6) for kz in (1, 2, 4)}
CONFIGS["order 4"] = dict(order=4, kz=4, mb=6)
CONFIGS["order 4, odd rows"] = dict(order=4, kz=0, mb=0)        # nx = 45: the scalar kernels


def trace_of(order, kz, mb):
    """Traces of a 44^3 box with graded cells, every fourth step: [receiver][step], FP64 sums of FP32 field values."""
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=20 if mb else 21, n_st=4, ratio=1.05, npml=8, n_freq=2, nt=160, n_rec=3)
    eng = Engine.from_workload(wl, max_src=1, autotune=False, order=order)
    if mb:
        eng.set_launch(kz_h=kz, mb_h=mb, lean_h=2, kz_e=kz, mb_e=mb, lean_e=2)
    tr = eng.fwd_model(eng.model_tensor(wl.rho_true), wl.src, wl.rec, trace=True)[-1]
    eng.check()
    eng.close()
    return tr[0, :, 3::4].cpu()


@pytest.mark.parametrize("name", CONFIGS)
def test_traces_are_what_they_were(name):
    tr = trace_of(**CONFIGS[name])
    with open(GOLDEN) as f:
        want = torch.tensor(json.load(f)[name], dtype=torch.float64)
    assert want.abs().max() > 0
    # equal field bits leave the order and fusion of eight FP64 products: 16 roundings of 1.1e-16 of terms that are of
    # the order of the trace's peak.  One FP32 rounding on the way is 6e-8 of a value, 1e-3 of the peak or more.
    assert ((tr - want).abs().amax(-1) <= 1e-13 * want.abs().amax(-1)).all()


# 96 x 88 x 90 cells: some of these launches end in one-plane blocks (1.2 to 8 waves), the others do not
@pytest.mark.parametrize("kz", [1, 2, 4])
def test_instances_give_the_same_bits(kz):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=84, n_core_y=76, n_core_z=78, npml=6, n_freq=2, nt=64, n_rec=4)
    out = []
    for w, mb in ((1, 6), (1, 8), (2, 4), (2, 6), (2, 8)):
        eng = Engine.from_workload(wl, max_src=1, autotune=False)
        eng.set_launch(kz_h=kz, mb_h=mb, lean_h=w, kz_e=kz, mb_e=mb, lean_e=w)
        d, E = eng.fwd_model(eng.model_tensor(wl.rho_true), wl.src, wl.rec, keep_volume=True)
        eng.check()
        eng.close()
        out.append((d, E))
    for d, E in out[1:]:
        assert torch.equal(d, out[0][0]) and torch.equal(E, out[0][1])


# A tuned context fixes its rounding by the size of a launch: the same bits for every configuration, planes per thread
# among them, and for every tuning
@pytest.mark.parametrize("n,S", [(24, 1), (24, 3), (84, 1), (84, 3)])
def test_tuned_contexts_give_the_same_bits(n, S):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=n, n_core_y=n - 4, n_core_z=n - 3, npml=6, n_freq=2, nt=64, n_rec=4)
    x, z = wl.src.x[0], wl.src.z[0]
    src = W.Points.make([[x, 0.0, z], [x - 40.0, 90.0, z + 30.0], [x + 60.0, -50.0, z]][:S], [0, 1, 2][:S])
    out = []
    for again in range(2):
        eng = Engine.from_workload(wl, max_src=S)
        rho = eng.model_tensor(wl.rho_true)
        for w, kz, mb in ((1, 1, 6), (2, 1, 8), (1, 2, 8), (2, 2, 4), (1, 4, 6), (2, 4, 8)):
            eng.set_launch(kz_h=kz, mb_h=mb, lean_h=w, kz_e=kz, mb_e=mb, lean_e=w, block=16, flush_mode=0)
            out.append(eng.fwd_model(rho, src, wl.rec, keep_volume=True))
        eng.check()
        eng.close()
    for d, E in out[1:]:
        assert torch.equal(d, out[0][0]) and torch.equal(E, out[0][1])


# Fourth order: the same bits for every planes per thread and blocks per SM, with and without one-plane blocks
@pytest.mark.parametrize("nx", [96, 82])
def test_fourth_order_instances_give_the_same_bits(nx):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=nx - 12, n_core_y=76, n_core_z=78, npml=6, n_freq=2, nt=64, n_rec=4)
    out = []
    for kz in (2, 4, 8):
        for mb in (4, 6, 8):
            eng = Engine.from_workload(wl, max_src=1, autotune=False, order=4)
            eng.set_launch(kz_h=kz, mb_h=mb, lean_h=2, kz_e=kz, mb_e=mb, lean_e=2)
            d, E = eng.fwd_model(eng.model_tensor(wl.rho_true), wl.src, wl.rec, keep_volume=True)
            eng.check()
            eng.close()
            out.append((d, E))
    for d, E in out[1:]:
        assert torch.equal(d, out[0][0]) and torch.equal(E, out[0][1])


# Rows that are no multiple of four: the lean kernels round as the scalar or four-cell kernels that were picked there
# before, by the size of a launch, and add the taps of an edge one by one as they do.  118 x 93 x 97 cells with three sources exceed L2 (E walks z downwards), with one some launches end in
# one-plane blocks.
@pytest.mark.parametrize("nx,ny,nz,npml,S", [(47, 39, 41, 8, 2), (42, 37, 38, 5, 1), (118, 93, 97, 7, 3),
                                             (111, 93, 97, 6, 1)])
def test_other_rows_round_as_the_general_kernels(nx, ny, nz, npml, S):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=nx - 2 * npml, n_core_y=ny - 2 * npml, n_core_z=nz - 2 * npml, npml=npml, n_freq=2,
                     nt=256, n_rec=5)
    x, z = wl.src.x[0], wl.src.z[0]
    src = W.Points.make([[x, 0.0, z], [x - 40.0, 90.0, z + 30.0], [x + 60.0, -50.0, z]][:S], [0, 1, 2][:S])
    eng = Engine.from_workload(wl, max_src=S)
    assert eng.nx == nx
    rho = eng.model_tensor(wl.rho_true)
    near = W.Points.make([[x + 9.0 * r, 5.0 * r, z] for r in range(5)], [0, 1, 0, 2, 0])   # they share edges
    resid = torch.randn((S, near.n, 2), generator=torch.Generator().manual_seed(1), dtype=torch.complex128).to(rho.device)
    basis, _, _ = eng.estimate_adjoint_basis()
    out = []
    for w, kz, mb in ((0, 1, 4), (1, 1, 8), (1, 4, 6), (2, 1, 6), (2, 2, 4), (2, 2, 8), (2, 4, 6)):
        cells = nx * ny * nz * S
        eng.set_launch(kz_h=kz, mb_h=mb, lean_h=w, vec_h=int(w == 0 and cells >= 200e3), kz_e=kz, mb_e=mb, lean_e=w,
                       vec_e=int(w == 0 and cells >= 1.8e6))
        d, E = eng.fwd_model(rho, src, wl.rec, keep_volume=True)
        V = eng.adjoint_model(rho, near, resid, basis)
        out.append((d, E, V))
    eng.check()
    eng.close()
    for got in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got, out[0]))
