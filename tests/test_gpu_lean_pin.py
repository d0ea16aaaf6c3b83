"""Lean kernels on rows that are no multiple of four: csem_autotune brings them (and their memory) there, and a tuned
context takes every configuration of them by hand, so a tuned run can be repeated."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402


def engine(nx, npml, tune=True, n_core_y=14, n_core_z=15, **kw):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=nx - 2 * npml, n_core_y=n_core_y, n_core_z=n_core_z, npml=npml, n_freq=2, nt=256, n_rec=5)
    eng = Engine.from_workload(wl, max_src=2, autotune=tune, **kw)
    assert eng.nx == nx
    return wl, eng


def test_memory_is_taken_by_tuning_only():
    from paper_2211_16665_gb300 import _capi
    wl, eng = engine(66, 7, tune=False, n_core_y=60, n_core_z=60)
    before = _capi.get_info(eng.ctx).workspace_bytes
    with pytest.raises(_capi.CsemError):
        eng.set_launch(lean_h=2, kz_h=1, mb_h=6)
    _capi.autotune(eng.ctx, 2, None)
    after = _capi.get_info(eng.ctx).workspace_bytes
    assert after - before >= (12 * 2 + 3) * eng.vol * 4
    _capi.autotune(eng.ctx, 2, None)
    assert _capi.get_info(eng.ctx).workspace_bytes == after
    eng.close()


@pytest.mark.parametrize("nx,npml", [(17, 6), (23, 5), (33, 1), (66, 7), (67, 8), (129, 10), (131, 3), (30, 0)])
def test_tuned_configuration_can_be_pinned(nx, npml):
    wl, eng = engine(nx, npml)
    cfg = eng.launch_config()
    step, fl = cfg["step"], cfg["flush"]
    runs = []
    for pin in (False, True):
        if pin and step["kernel"] == "split":
            kw = dict(block=fl["snapshots"], flush_mode=(fl["kernel"] == "bulk-copy") + 2 * fl["overlapped"])
            for h in "he":
                s = step[h]
                kw["kz_" + h] = s["z_planes"]
                kw["mb_" + h] = s.get("blocks_per_sm", 4)
                kw["lean_" + h] = s.get("cells_per_thread", 0)
                kw["vec_" + h] = int(s["kernel"] == "four cells per thread")
                kw["tma_" + h] = s.get("rows_per_block", 0)
            eng.set_launch(**kw)
            assert eng.launch_config() == cfg
        d, E = eng.fwd_model(eng.model_tensor(wl.rho_true), wl.src, wl.rec, keep_volume=True)
        runs.append((d.clone(), E.clone()))
    eng.check()
    eng.close()
    assert all(torch.equal(a, b) for a, b in zip(*runs))


# every lean configuration on odd rows and rows of 2 mod 4, against the scalar kernels: by column, so that the last
# cell pair (which may hold the entry nx) and the slabs' edges show
@pytest.mark.parametrize("nx,npml", [(17, 6), (23, 5), (33, 1), (66, 7), (67, 8), (129, 10), (131, 3), (30, 0)])
@pytest.mark.parametrize("kz", [1, 2, 4])
def test_every_lean_configuration_matches_scalar_kernels(nx, npml, kz):
    wl, eng = engine(nx, npml)
    rho = eng.model_tensor(wl.rho_true)
    src = W.Points.make([[wl.src.x[0], 0.0, wl.src.z[0]], [wl.src.x[0] - 40.0, 90.0, wl.src.z[0]]], [0, 1])
    out = []
    for w, mb in ((0, 4), (1, 6), (1, 8), (2, 4), (2, 6), (2, 8)):
        eng.set_launch(kz_h=kz, mb_h=mb, lean_h=w, kz_e=kz, mb_e=mb, lean_e=w)
        d, E = eng.fwd_model(rho, src, wl.rec, keep_volume=True)
        assert not bool(torch.view_as_real(E[..., nx + 1:]).any())
        out.append((d.clone(), E.clone()))
    eng.check()
    eng.close()
    d0, E0 = out[0]
    # 256 steps of FP32 rounding (6e-8 each) by column; a missed cell is off by a good part of itself
    for d, E in out[1:]:
        assert (d - d0).norm() <= 1e-5 * d0.norm()
        num = (E - E0).abs().square().sum(dim=(0, 1, 2, 3, 4)).sqrt()
        den = E0.abs().square().sum(dim=(0, 1, 2, 3, 4)).sqrt()
        assert (num <= 1e-3 * den + 1e-35).all()
