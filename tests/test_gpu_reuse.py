"""Runs do not clear their volumes or their whole snapshot ring: what an earlier run, another launch configuration
or another owner of the memory left there must not reach a result."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_16665_gb300 import workloads as W  # noqa: E402

LEAN = dict(kz_h=4, mb_h=8, kz_e=4, mb_e=8, lean_h=2, lean_e=2)
CONFIGS = [dict(block=16), dict(block=32, flush_mode=1), dict(block=64, flush_mode=1), dict(block=128, flush_mode=1),
           dict(block=128, flush_mode=0), dict(LEAN, block=64, flush_mode=3), dict(LEAN, block=16, flush_mode=1)]


def engine(nt=200, n_freq=2, **kw):
    from paper_2211_16665_gb300.engine import Engine
    wl = W.small_box(n_core=16, n_core_y=13, n_core_z=14, npml=6, n_freq=n_freq, nt=nt)
    return wl, Engine.from_workload(wl, autotune=False, **kw)


def poison(shape, dtype):
    t = torch.full(shape, float("nan"), dtype=dtype, device="cuda")
    del t           # the caching allocator gives this block to the next request of its size


@pytest.mark.parametrize("nt", [1, 15, 64, 65, 128, 200, 321])
def test_volumes_are_written_not_accumulated_into(nt):
    wl, eng = engine(nt)
    rho = eng.model_tensor(wl.rho)
    basis, _, _ = eng.estimate_adjoint_basis()
    ref = None
    for cfg in CONFIGS:
        eng.set_launch(**cfg)
        out = []
        for _ in range(2):      # the second run also finds the first one's compensation terms
            poison(eng.volume_shape(1), eng.cplx)
            d, E = eng.fwd_model(rho, wl.src, wl.rec, keep_volume=True)
            poison(eng.volume_shape(1), eng.cplx)
            V = eng.adjoint_model(rho, wl.rec, d, basis)
            out.append((E, V))
        assert all(torch.equal(a, b) for a, b in zip(*out))
        assert all(bool(torch.isfinite(torch.view_as_real(x)).all()) for x in out[0])
        if ref is None:
            ref = out[0]
        # other kernels and block lengths only round differently: a few FP32 units per step
        assert all((a - b).norm() <= 1e-5 * b.norm() for a, b in zip(out[0], ref))
    eng.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_a_run_after_one_that_blew_up_is_that_of_a_fresh_engine(precision):
    wl, eng = engine(precision=precision)
    good, bad = eng.model_tensor(wl.rho), eng.model_tensor(wl.rho * 1e9)     # far above the stability limit: overflows
    kinds = [dict(block=16)] + ([dict(LEAN, block=64, flush_mode=1), dict(fused_kz=8, block=32),
                                 dict(onepass=(8, 4, 4), block=32), dict(wspec=(8, 4, 2), block=32),
                                 dict(wave=(2, 4, 8), block=32)] if precision == 32 else [dict(fused_kz=8, block=32)])
    for cfg in kinds:
        eng.set_launch(**cfg)
        d, E = eng.fwd_model(bad, wl.src, wl.rec, keep_volume=True)
        assert not bool(torch.isfinite(torch.view_as_real(E)).all())
        again = [eng.fwd_model(good, wl.src, wl.rec, keep_volume=True)]       # same configuration
        eng.fwd_model(bad, wl.src, wl.rec)
        other = kinds[0] if cfg is not kinds[0] else kinds[-1]
        eng.set_launch(**other)                                               # another one finds the ring as it is
        again.append(eng.fwd_model(good, wl.src, wl.rec, keep_volume=True))
        for c, got in zip((cfg, other), again):
            _, fresh = engine(precision=precision)
            fresh.set_launch(**c)
            want = fresh.fwd_model(good, wl.src, wl.rec, keep_volume=True)
            fresh.close()
            assert all(torch.equal(a, b) for a, b in zip(got, want))
    eng.close()
