"""The basis estimate at the edges of its range split (512 ranges per column, 64 per CTA, at most 128 samples each
in shared memory): one sample, fewer samples than ranges, ragged last ranges, the longest run that fits and the
first that does not, and every frequency count."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rows(dt, nt, freqs, f0):
    a = 2 * np.pi * np.sqrt(np.asarray(freqs) * f0)
    z = np.exp((-1 + 1j) * a[:, None] * ((np.arange(nt) + 0.5) * dt))
    return np.concatenate([z.real, z.imag])


def estimate(dt, nt, freqs, gamma, relative=1):
    from paper_2211_16665_gb300 import _capi
    out = torch.full((nt, 2 * len(freqs)), float("nan"), dtype=torch.float64, device="cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    fit, its = _capi.estimate_adjoint_basis(dt, nt, np.asarray(freqs, float), 1.0, gamma, relative, 400, 1e-14,
                                            ctypes.c_void_p(out.data_ptr()), st)
    return out.cpu().numpy(), fit, its


@pytest.mark.parametrize("nt", [1, 31, 511, 512, 513, 1025, 65536, 65537])
@pytest.mark.parametrize("nf", [1, 2, 3])
def test_basis_matches_the_dense_solution(nt, nf):
    freqs = [0.2, 0.7, 2.0][:nf]
    dt = 4.0 / (nt + 1)
    gamma = 1e-3
    x, fit, its = estimate(dt, nt, freqs, gamma)
    B = rows(dt, nt, freqs, 1.0)
    G = B @ B.T
    g = gamma * np.linalg.eigvalsh(G)[-1]
    ref = B.T @ np.linalg.inv(G + g * np.eye(2 * nf))
    # condition number of G + g I at most 1 + 1/gamma = 1e3; CG stops at 1e-14 of the right-hand side and the
    # dense solution carries cond * eps: 1e3 * (1e-14 + 2e-16 * sums) is below 1e-10
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
    assert abs(fit - np.abs(B @ x - np.eye(2 * nf)).max()) <= 1e-10
    assert its <= 2 * nf + 6


@pytest.mark.parametrize("nf", range(1, 9))
def test_every_frequency_count_gives_its_fit(nf):
    freqs = np.geomspace(0.1, 1.5, nf) if nf > 1 else [0.5]
    nt, dt = 3001, 2e-3
    x, fit, its = estimate(dt, nt, freqs, 1e-6)
    B = rows(dt, nt, freqs, 1.0)
    # both products carry a rounding error of at most nt eps sum |B| |x| (worst case, nt eps = 7e-13)
    bound = 7e-13 * (np.abs(B) @ np.abs(x)).max() + 1e-12
    assert abs(fit - np.abs(B @ x - np.eye(2 * nf)).max()) <= bound
    assert 0 < its <= 400
