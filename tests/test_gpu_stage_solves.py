"""The small dense solves of a step (Cholesky with inverse, FP32 Jacobi and replay, Newton passes, FP64 Jacobi) at the
edges of their ranges: ranks 1 to 32 (K = 5 .. 160, odd and even), eigenvalues equal, spread and nearly equal.

Bound on rho = V Lambda V^*: an eigenvector's error is C eps |M| / gap with gap ~ lambda_i - lambda_j, and enters rho times
lambda_i - lambda_j, so rho is off by C eps |M| <= C eps whatever the gaps; C <~ 10 K <= 1600 leaves 4e-13 < 1e-12.
"""
import numpy as np
import pytest

import lrei_inputs as li
from oracle import model, dense_ei as de

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402

SPECTRA = {
    "equal": lambda r: np.ones(r),
    "spread": lambda r: 0.8 ** np.arange(r),
    "near": lambda r: 1.0 - 1e-9 * np.arange(r),
}


@pytest.mark.parametrize("spectrum", sorted(SPECTRA))
@pytest.mark.parametrize("r", [1, 2, 7, 16, 31, 32])
def test_step_matches_dense(r, spectrum):
    n = 8
    w = li.workload(1, n=n, r=r)
    rng = np.random.default_rng(100 * r + len(spectrum))
    V = np.linalg.qr(rng.standard_normal((1 << n, r)) + 1j * rng.standard_normal((1 << n, r)))[0]
    lam = SPECTRA[spectrum](r)
    lam = lam / lam.sum()
    H = model.hamiltonian(n, w.bonds, w.B)
    L = Lrei(n, w.bonds, w.B, 0.4, "qll", "fp64", r)
    L.set_state(torch.from_numpy(V).to("cuda"), lam)
    L.step(0.02, "rk4", 1)
    Vd, mud = de.ei_rk_step(V, lam, H, 0.4, "qll", 0.02, "rk4")
    Vg, lg, _ = L.get_state()
    Vg = Vg.cpu().numpy()
    assert np.abs(Vg.conj().T @ Vg - np.eye(r)).max() < 1e-12
    assert np.abs(de.state(Vg, lg) - de.state(Vd, lam)).max() < 1e-12
    assert np.abs(L.observables()["ritz"] - mud).max() < 1e-12
