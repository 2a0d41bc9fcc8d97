"""Observables of an ill-conditioned factor (the allocation-free call takes any) against long double.

||[rho, H]||^2 is judged by the error of the same formula, X = chol(V^*V)^{-1} and Gbar = X V^*HV X^H, evaluated by numpy in FP64 on
the same factors: both round the Grams alike, so over eight draws the r.m.s. errors differ by a factor of a few; ten is allowed.  (A
formula that loses another condition number is off by a hundred times at 1e5.)  V spans eight eigenvectors of H,
which makes the commutator the small difference of two large sums.
"""
import numpy as np
import pytest

import lrei_inputs as li
from oracle import model

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import load_library  # noqa: E402
from test_zz_no_alloc import _noalloc  # noqa: E402


def _inverse_factor(A):
    """L^{-1} for A = L L^H, column by column (any precision)."""
    k = len(A)
    L, X = np.zeros_like(A), np.zeros_like(A)
    for j in range(k):
        L[j, j] = np.sqrt(A[j, j].real - (np.abs(L[j, :j]) ** 2).sum())
        for i in range(j + 1, k):
            L[i, j] = (A[i, j] - (L[i, :j] * L[j, :j].conj()).sum()) / L[j, j]
    for j in range(k):
        for i in range(j, k):
            X[i, j] = ((1 if i == j else 0) - (L[i, j:i] * X[j:i, j]).sum()) / L[i, i]
    return X


def _commutator2(V, H, lam):
    HV = H @ V
    X = _inverse_factor(V.conj().T @ V)
    G, A = X @ (V.conj().T @ HV) @ X.conj().T, X @ (HV.conj().T @ HV) @ X.conj().T
    return 2 * (lam ** 2 * A.diagonal().real).sum() - 2 * (lam[:, None] * lam[None, :] * np.abs(G) ** 2).sum()


def _unitary(r, rng):
    return np.linalg.qr(rng.standard_normal((r, r)) + 1j * rng.standard_normal((r, r)))[0]


@pytest.mark.parametrize("scale", [1.0, 1e-100, 1e100])
@pytest.mark.parametrize("condition", [1e2, 1e4, 1e5])
def test_commutator(condition, scale):
    r = 8
    w = li.workload(2, n=8, r=r)
    H = np.asarray(model.hamiltonian(w.n, w.bonds, w.B))
    basis = np.linalg.eigh(H)[1][:, :r]
    rng = np.random.default_rng(int(np.log10(condition)))
    lib = load_library()
    err, plain = [], []
    for _ in range(8):
        V = basis @ _unitary(r, rng) @ np.diag(np.logspace(0, -np.log10(condition), r)) @ _unitary(r, rng)
        lam = np.sort(rng.dirichlet(np.ones(r)))[::-1]
        ref = float(_commutator2(V.astype(np.clongdouble), H.astype(np.clongdouble), lam))
        got = _noalloc(lib, w, torch.from_numpy(V * scale).cuda(), lam, 0)
        err.append(got["comm_norm"] ** 2 / ref - 1)
        plain.append(_commutator2(V, H, lam) / ref - 1)
    rms = lambda x: np.sqrt(np.mean(np.square(x)))  # noqa: E731
    assert rms(err) < 10 * rms(plain)
