"""The complex64 tile passes of ranks that are no tile width (columns padded with zeros), and the right-hand side over them.

Bounds as for the other complex64 passes: Gram entries 2e-6 of their columns' norms (at most 256 rows per plain FP32 sum),
steps and right-hand sides 5e-6 of the norm against the same calls in complex128.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402

N = 13   # above the rows that are summed entry by entry


@pytest.mark.parametrize("m", [1, 3, 5, 8])
@pytest.mark.parametrize("r", [1, 2, 3, 5, 7, 9, 12, 15, 17, 24, 31])
def test_gram(r, m):
    L = Lrei(N, li.chain_bonds(N, False), (0.0, 0.0, 0.5), 0.1, "qll", "mixed", r)
    g = torch.Generator(device="cuda")
    g.manual_seed(r * 10 + m)
    V = torch.zeros((1 << N, r), dtype=torch.complex64, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    blocks = [torch.randn((1 << N, r), dtype=torch.complex64, device="cuda", generator=g) for _ in range(m)]
    P = L.gram(blocks).cpu().numpy()
    left = torch.cat(blocks, dim=1).cpu().numpy().astype(np.complex128)
    last = left[:, -r:]
    scale = np.linalg.norm(left, axis=0)[:, None] * np.linalg.norm(last, axis=0)[None, :]
    assert (np.abs(P - left.conj().T @ last) / scale).max() < 2e-6


def _contexts(r, mdl):
    w = li.workload(2, n=N, r=r)
    out = []
    for precision, dtype in (("fp64", torch.complex128), ("mixed", torch.complex64)):
        L = Lrei(w.n, w.bonds, w.B, w.kappa, mdl, precision, r)
        L.set_state(torch.from_numpy(w.V).to("cuda", dtype), w.lam)
        out.append(L)
    return out


def _close(a, b):
    a, b = a.to(torch.complex128), b.to(torch.complex128)
    return float((a - b).norm() / b.norm()) < 5e-6


@pytest.mark.parametrize("scheme,r", [("rk4", 1), ("rk4", 5), ("ab3", 7), ("rk4", 12), ("rk2", 20), ("rk4", 27)])
def test_step_matches_complex128(scheme, r):
    states = []
    for L in _contexts(r, "qllg"):
        L.step(0.005, scheme, 4)
        V, lam, _ = L.get_state()
        V = V.to(torch.complex128)
        X = torch.randn((1 << N, 4), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        states.append((V * torch.as_tensor(lam, device="cuda")) @ (V.mH @ X))   # rho X
    assert _close(states[1], states[0])


@pytest.mark.parametrize("complement", [0, 1])
@pytest.mark.parametrize("r", [1, 5, 8, 11, 16, 19])
def test_rhs_matches_complex128(r, complement):
    F = []
    for L in _contexts(r, "qll"):
        Z, W, _ = L.rhs(complement)
        V = L.get_state()[0].to(torch.complex128)
        Z, W = Z.to(torch.complex128), W.to(torch.complex128)
        X = torch.randn((1 << N, 4), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        F.append(Z @ (V.mH @ X) + V @ (W.mH @ X))   # f(rho) X
    assert _close(F[1], F[0])
