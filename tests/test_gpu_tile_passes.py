"""The complex64 tile passes (packed FP32 pairs) at every block count and rank they have an instance for.

Gram: a lane sums at most 256 rows (512 products) in FP32 before the compensated sums, so with random signs an
entry is off by about sqrt(512) 2^-25 = 7e-7 of its columns' norms; 2e-6 is asserted.  Projection and steps: against the same
calls in complex128, whose factors differ by FP32 roundings of the entries (6e-8 each, a few tens of them): 5e-6 of the norm.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 6, 8])
@pytest.mark.parametrize("n,r", [(5, 8), (10, 8), (5, 16), (10, 16), (6, 32), (10, 32)])
def test_gram(n, r, m):
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "mixed", r)
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 1000 + r * 10 + m)
    V = torch.zeros((1 << n, r), dtype=torch.complex64, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    blocks = [torch.randn((1 << n, r), dtype=torch.complex64, device="cuda", generator=g) for _ in range(m)]
    P = L.gram(blocks).cpu().numpy()
    left = torch.cat(blocks, dim=1).cpu().numpy().astype(np.complex128)
    last = left[:, -r:]
    scale = np.linalg.norm(left, axis=0)[:, None] * np.linalg.norm(last, axis=0)[None, :]
    assert (np.abs(P - left.conj().T @ last) / scale).max() < 2e-6


@pytest.mark.parametrize("scheme,r", [("rk1", 8), ("rk4", 8), ("ab4", 8), ("rk1", 16), ("rk2", 16), ("rk4", 16), ("ab3", 16),
                                      ("rk1", 32), ("rk2", 32), ("rk3", 32), ("rk4", 32)])
def test_step_matches_complex128(scheme, r):
    n = 9
    w = li.workload(2, n=n, r=r)
    rho = {}
    for precision, dtype in (("fp64", torch.complex128), ("mixed", torch.complex64)):
        L = Lrei(w.n, w.bonds, w.B, w.kappa, "qllg", precision, r)
        L.set_state(torch.from_numpy(w.V).to("cuda", dtype), w.lam)
        L.step(0.005, scheme, 5)
        V, lam, _ = L.get_state()
        V = V.to(torch.complex128)
        rho[precision] = (V * torch.as_tensor(lam, device="cuda")) @ V.mH
    assert float((rho["mixed"] - rho["fp64"]).norm() / rho["fp64"].norm()) < 5e-6
