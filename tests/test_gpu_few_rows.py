"""Both sides of the line between the passes of few rows (up to 4096, a sum per entry) and the tiled ones.

Gram entries against long double, relative to their columns' norms: FP64 sums of N <= 2^14 random products are off by about
sqrt(N) 2^-53 = 1.4e-14 in the order of a plain sum, which both paths stay below by splitting it; 2e-14 is asserted for
complex128 and, for complex64 tiles (at most 256 rows per plain FP32 sum), 2e-6.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,r,m", [(3, 1, 1), (4, 5, 2), (9, 3, 1), (10, 3, 1), (10, 11, 4), (12, 7, 5), (12, 8, 4), (12, 8, 5),
                                   (13, 1, 1), (13, 5, 3), (13, 9, 2), (14, 17, 3)])
def test_gram(n, r, m, precision):
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", precision, r)
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 1000 + r * 10 + m)
    V = torch.zeros((1 << n, r), dtype=dt, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    blocks = [torch.randn((1 << n, r), dtype=dt, device="cuda", generator=g) for _ in range(m)]
    P = L.gram(blocks).cpu().numpy()
    left = torch.cat(blocks, dim=1).cpu().numpy().astype(np.clongdouble)
    last = left[:, -r:]
    norm = lambda X: np.sqrt((X.real ** 2 + X.imag ** 2).sum(0))  # noqa: E731
    err = np.abs(P - left.conj().T @ last) / (norm(left)[:, None] * norm(last)[None, :])
    assert err.max() < (2e-14 if precision == "fp64" else 2e-6)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,r", [(4, 3), (7, 5), (8, 7), (9, 11), (10, 4), (12, 6), (13, 6)])
def test_set_state_is_orthonormal(n, r, precision):
    # a projection in place: columns 100 apart become orthonormal and keep the density matrix
    g = torch.Generator()
    g.manual_seed(n * 100 + r)
    Q = torch.linalg.qr(torch.randn((1 << n, r), dtype=torch.complex128, generator=g))[0]
    V = (Q * torch.logspace(-1, 1, r, dtype=torch.float64)).cuda()
    lam = np.full(r, 1.0 / r)
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", precision, r)
    L.set_state(V.to(torch.complex128 if precision == "fp64" else torch.complex64), lam)
    W, mu, _ = L.get_state()
    W = W.to(torch.complex128)
    tol = 1e-12 if precision == "fp64" else 2e-6
    assert float((W.mH @ W - torch.eye(r, device="cuda")).abs().max()) < tol
    rho = lambda X, w: (X * torch.as_tensor(w, device="cuda")) @ X.mH  # noqa: E731
    ref = rho(V, lam)
    assert float((rho(W, mu) - ref).norm() / ref.norm()) < tol
