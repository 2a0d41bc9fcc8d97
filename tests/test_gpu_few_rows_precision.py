"""Complex64 passes of few rows are as good as FP64 arithmetic on their complex64 inputs.

Gram entries: products and sums keep their rounding errors (pairs of FP32, about 2^-46 of the sum of moduli; 2^-44 of the norms is
asserted, which FP32 sums miss by 2^15).  Right-hand side: Z and W are rounded to complex64 once per pass, so against the same products in
complex128 from the same factor an entry is off by a few half units of the largest partial result, 4 x 2^-24 of the largest entry; FP32
coefficients and sums of r terms would be off by several times that.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


@pytest.mark.parametrize("n,r,m", [(3, 2, 1), (6, 8, 3), (9, 5, 4), (9, 16, 2), (10, 11, 5), (10, 32, 1), (12, 3, 6), (12, 16, 1), (12, 7, 5)])
def test_gram(n, r, m):
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "mixed", r)
    V = torch.zeros((1 << n, r), dtype=torch.complex64, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    g = torch.Generator(device="cuda")
    g.manual_seed(100 * n + r)
    blocks = [torch.randn((1 << n, r), dtype=torch.complex64, device="cuda", generator=g) for _ in range(m)]
    X = torch.cat(blocks, dim=1).to(torch.complex128)
    norm = X.norm(dim=0)
    err = (L.gram(blocks) - X.mH @ X[:, -r:]).abs() / (norm[:, None] * norm[None, -r:])
    assert float(err.max()) < 2.0 ** -44


@pytest.mark.parametrize("n,r", [(6, 8), (8, 5), (9, 16), (10, 11), (12, 3), (12, 16)])
def test_rhs(n, r):
    w = li.workload(2, n=n, r=r)
    L = Lrei(w.n, w.bonds, w.B, w.kappa, "qll", "mixed", r)
    L.set_state(torch.from_numpy(w.V).cuda().to(torch.complex64), w.lam)
    V, lam, _ = L.get_state()
    Y = torch.empty_like(V)
    L.apply_h(V, Y)
    Z, W, G = L.rhs(0)
    V, Y, Z, W = (x.to(torch.complex128) for x in (V, Y, Z, W))
    lam = torch.as_tensor(lam, device="cuda")
    Gr = V.mH @ Y
    c = ((1j - w.kappa * lam) * lam).conj()
    Wr = Y * c - V @ (Gr * c)
    d = lam[:, None] - lam[None, :]
    Gh = (Gr + Gr.mH) / 2
    Zr = V @ ((1j * d - w.kappa * d * d) * Gh) + W
    for a, b in ((W, Wr), (Z, Zr)):
        big = max(float((Y * c).abs().max()), float(b.abs().max()))
        assert float((a - b).abs().max()) < 4 * 2.0 ** -24 * big
