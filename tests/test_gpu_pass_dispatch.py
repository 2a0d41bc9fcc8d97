"""Passes on both sides of the lines between the kernels: rows summed entry by entry or tiled (4096 rows, and 2^20 multiply-adds of a
Gram), projections of ranks 1 and 2 in complex128 below and from 2^16 rows on, and blocks whose rows are no whole
groups of four columns (loaded by elements).

Steps against the same step from a factor with its columns turned by phases, which every path must carry through: the density
matrix agrees to 1e-12 in complex128 and to 5e-6 of its norm in complex64, as in the other step tests.  Right-hand sides against
plain torch in complex128: 1e-12 and 5e-6 of the norm.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402

TOL = {"fp64": 1e-12, "mixed": 5e-6}


def _context(n, r, precision):
    w = li.workload(2, n=n, r=r)
    L = Lrei(w.n, w.bonds, w.B, w.kappa, "qll", precision, r)
    return w, L


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,r", [(6, 8), (7, 8), (8, 5), (8, 16), (9, 5), (9, 16), (10, 17), (12, 3), (12, 16), (13, 16), (14, 2), (16, 1), (16, 2),
                                 (14, 23), (14, 31)])
def test_step_does_not_see_the_columns_phases(n, r, precision):
    w, L = _context(n, r, precision)
    V = torch.from_numpy(w.V).cuda()
    phase = torch.polar(torch.ones(r, dtype=torch.float64), torch.linspace(0.3, 2.9, r, dtype=torch.float64)).cuda()
    X = torch.randn((1 << n, 4), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out = []
    for U in (V, V * phase):
        L.set_state(U.to(L.torch_dtype), w.lam)
        L.step(0.01, "rk4", 2)
        W, lam, _ = L.get_state()
        W = W.to(torch.complex128)
        out.append((W * torch.as_tensor(lam, device="cuda")) @ (W.mH @ X))
    assert float((out[0] - out[1]).norm() / out[0].norm()) < TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,r", [(6, 8), (8, 5), (8, 8), (9, 5), (12, 16), (13, 3), (16, 2), (14, 23)])
def test_rhs(n, r, precision):
    w, L = _context(n, r, precision)
    L.set_state(torch.from_numpy(w.V).cuda().to(L.torch_dtype), w.lam)
    V, lam, _ = L.get_state()
    Y = torch.empty_like(V)
    L.apply_h(V, Y)
    Z, W, G = L.rhs(0)
    V, Y, Z, W = (x.to(torch.complex128) for x in (V, Y, Z, W))
    lam = torch.as_tensor(lam, device="cuda")
    Gr = V.mH @ Y
    Gr = (Gr + Gr.mH) / 2
    d = lam[:, None] - lam[None, :]
    X11 = (1j * d - w.kappa * d * d) * Gr
    Wr = (Y - V @ Gr) * ((1j - w.kappa * lam) * lam).conj()
    for a, b in ((W, Wr), (Z, V @ X11 + Wr)):
        assert float((a - b).norm() / b.norm()) < TOL[precision]
