"""Complex64 blocks that start on an element but not on 16 bytes (a view into a larger buffer): same results as aligned ones.

The kernels that load 16 bytes at a time are left out for them, so sums are grouped otherwise: 2e-6 of the largest entry (H V,
right-hand side: a few tens of FP32 roundings) or of the columns' norms (Gram).
"""
import ctypes

import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


def _shifted(X):
    buf = torch.zeros(X.numel() + 1, dtype=X.dtype, device="cuda")
    Y = buf[1:].view(X.shape)
    Y.copy_(X)
    assert Y.data_ptr() % 16 == 8
    return Y


@pytest.mark.parametrize("n", [9, 13])
@pytest.mark.parametrize("r", [1, 2, 4, 6, 8, 16, 24, 32])
def test_shifted_blocks(n, r):
    w = li.workload(2, n=n, r=r)
    L = Lrei(w.n, w.bonds, w.B, w.kappa, "qll", "mixed", r)
    L.set_state(torch.from_numpy(w.V).to("cuda", torch.complex64), w.lam)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + r)
    blocks = [torch.randn((1 << n, r), dtype=torch.complex64, device="cuda", generator=g) for _ in range(3)]
    close = lambda a, b: float((a - b).abs().max() / b.abs().max()) < 2e-6  # noqa: E731
    Y = torch.empty_like(blocks[0])
    L.apply_h(blocks[0], Y)
    for X in (blocks[0], _shifted(blocks[0])):
        out = _shifted(torch.zeros_like(Y))
        L.apply_h(X, out)
        assert close(out, Y)
    norm = torch.cat(blocks, dim=1).norm(dim=0)
    ref = L.gram(blocks)
    for which in range(3):
        mixed = [_shifted(b) if i == which else b for i, b in enumerate(blocks)]
        err = (L.gram(mixed) - ref).abs() / (norm[:, None] * norm[None, -r:])
        assert float(err.max()) < 2e-6
    Z, W, G = L.rhs(0)
    Zs, Ws = _shifted(torch.zeros_like(Z)), _shifted(torch.zeros_like(W))
    Gs = np.zeros(2 * r * r)
    code = L._lib.lrei_rhs(L._h, ctypes.c_void_p(Zs.data_ptr()), ctypes.c_void_p(Ws.data_ptr()),
                           Gs.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 0)
    assert code == 0
    assert close(Zs, Z) and close(Ws, W)
