"""FP64 Jacobi sweeps of set_state: none where the small matrix is diagonal to rounding already.

An orthonormal factor with equal weights gives L^H Lambda L = I / r up to the rounding of its Gram, a few 2^-53 / r with random
signs in each entry off the diagonal: sqrt(r (r - 1)) entries of 1e-16 against the diagonal's sqrt(r) are 5.6e-16 of the
Frobenius norm at r = 32, and the solver stops at 1e-15 of it.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei, eig_counters  # noqa: E402


@pytest.mark.parametrize("r", [1, 2, 8, 16, 31, 32])
@pytest.mark.parametrize("n", [8, 13])
def test_equal_weights_need_no_sweep(n, r):
    g = torch.Generator()
    g.manual_seed(10 * n + r)
    V = torch.linalg.qr(torch.randn((1 << n, r), dtype=torch.complex128, generator=g))[0].cuda()
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "fp64", r)
    before = eig_counters()
    L.set_state(V, np.full(r, 1.0 / r))
    after = eig_counters()
    assert after["fp64_calls"] == before["fp64_calls"] + 1
    assert after["fp64_sweeps"] == before["fp64_sweeps"]
    W, lam, _ = L.get_state()
    # not rotated inside the degenerate space: each column is one of those given, in some order
    overlap = (V.mH @ W).abs()
    assert float((overlap.amax(0) - 1).abs().max()) < 1e-13
    assert np.abs(lam - 1.0 / r).max() < 1e-15
