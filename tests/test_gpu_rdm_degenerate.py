"""Two-spin density matrices that are a multiple of the identity up to rounding.

Their off-diagonal entries are rounding noise (1e-17), which a Jacobi sweep only replaces by other noise: the 4 x 4 solves have to
stop at once, as they do for a matrix that is diagonal.  Both runs have the same 4096 pairs and sizes, so the time of the call may
differ by its few sweeps only; twice the time is allowed, the sweep limit would take several times as long.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402

PAIRS = [(0, 1)] * 4096


def _context(n, U):
    """rho = U I U^* / 4 on the first two spins, all others up."""
    V = torch.zeros((1 << n, 4), dtype=torch.complex128)
    V[:: 1 << (n - 2)] = U
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "fp64", 4)
    L.set_state(V.cuda(), np.full(4, 0.25))
    return L


def _time(L):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(6):
        torch.cuda.synchronize()
        a.record()
        out = L.two_spin_rdm(PAIRS)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best, out


def test_maximally_mixed_pair():
    n = 8
    g = torch.Generator()
    g.manual_seed(5)
    U = torch.linalg.qr(torch.randn((4, 4), dtype=torch.complex128, generator=g))[0]
    exact, _ = _time(_context(n, torch.eye(4, dtype=torch.complex128)))
    noisy, (R, concurrence, negativity) = _time(_context(n, U))
    assert np.abs(R - np.eye(4) / 4).max() < 1e-15
    assert concurrence.max() == 0.0 and negativity.max() < 1e-15
    assert noisy < 2.0 * exact
