"""How far complex64 Grams are off: the rounding of the plain FP32 sums, and nothing beside it.

A lane sums L rows in plain FP32, everything after is compensated (or FP64).  A diagonal entry adds two products per row; an
addition is off by at most a uniform half unit, 2^-23 / sqrt(12) = 3.4e-8 of its partial sum (r.m.s.), so a lane's sum by
3.4e-8 sqrt(2 L / 3) of itself and the N / L independent ones together by 3.4e-8 L sqrt(2 / (3 N)) of the entry.  1.5 times
that is allowed for the r.m.s. of the 20 or more diagonal entries taken, 6 times that for any entry (off the diagonal the
partial sums are smaller).  N = 2^18: many tiles per CTA.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


def _rows(r, m):
    """Rows of a lane's plain sum."""
    if r in (8, 16, 32):
        return {8: 32, 16: 128, 32: 256 if m <= 5 else 32}[r]
    return 16 if r < 8 or (r < 16 and m <= 3) else (24 if r < 16 else (128 if m <= 5 else 32))


@pytest.mark.parametrize("m", [1, 2, 5, 8])
@pytest.mark.parametrize("r", [2, 5, 7, 8, 9, 12, 15, 16, 24, 29, 32])
def test_gram(r, m):
    if r in (24, 29) and m < 4:
        m = 4
    n = 18
    N = 1 << n
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "mixed", r)
    V = torch.zeros((N, r), dtype=torch.complex64, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    g = torch.Generator(device="cuda")
    g.manual_seed(100 * r + m)
    diag = []
    bound = 1.5 * 2.0 ** -23 / np.sqrt(12) * _rows(r, m) * np.sqrt(2 / (3 * N))
    for _ in range(-(-20 // r)):
        blocks = [torch.randn((N, r), dtype=torch.complex64, device="cuda", generator=g) for _ in range(m)]
        P = L.gram(blocks)
        X = torch.cat(blocks, dim=1).to(torch.complex128)
        norm = X.norm(dim=0)
        err = (P - X.mH @ X[:, -r:]).abs() / (norm[:, None] * norm[None, -r:])
        assert float(err.max()) < 6 * bound
        diag.append(err[-r:].diagonal())
    assert float(torch.cat(diag).square().mean().sqrt()) < bound
