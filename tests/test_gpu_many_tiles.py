"""The tiled passes above the sizes that are summed entry by entry (4096 rows), with several tiles per CTA: every block count and
width, exponents that change while a CTA's sums run, ring buffers that wrap, flushes and drains in the middle.

Complex128 Grams: 1e-14 of the columns' norms, by the same reasoning as at small sizes (an entry is cut 2^-52 or so below the
largest of its column in the tile; random signs); the reference sums products of 64 rows in long double.  Complex64 Grams:
at most 256 rows (512 products) in plain FP32 per lane and 2^16 / 256 or more independent lanes, 3.4e-8 sqrt(2 / (3 2^16)) 256 =
2.8e-8 r.m.s. of a diagonal entry at worst, so 1e-7 for any.  Steps in complex64 against complex128: 5e-6 of the norm, as at small sizes.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402


def _context(n, r, precision):
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", precision, r)
    V = torch.zeros((1 << n, r), dtype=L.torch_dtype, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    return L


def _block(n, r, g, kind, dtype=torch.complex128):
    N = 1 << n
    X = torch.randn((N, r), dtype=dtype, device="cuda", generator=g)
    if kind == "columns":      # both ends of the exponents take the direct path
        X = X * 10.0 ** torch.linspace(-150, 100, r, device="cuda", dtype=torch.float64)
    if kind == "rows":         # a column's exponent changes from tile to tile
        X = X * torch.logspace(0, -12, N, dtype=torch.float64, device="cuda")[:, None]
    if kind == "jump":         # a column's exponent changes on tiles that another column sends down the direct path
        X[N // 4:, 0] *= 2.0 ** 20
        X[N // 4: N // 2, r - 1] *= 1e-160
    if kind == "zeros":
        X[: N // 2] = 0
        X[:, 0] = 0
    return X.contiguous()


def _reference(blocks):
    X = torch.cat(blocks, dim=1)
    r = blocks[-1].shape[1]
    C = X.reshape(-1, 64, X.shape[1])
    return (C.mH @ C[:, :, -r:]).cpu().numpy().astype(np.clongdouble).sum(0), X


@pytest.mark.parametrize("n,r,m", [(13, 5, 3), (13, 17, 4), (13, 32, 5), (14, 7, 13), (16, 1, 1), (16, 3, 2), (16, 8, 3), (16, 16, 5), (16, 24, 2)])
@pytest.mark.parametrize("kind", ["plain", "columns", "rows", "jump", "zeros"])
def test_gram_complex128(n, r, m, kind):
    L = _context(n, r, "fp64")
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 1000 + r * 10 + m)
    blocks = [_block(n, r, g, kind) for _ in range(m)]
    ref, X = _reference(blocks)
    norm = X.abs().square().cpu().numpy().astype(np.longdouble).sum(0) ** 0.5
    scale = np.maximum(norm[:, None] * norm[None, -r:], np.longdouble(1e-300))
    assert float((np.abs(L.gram(blocks).cpu().numpy() - ref) / scale).max()) < 1e-14


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("n", [13, 16])
def test_gram_complex128_with_a_non_finite_entry(n, bad):
    # the entry spoils its column's and its row's products and no other
    r = 6
    L = _context(n, r, "fp64")
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A, B = _block(n, r, g, "plain"), _block(n, r, g, "plain")
    ref, X = _reference([A, B])
    A[4137, 2] = bad
    P = L.gram([A, B])
    good = np.arange(2 * r) != 2
    assert not torch.isfinite(torch.view_as_real(P[2])).any()
    assert float(np.abs(P.cpu().numpy() - ref)[good].max()) < 1e-14 * (1 << n) * 4


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("r", [8, 16, 32])
def test_gram_complex64(r, m):
    n = 16
    L = _context(n, r, "mixed")
    g = torch.Generator(device="cuda")
    g.manual_seed(r * 10 + m)
    blocks = [_block(n, r, g, "plain", torch.complex64) for _ in range(m)]
    ref, X = _reference([b.to(torch.complex128) for b in blocks])
    norm = X.norm(dim=0).cpu().numpy()
    assert (np.abs(L.gram(blocks).cpu().numpy() - ref) / (norm[:, None] * norm[None, -r:])).max() < 1e-7


@pytest.mark.parametrize("scheme,r", [("rk4", 8), ("ab4", 8), ("rk2", 16), ("rk4", 16), ("ab3", 16), ("rk4", 32), ("rk4", 11), ("rk4", 27)])
def test_step_complex64_matches_complex128(scheme, r):
    w = li.workload(2, n=15, r=r)
    states = []
    for precision, dtype in (("fp64", torch.complex128), ("mixed", torch.complex64)):
        L = Lrei(w.n, w.bonds, w.B, w.kappa, "qllg", precision, r)
        L.set_state(torch.from_numpy(w.V).to("cuda", dtype), w.lam)
        L.step(0.005, scheme, 5)
        V, lam, _ = L.get_state()
        V = V.to(torch.complex128)
        X = torch.randn((1 << w.n, 4), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        states.append((V * torch.as_tensor(lam, device="cuda")) @ (V.mH @ X))   # rho X
    assert float((states[1] - states[0]).norm() / states[0].norm()) < 5e-6
