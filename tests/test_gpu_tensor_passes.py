"""The complex128 tile passes on the tensor cores (digit planes) against numpy's long double.

Gram entries are judged against the product of their columns' norms.  A column is cut to 55 bits below
2^e, e at most 4 above the exponent of its largest entry in the tile, so each factor of a product is off by
at most 2^-52 of that entry; with random signs the sum of N products is off by less than
4 * 2^-52 of the norms' product, the digit products left out by less than 2^-52, and the sums of the CTAs'
partials by sqrt(N) 2^-53: 1e-14 covers N <= 2^12 with room.  (The reference is long double: torch's own FP64
Gram of 2^12 rows whose entries fall by 1e-12 is off by 1.6e-14.)  The projection's check is the
orthonormality of a set state (its Gram is measured by the same pass) and the state itself.
"""
import numpy as np
import pytest

import lrei_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import Lrei  # noqa: E402

TOL = 1e-14


def _context(n, r):
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "fp64", r)
    V = torch.zeros((1 << n, r), dtype=torch.complex128, device="cuda")
    V[torch.arange(r), torch.arange(r)] = 1.0
    L.set_state(V, np.full(r, 1.0 / r))
    return L


def _block(n, r, g, kind):
    N = 1 << n
    X = torch.randn((N, r), dtype=torch.complex128, device="cuda", generator=g)
    if kind == "columns":      # columns 1e-150 .. 1e100 apart (both ends of the exponents take the direct path)
        X = X * 10.0 ** torch.linspace(-150, 100, r, device="cuda", dtype=torch.float64)
    if kind == "rows":         # a column's exponent changes from tile to tile
        X = X * torch.logspace(0, -12, N, dtype=torch.float64, device="cuda")[:, None]
    if kind == "spikes":       # a few large entries over a small background
        X = X * 1e-3
        X[torch.randint(0, N, (5,), device="cuda", generator=g)] *= 1e6
    if kind == "zeros":        # a zero column, half of the rows zero
        X[: N // 2] = 0
        X[:, 0] = 0
    return X.contiguous()


def _gram_error(L, blocks):
    P = L.gram(blocks).cpu().numpy()
    left = np.concatenate([b.cpu().numpy() for b in blocks], axis=1).astype(np.clongdouble)
    last = left[:, -blocks[-1].shape[1]:]
    ref = left.conj().T @ last
    norm = lambda X: np.sqrt((X.real ** 2 + X.imag ** 2).sum(0))  # noqa: E731
    scale = np.maximum(norm(left)[:, None] * norm(last)[None, :], np.longdouble(1e-300))
    return float((np.abs(P - ref) / scale).max())


@pytest.mark.parametrize("n,r,m", [(7, 5, 3), (8, 1, 1), (8, 3, 2), (8, 8, 1), (8, 9, 2), (8, 16, 5), (9, 17, 4),
                                   (9, 32, 5), (10, 7, 13), (12, 16, 8)])
@pytest.mark.parametrize("kind", ["plain", "columns", "rows", "spikes", "zeros"])
def test_gram(n, r, m, kind):
    L = _context(n, r)
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 1000 + r * 10 + m)
    blocks = [_block(n, r, g, kind) for _ in range(m)]
    assert _gram_error(L, blocks) < TOL


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_gram_with_a_non_finite_entry(bad):
    # the entry spoils its column's and its row's products and no other
    n, r = 8, 6
    L = _context(n, r)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A, B = _block(n, r, g, "plain"), _block(n, r, g, "plain")
    ref = torch.cat([A.mH @ B, B.mH @ B])
    A[37, 2] = bad
    P = L.gram([A, B])
    good = torch.ones(2 * r, dtype=torch.bool, device="cuda")
    good[2] = False
    assert not torch.isfinite(torch.view_as_real(P[2])).any()
    assert float((P[good] - ref[good]).abs().max()) < TOL * (1 << n) * 4


@pytest.mark.parametrize("n,r", [(7, 5), (8, 2), (9, 8), (10, 16), (10, 17), (11, 32)])
def test_projection_of_a_badly_scaled_factor(n, r):
    # columns 1e6 apart: the state that is set is orthonormal to rounding and spans the same density matrix
    g = torch.Generator(device="cuda")
    g.manual_seed(n + r)
    V = torch.randn((1 << n, r), dtype=torch.complex128, device="cuda", generator=g)
    V = torch.linalg.qr(V.cpu())[0].cuda() * 10.0 ** torch.linspace(-3, 3, r, device="cuda", dtype=torch.float64)
    lam = np.full(r, 1.0 / r)
    L = Lrei(n, li.chain_bonds(n, False), (0.0, 0.0, 0.5), 0.1, "qll", "fp64", r)
    L.set_state(V, lam)
    W, mu, _ = L.get_state()
    assert float((W.mH @ W - torch.eye(r, device="cuda")).abs().max()) < 1e-12
    rho = lambda X, w: (X * torch.as_tensor(w, device="cuda")) @ X.mH  # noqa: E731
    ref = rho(V, lam)
    assert float((rho(W, mu) - ref).norm() / ref.norm()) < 1e-13


@pytest.mark.parametrize("n,r,scheme", [(8, 3, "rk4"), (8, 16, "rk4"), (8, 20, "rk4"), (9, 32, "rk4"), (8, 20, "ab4")])
def test_step_keeps_the_invariants(n, r, scheme):
    # every pass width of the step (projections split by columns among them)
    w = li.workload(2, n=n, r=r)
    L = Lrei(w.n, w.bonds, w.B, w.kappa, "qllg", "fp64", r)
    L.set_state(torch.from_numpy(w.V).cuda(), w.lam)
    L.step(0.005, scheme, 6)
    o = L.observables()
    assert abs(o["trace"] - 1.0) < 1e-12 and o["orth_err"] < 1e-12
    assert abs(o["purity"] - np.sum(w.lam ** 2)) < 1e-12
