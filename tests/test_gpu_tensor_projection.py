"""The projection of the complex128 tile passes on the tensor cores (digit planes), driven by itself: new = sum_m q_m C_m + s C_s
for chosen blocks and coefficients, row by row against torch's FP64 products or exact integers.

Bound of a row: an entry is cut to half of 2^(e - 55), e at most 3 above the exponent of its column's largest entry in the tile,
so it is off by 2^-53 of that entry at most, and so are the coefficients (each scaled by its row's exponent) of the largest in
their column; digit products left out stay below 2^-52 of the two, and 2^3 of slack on either side gives for a sum over K columns
K 2^-47 max_k max_tile |x_k| |c_kj|.  Groups of 32 rows aligned to 32 hold whole tiles (of 32 or 16 rows).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2508_21200_gb300 import build as lib_build  # noqa: E402

SOURCE = r"""
#include "tsk.cuh"
extern "C" int project(long long N, int r, int nq, const void *const *q, const void *src, const void *coefQ,
                       const void *coefS, void *out, void *partial, int *status, int nsm) {
  if (lrei::ts_init()) return -1;
  lrei::TSArgs a{};
  a.N = N;
  a.r = r;
  a.nq = nq;
  for (int m = 0; m < nq; ++m) a.q[m] = q[m];
  a.src = src;
  a.mode = src ? 1 : 2;
  a.coefQ = static_cast<const lrei::zd *>(coefQ);
  a.coefS = static_cast<const lrei::zd *>(coefS);
  a.out = out;
  a.partial = static_cast<double *>(partial);
  a.status = status;
  return lrei::launch_tsx(a, nsm, 0);
}
"""


@pytest.fixture(scope="module")
def project(tmp_path_factory):
    lib = lib_build.ensure_built()
    d = tmp_path_factory.mktemp("project")
    (d / "project.cu").write_text(SOURCE)
    subprocess.run([lib_build._nvcc(), *lib_build.ARCH, *lib_build.FLAGS, "-shared", str(d / "project.cu"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib), "-o", str(d / "project.so")], check=True)
    f = ctypes.CDLL(str(d / "project.so")).project
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 7 + [ctypes.c_int]
    nsm = torch.cuda.get_device_properties(0).multi_processor_count

    def run(q, src, C, in_place=False):
        """[q_0 .., src] C (C: (blocks r) x r), into q_0 with in_place."""
        N, r = q[0].shape
        nq = len(q)
        Cq = C[: nq * r].T.contiguous()                     # column-major
        Cs = C[nq * r:].T.contiguous() if src is not None else None
        out = q[0] if in_place else torch.empty_like(q[0])
        partial = torch.empty((2 * nsm + 16) * 13 * r * r * 2, dtype=torch.float64, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        ptrs = (ctypes.c_void_p * nq)(*[x.data_ptr() for x in q])
        torch.cuda.synchronize()
        n = f(N, r, nq, ctypes.cast(ptrs, ctypes.c_void_p), src.data_ptr() if src is not None else None, Cq.data_ptr(),
              Cs.data_ptr() if Cs is not None else None, out.data_ptr(), partial.data_ptr(), status.data_ptr(), nsm)
        torch.cuda.synchronize()
        assert n > 0 and int(status) == 0
        return out
    return run


def _phases(shape, g):
    """Entries of modulus one, so that every tile's largest component is at least 2^-1/2: one exponent for all tiles."""
    return torch.polar(torch.ones(shape, dtype=torch.float64, device="cuda"),
                       2 * np.pi * torch.rand(shape, dtype=torch.float64, device="cuda", generator=g))


def _check(X, C, out):
    ref = X @ C
    N, K = X.shape
    big = X.abs().reshape(N // 32, 32, K).amax(1)                              # per tile and column
    M = (big[:, :, None] * C.abs()[None]).amax(1).repeat_interleave(32, 0)     # per tile and output
    err = (out - ref).abs() - K * 2.0 ** -47 * M
    assert float(err.max()) <= 0.0


def _input(kind, N, r, m, g):
    X = torch.cat([_phases((N, r), g) for _ in range(m)], dim=1)
    a, b = 0, m * r - 1                       # two columns
    quarter, late = slice(N // 4, N // 2), slice(N // 4, N)
    if kind == "jump":       # column a grows 2^20 while b is below the exponents that are cut, in every CTA's next tile
        X[late, a] *= 2.0 ** 20
        X[quarter, b] *= 1e-160
    if kind == "appears":    # column a is zero until then
        X[: N // 4, a] = 0
        X[quarter, b] *= 1e-160
    if kind == "falls":
        X[late, a] *= 2.0 ** -20
        X[quarter, b] *= 1e160
    if kind == "rows":       # exponents change from tile to tile
        X = X * torch.logspace(0, -12, N, dtype=torch.float64, device="cuda")[:, None]
    if kind == "spikes":
        X[torch.randint(0, N, (9,), device="cuda", generator=g)] *= 1e9
    if kind == "zeros":
        X[: N // 2] = 0
        X[:, a] = 0
    return X


# several tiles per CTA: one CTA takes a tile of 32 or 16 rows in turn with at most 3 x 152 others
@pytest.mark.parametrize("r,nq,extend", [(3, 1, False), (8, 2, True), (5, 4, True), (16, 4, True), (17, 3, False), (32, 4, True),
                                         (17, 6, True)])
@pytest.mark.parametrize("kind", ["plain", "jump", "appears", "falls", "rows", "spikes", "zeros"])
def test_rows(project, r, nq, extend, kind):
    N, m = 1 << 16, nq + (1 if extend else 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(r * 10 + nq)
    X = _input(kind, N, r, m, g)
    C = torch.randn((m * r, r), dtype=torch.complex128, device="cuda", generator=g)
    blocks = [X[:, i * r:(i + 1) * r].contiguous() for i in range(m)]
    out = project(blocks[:nq], blocks[nq] if extend else None, C)
    _check(X, C, out)


@pytest.mark.parametrize("r,nq", [(4, 1), (16, 5), (24, 2)])
def test_in_place(project, r, nq):
    N = 1 << 14
    g = torch.Generator(device="cuda")
    g.manual_seed(r)
    X = _input("rows", N, r, nq, g)
    C = torch.randn((nq * r, r), dtype=torch.complex128, device="cuda", generator=g)
    blocks = [X[:, i * r:(i + 1) * r].clone() for i in range(nq)]
    _check(X, C, project(blocks, None, C, in_place=True))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite(project, bad):
    # an entry spoils its row, a coefficient its column, and nothing else
    N, r = 1 << 15, 6
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    X = _phases((N, 2 * r), g)
    C = torch.randn((2 * r, r), dtype=torch.complex128, device="cuda", generator=g)
    ref = X @ C
    Xb = X.clone()
    Xb[20001, 3] = bad
    out = project([Xb[:, :r].contiguous()], Xb[:, r:].contiguous(), C)
    assert not torch.isfinite(torch.view_as_real(out[20001])).any()
    good = torch.arange(N, device="cuda") != 20001
    assert float((out - ref)[good].abs().max()) < 2 * r * 2.0 ** -47 * float(C.abs().max())
    Cb = C.clone()
    Cb[2, 4] = bad
    out = project([X[:, :r].contiguous()], X[:, r:].contiguous(), Cb)
    assert not torch.isfinite(torch.view_as_real(out[:, 4])).any()
    cols = torch.arange(r, device="cuda") != 4
    assert float((out - ref)[:, cols].abs().max()) < 2 * r * 2.0 ** -47 * float(C.abs().max())


def _digits(shape, rng):
    """Integers sum_s d_s 2^(8 (6 - s)), 119 <= d_s <= 127 (the last a multiple of 4, so that 53 bits hold them): every digit
    near the largest."""
    d = rng.integers(119, 128, (7, *shape))
    d[6] = 124
    return sum(d[s].astype(object) << (8 * (6 - s)) for s in range(7))


@pytest.mark.parametrize("r,nq", [(16, 3), (32, 4), (17, 6)])
def test_sums_of_the_largest_digits(project, r, nq):
    # All products of one sign and near 2^14, K = 64, 160 and 119 complex columns of them.  Exact: the inputs and the first four
    # classes of digit products.  The fifth passes 2^24 in the last fifth of 128 columns: at most 16 instructions that may cut
    # 2 units of 2^-46 each, 5e-13 of products near one; the sum has at least 100 of these, so 4e-15 of it leaves room for the
    # digit products left out (2^-52) and the rounding of the result.
    N, K = 8192, (nq + 1) * r
    rng = np.random.default_rng(r)
    rows = rng.integers(0, 64, N)                         # 64 different rows
    xr, xi, cr, ci = (_digits(s, rng) for s in ((64, K), (64, K), (K, r), (K, r)))
    x = (xr.astype(np.float64) + 1j * xi.astype(np.float64))[rows]
    x[: N // 2] /= 2                                      # the exponents stay one above these rows' and are those of the others
    c = cr.astype(np.float64) - 1j * ci.astype(np.float64)
    X, C = torch.from_numpy(x).cuda(), torch.from_numpy(c).cuda()
    blocks = [X[:, i * r:(i + 1) * r].contiguous() for i in range(nq + 1)]
    out = project(blocks[:nq], blocks[nq], C).cpu().numpy()[N // 2:]
    re = xr.dot(cr) + xi.dot(ci)                          # exact integers
    got = out.real
    err = max(abs(int(got[k, j]) - re[rows[N // 2 + k], j]) / re[rows[N // 2 + k], j] for k in range(0, N // 2, 7)
              for j in range(r))
    assert err < 4e-15


@pytest.mark.parametrize("r,nq,extend", [(1, 1, False), (3, 1, False), (8, 2, True), (16, 4, True), (17, 3, False), (32, 4, True)])
@pytest.mark.parametrize("columns", ["alike", "apart"])
def test_rows_of_very_different_size(project, r, nq, extend, columns):
    # Neighbouring rows 2^-90 .. 2^90 apart, and with "apart" the columns of the blocks too, undone by the rows of C: each row is as
    # good as its own entries allow.  An entry x_rk is off by half of 2^-55 of the next power of two above the largest |x_rk| a_k, a_k
    # the next above max_j |c_kj|, and so are the coefficients, of one: K 2^-53 x 4 together with the products left out (K 2^-52),
    # below K 2^-49 max_k |x_rk| max_j |c_kj|, in which 2^3 covers the modulus of complex entries and torch's own sum.
    N, m = 1 << 15, nq + (1 if extend else 0)
    K = m * r
    g = torch.Generator(device="cuda")
    g.manual_seed(r * 10 + nq)
    uniform = lambda n, bits: (2.0 ** (bits * (2 * torch.rand(n, dtype=torch.float64, device="cuda", generator=g) - 1)))  # noqa: E731
    X = torch.randn((N, K), dtype=torch.complex128, device="cuda", generator=g) * uniform(N, 90)[:, None]
    X[17::64] = 0
    C = torch.randn((K, r), dtype=torch.complex128, device="cuda", generator=g)
    if columns == "apart":
        s = uniform(K, 60)
        X, C = X * s, C / s[:, None]
    blocks = [X[:, i * r:(i + 1) * r].contiguous() for i in range(m)]
    out = project(blocks[:nq], blocks[nq] if extend else None, C)
    M = (X.abs() * C.abs().amax(1)).amax(1, keepdim=True)
    assert float(((out - X @ C).abs() - K * 2.0 ** -49 * M).max()) <= 0.0
    assert float(out[17::64].abs().max()) == 0.0
