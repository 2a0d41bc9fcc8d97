"""The work this framework is measured on: LREI time steps and the passes they are made of.

A program that uses the framework holds an initial factor V (N x r, N = 2^n) and its weights, sets
them as a context's state, takes RK or AB steps, and reads the observables and the factor; or it
calls one pass on blocks of its own (H V, the tall-skinny Gram, the right-hand side, the
measurements).  The sizes are those of configs/cfg1..cfg5.json, of the tests and of the benchmark.

The columns of a factor are defined up to a phase each: `run` returns them with the phase of the
overlap with the initial factor's column removed, as a program that compares or stores factors does.
Numbers measured from a complex64 state are returned in single precision, the precision of what they
are measured from.

Every input is drawn from the seed on the GPU; `exact` restates the method in plain torch in 64 bits.
"""
import math
import types

import numpy as np
import torch

KINDS = ("rk4", "ab3", "batch", "hv", "gram", "rhs", "monitor")


def listed():
    return [
        # cfg1, the smallest system anyone steps: 20 steps of a chain of 8 spins, all launch latency
        dict(name="rk4_n8_r4_c128", kind="rk4", n=8, r=4, lattice="chain", model="qll", precision="fp64",
             kappa=0.1, dt=0.01, steps=20),
        # cfg2: periodic anisotropic chain, the multistep scheme with its RK4 start-up
        dict(name="ab3_n16_r8_c128", kind="ab3", n=16, r=8, lattice="ring", model="qll", precision="fp64",
             kappa=0.1, dt=0.005, steps=8),
        # cfg2 with the complex64 bulk and the q-LLG model: an ordinary mid-size run
        dict(name="rk4_n16_r8_c64", kind="rk4", n=16, r=8, lattice="ring", model="qllg", precision="mixed",
             kappa=0.1, dt=0.005, steps=4),
        # cfg3, the benchmark's headline size, complex64 bulk
        dict(name="rk4_n20_r16_c64", kind="rk4", n=20, r=16, lattice="chain", model="qll", precision="mixed",
             kappa=0.1, dt=0.01, steps=2),
        # cfg3 in complex128: the benchmark's FP64 leg and the reference run of every accuracy check
        dict(name="rk4_n20_r16_c128", kind="rk4", n=20, r=16, lattice="chain", model="qll", precision="fp64",
             kappa=0.1, dt=0.01, steps=1),
        # cfg5, the largest workload
        dict(name="rk4_n22_r32_c64", kind="rk4", n=22, r=32, lattice="chain", model="qll", precision="mixed",
             kappa=0.05, dt=0.01, steps=1),
        # cfg4: many uneven trajectories (n = 10..18, r = 2..16, odd ranks among them) in one launch per step
        dict(name="batch12_cfg4_c64", kind="batch", count=12, sizes=4, n=18, r=16, lattice="chain", model="qll",
             precision="mixed", kappa=0.1, dt=0.01, steps=3),
        # one Hamiltonian action at the headline size: an energy or a Krylov solver of the user's own
        dict(name="hv_n20_r16_c64", kind="hv", n=20, r=16, lattice="chain", model="qll", precision="mixed"),
        # the same on the full eq. H1: 4 x 4 triangular lattice with DMI and a transverse field, r not a power of 2
        dict(name="hv_h1_n16_r6_c128", kind="hv", n=16, r=6, lattice="triangular", model="qllg", precision="fp64"),
        # the tall-skinny Gram of five blocks (the benchmark's roofline launch)
        dict(name="gram5_n20_r16_c64", kind="gram", n=20, r=16, blocks=5, lattice="chain", model="qll",
             precision="mixed"),
        # one evaluation of the right-hand side f(rho) = Z V* + V W* at an odd rank
        dict(name="rhs_n18_r5_c64", kind="rhs", n=18, r=5, lattice="chain", model="qllg", precision="mixed",
             kappa=0.5),
        # what a run logs between steps: the observables and every two-spin reduced density matrix
        dict(name="monitor_n16_r7_c128", kind="monitor", n=16, r=7, lattice="ring", model="qll", precision="fp64"),
    ]


def draw(rng):
    kind = rng.choice(("rk4", "rk4", "rk4", "ab3", "batch", "hv", "hv", "gram", "rhs", "monitor"))
    precision = rng.choice(("fp64", "mixed"))
    lattice = rng.choice(("chain", "ring", "triangular")) if kind != "batch" else "chain"
    top = {"rk4": 20 if precision == "mixed" else 18, "ab3": 17, "batch": 16, "hv": 21, "gram": 20, "rhs": 19,
           "monitor": 18}[kind]
    n = rng.randint(8, top)
    if lattice == "triangular":
        n = rng.choice([m for m in (8, 9, 12, 15, 16, 20) if m <= top])
    r = max(1, min(32, int(round(math.exp(rng.uniform(math.log(2), math.log(32)))))))
    if kind in ("rk4", "ab3"):
        r = min(r, 20)
    c = dict(kind=kind, n=n, r=r, lattice=lattice, model=rng.choice(("qll", "qllg")), precision=precision)
    if kind in ("rk4", "ab3", "batch", "rhs"):
        c["kappa"] = round(10.0 ** rng.uniform(-2.0, 0.0), 4)
    if kind in ("rk4", "ab3", "batch"):
        c["dt"] = rng.choice((0.005, 0.01))
        c["steps"] = rng.randint(4, 6) if kind == "ab3" else rng.randint(2, 4) if n <= 16 else 1
    if kind == "batch":
        c["r"] = min(r, 16)
        c["count"] = rng.randint(4, 10)
        c["sizes"] = rng.randint(5, 1 << 20)
    if kind == "gram":
        c["blocks"] = rng.randint(1, 6)
    return c


# ------------------------------------------------------------------------------------ inputs
def _pairs(lattice, n):
    """Nearest-neighbour site pairs: an open chain, a ring, or a periodic triangular lattice."""
    if lattice == "chain":
        return [(i, i + 1) for i in range(n - 1)]
    if lattice == "ring":
        return [(i, (i + 1) % n) for i in range(n)]
    lx = max(d for d in range(2, n) if n % d == 0 and d * d <= n)
    ly, seen, out = n // lx, set(), []
    for y in range(ly):
        for x in range(lx):
            for dx, dy in ((1, 0), (0, 1), (1, 1)):
                i, j = y * lx + x, ((y + dy) % ly) * lx + (x + dx) % lx
                if i != j and frozenset((i, j)) not in seen:
                    seen.add(frozenset((i, j)))
                    out.append((i, j))
    return out


def _model(case, n, rng):
    """Bonds, field and DMI of the case: isotropic chains (cfg1, 3, 4, 5), the anisotropic ring (cfg2), or the
    paper's triangular lattice with DMI along z and a field along x (eq. H1)."""
    pairs = _pairs(case["lattice"], n)
    m = len(pairs)
    aniso = rng.uniform(-0.2, 0.2, m) if case["lattice"] == "ring" else np.zeros(m)
    B = {"chain": (0.0, 0.0, 0.5), "ring": (0.0, 0.0, 1.0), "triangular": (0.116, 0.0, 0.0)}[case["lattice"]]
    dz = np.full(m, 0.4) if case["lattice"] == "triangular" else None
    bonds = types.SimpleNamespace(site_i=np.array([p[0] for p in pairs], dtype=np.int32),
                                  site_j=np.array([p[1] for p in pairs], dtype=np.int32),
                                  jxy=np.ones(m), jz=1.0 + aniso)
    return bonds, B, dz


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _type(case):
    return torch.complex128 if case["precision"] == "fp64" else torch.complex64


def _orthonormal(n, r, seed):
    """Haar-distributed orthonormal columns (a complex Gaussian matrix, Cholesky QR twice), complex128."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    X = torch.randn((1 << n, r), dtype=torch.complex128, device=_device(), generator=g)
    for _ in range(2):
        L = torch.linalg.cholesky((X.mH @ X).cpu())
        X = X @ torch.linalg.inv(L).mH.to(X.device)
    return X


def _weights(r, rng):
    """A decreasing trace-one spectrum, Dirichlet(1) as in the workload recipes."""
    lam = np.sort(rng.dirichlet(np.full(r, 1.0)))[::-1]
    return np.ascontiguousarray(lam / lam.sum())


def _one(case, n, r, seed):
    """The model and the initial state of one trajectory, without the framework."""
    rng = np.random.default_rng(seed)
    bonds, B, dz = _model(case, n, rng)
    lam = _weights(r, rng)
    return bonds, B, dz, lam, _orthonormal(n, r, seed).to(_type(case)).contiguous()


def _members(case):
    """Sizes of a batch's trajectories: n = 10..18 and r = 2..16 as in cfg4, up to the case's own limits."""
    rng = np.random.default_rng(case["sizes"])
    return [(int(rng.integers(min(10, case["n"]), case["n"] + 1)), int(rng.integers(2, max(3, case["r"] + 1))),
             float(10.0 ** rng.uniform(-3.0, 0.0))) for _ in range(case["count"])]


def _blocks(case, seed):
    return [_orthonormal(case["n"], case["r"], seed + 1000003 * k).to(_type(case)).contiguous()
            for k in range(case["blocks"])]


# ------------------------------------------------------------------------------------ the calls
def _context(case, n, r, kappa, made):
    from paper_2508_21200_gb300 import Lrei
    bonds, B, dz, lam, V = made
    L = Lrei(n, bonds, B, kappa, case["model"], case["precision"], r)
    if dz is not None:
        L.set_dmi(dz)
    return L


def prepare(case, seed):
    n, r, kind = case["n"], case["r"], case["kind"]
    s = types.SimpleNamespace(case=case, kind=kind)
    if kind == "batch":
        from paper_2508_21200_gb300 import Batch
        s.ctx, s.V, s.lam = [], [], []
        for t, (nt, rt, kt) in enumerate(_members(case)):
            made = _one(case, nt, rt, seed + 7919 * t)
            s.ctx.append(_context(case, nt, rt, kt, made))
            s.V.append(made[4])
            s.lam.append(made[3])
            s.ctx[-1].set_state(made[4], made[3])
        s.batch = Batch(s.ctx)
        return s
    made = _one(case, n, r, seed)
    s.ctx = _context(case, n, r, case.get("kappa", 0.1), made)
    s.lam, s.V = made[3], made[4]
    if kind == "hv":
        s.Y = torch.empty_like(s.V)
    elif kind == "gram":
        s.blocks = _blocks(case, seed)
        s.ctx.set_state(s.V, s.lam)
    elif kind in ("rhs", "monitor"):
        s.ctx.set_state(s.V, s.lam)
        s.pairs = [(i, j) for i in range(n) for j in range(i + 1, n)]
    return s


def _record(case, o):
    """A run's log line (the observables) and the spectra."""
    real = np.float64 if case["precision"] == "fp64" else np.float32
    line = np.array([o[k] for k in ("energy", "mx", "my", "mz", "purity", "trace", "comm_norm")], dtype=real)
    return line, np.asarray(o["ritz"], dtype=real), np.asarray(o["lambda0"], dtype=real)


def _aligned(V0, V):
    """V with each column's phase relative to the initial column removed."""
    z = (V0.conj() * V).sum(0)
    return V * (z.conj() / z.abs())


def run(state):
    case, kind = state.case, state.kind
    if kind in ("rk4", "ab3"):
        L = state.ctx
        L.set_state(state.V, state.lam)
        L.step(case["dt"], kind, case["steps"])
        line, ritz, lam = _record(case, L.observables())
        V, _, t = L.get_state()
        return {"V": _aligned(state.V, V), "line": line, "ritz": ritz, "lam": lam, "t": t}
    if kind == "batch":
        for L, V, lam in zip(state.ctx, state.V, state.lam):
            L.set_state(V, lam)
        state.batch.step(case["dt"], case["steps"])
        out = []
        for L, V in zip(state.ctx, state.V):
            line, ritz, _ = _record(case, L.observables())
            out.append({"V": _aligned(V, L.get_state()[0]), "line": line, "ritz": ritz})
        return out
    if kind == "hv":
        state.ctx.apply_h(state.V, state.Y)
        return state.Y
    if kind == "gram":
        return state.ctx.gram(state.blocks).to(state.V.dtype)
    if kind == "rhs":
        Z, W, G = state.ctx.rhs(0)
        return {"Z": Z, "W": W, "G": G if case["precision"] == "fp64" else G.astype(np.complex64)}
    line, _, lam = _record(case, state.ctx.observables())
    R, concurrence, negativity = state.ctx.two_spin_rdm(state.pairs)
    real = line.dtype
    return {"line": line, "lam": lam, "R": R if real == np.float64 else R.astype(np.complex64),
            "concurrence": concurrence.astype(real), "negativity": negativity.astype(real)}


# ------------------------------------------------------------------------------------ the least work
def work(case):
    """Bytes: the factor in and out of each step or pass.  Flops (complex multiply-add = 8): per RK4 step four H V, and
    per stage the Gram V* H V and the complement (16 r^2 N), the Gram and projection of the final r columns (16 r^2 N);
    an AB step has one H V and one stage, its start-up steps are RK4 steps."""
    kind = case["kind"]
    elem = 16 if case["precision"] == "fp64" else 8

    def hv(n, r):
        m = len(_pairs(case["lattice"], n))
        flips = m / 2 + (n if case["lattice"] == "triangular" else 0)
        per = 8 if case["lattice"] == "triangular" else 4
        return float(1 << n) * r * per * (flips + 1)

    def steps(n, r):
        N, rk4 = float(1 << n), case["steps"] if kind != "ab3" else min(2, case["steps"])
        ab = case["steps"] - rk4
        one = 16.0 * r * r * N
        return {"bytes": case["steps"] * 2 * N * r * elem,
                "flops": rk4 * (4 * (hv(n, r) + one) + one) + ab * (hv(n, r) + 2 * one)}

    n, r = case["n"], case["r"]
    N = float(1 << n)
    if kind in ("rk4", "ab3"):
        return steps(n, r)
    if kind == "batch":
        w = [steps(nt, rt) for nt, rt, _ in _members(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "hv":
        return {"bytes": 2 * N * r * elem, "flops": hv(n, r)}
    if kind == "gram":
        m = case["blocks"]
        return {"bytes": m * N * r * elem + m * r * r * elem, "flops": 8.0 * m * r * r * N}
    if kind == "rhs":
        return {"bytes": 3 * N * r * elem, "flops": hv(n, r) + 24.0 * r * r * N}
    pairs = n * (n - 1) // 2
    return {"bytes": N * r * elem, "flops": hv(n, r) + 16.0 * r * r * N + pairs * 20.0 * r * N}


# ------------------------------------------------------------------------------------ in 64 bits
def _hamiltonian(made, n):
    """H as a function on N x r blocks (eq. H1: exchange, DMI along z, field), gathered bond by bond."""
    bonds, B, dz = made[:3]
    dev = _device()
    b = torch.arange(1 << n, device=dev)
    one = torch.ones(1 << n, dtype=torch.float64, device=dev)
    diag = 0.0 * one
    terms = []
    for k, (i, j) in enumerate(zip(bonds.site_i.tolist(), bonds.site_j.tolist())):
        pi, pj = n - 1 - i, n - 1 - j
        bi, bj = (b >> pi) & 1, (b >> pj) & 1
        anti = bi != bj
        diag += torch.where(anti, -0.5 * one, 0.5 * one) * float(bonds.jz[k])
        d = one * (0.0 if dz is None else float(dz[k]))
        amp = torch.complex(one * float(bonds.jxy[k]), torch.where(bi == 0, d, -d)) * anti
        terms.append((b ^ ((1 << pi) | (1 << pj)), amp))
    for p in range(n):
        up = ((b >> p) & 1) == 0
        diag += torch.where(up, 0.5 * one, -0.5 * one) * B[2]
        if B[0] or B[1]:
            terms.append((b ^ (1 << p), torch.complex(0.5 * B[0] * one, torch.where(up, -0.5 * B[1] * one, 0.5 * B[1] * one))))

    def apply(X):
        Y = diag[:, None] * X
        for at, amp in terms:
            Y += amp[:, None] * X[at]
        return Y
    return apply


def _start(lam, V):
    """rho_0 = V diag(lam) V* as orthonormal columns and decreasing eigenvalues."""
    Q, R = torch.linalg.qr(V.to(torch.complex128))
    w, E = torch.linalg.eigh(R @ (torch.as_tensor(lam, device=V.device).to(torch.complex128)[:, None] * R.mH))
    return Q @ E.flip(1), w.flip(0)


def _rhs(H, V, lam, kappa, model):
    """f(rho) = Z V* + V W* (Secs. 3.3-3.5 and 4), and G = V* H V."""
    HV = H(V)
    G = V.mH @ HV
    G = (G + G.mH) / 2
    d = lam[:, None] - lam[None, :]
    if model == "qllg":
        X, c = 1j * d * G / (1 - 1j * kappa * d), 1j * lam / (1 - 1j * kappa * lam)
    else:
        X, c = (1j * d - kappa * d * d) * G, (1j - kappa * lam) * lam
    W = (HV - V @ G) * c.conj()
    return V @ X + W, W, G


def _top(parts, r):
    """The r largest eigenpairs of sum U F* over (U, F) in parts, all ranges spanned by the U and F blocks."""
    U, F = torch.cat([p[0] for p in parts], 1), torch.cat([p[1] for p in parts], 1)
    span = []
    for p in parts:
        for x in p:
            if not any(x is y for y in span):
                span.append(x)
    Q, _ = torch.linalg.qr(torch.cat(span, 1))
    M = (Q.mH @ U) @ (Q.mH @ F).mH
    w, E = torch.linalg.eigh((M + M.mH) / 2)
    return Q @ E[:, -r:].flip(1), w[-r:].flip(0)


def _evolve(H, V, lam, kappa, model, dt, kind, steps):
    """LREI-RK4 (classic tableau) or LREI-AB3 with two RK4 steps first: the state and its last unprojected spectrum."""
    r, past, mu = V.shape[1], [], lam
    for k in range(steps):
        Z, W, _ = _rhs(H, V, lam, kappa, model)
        past = ([(V, Z, W)] + past)[:3]
        if kind == "ab3" and k >= 2:
            parts = [(V * lam, V)]
            for c, (v, z, w) in zip((23 / 12, -16 / 12, 5 / 12), past):
                parts += [(dt * c * z, v), (v, dt * c * w)]
            V, mu = _top(parts, r)
            continue
        stages, first = [(V, Z, W)], V * lam
        for a in (0.5, 0.5, 1.0):
            v, z, w = stages[-1]
            v, _ = _top([(first, V), (dt * a * z, v), (v, dt * a * w)], r)
            stages.append((v,) + _rhs(H, v, lam, kappa, model)[:2])
        parts = [(first, V)]
        for c, (v, z, w) in zip((1 / 6, 2 / 6, 2 / 6, 1 / 6), stages):
            parts += [(dt * c * z, v), (v, dt * c * w)]
        V, mu = _top(parts, r)
    return V, mu


def _measured(H, n, V, lam):
    """energy, mx, my, mz, purity, trace and ||[rho, H]|| of V diag(lam) V* with orthonormal V."""
    b = torch.arange(1 << n, device=V.device)
    HV = H(V)
    G = V.mH @ HV
    x, y, z = torch.zeros_like(V), torch.zeros_like(V), torch.zeros_like(V)
    for p in range(n):
        s = (0.5 - ((b >> p) & 1).to(torch.float64))[:, None]
        f = V[b ^ (1 << p)]
        x += 0.5 * f
        y += -1j * s * f
        z += s * V
    e = lambda A: float(((V.conj() * A).sum(0).real * lam).sum())  # noqa: E731
    comm = 2 * float(((HV.abs() ** 2).sum(0) * lam ** 2).sum()) - 2 * float((lam[:, None] * lam[None, :] * G.abs() ** 2).sum())
    return np.array([e(HV), e(x) / n, e(y) / n, e(z) / n, float((lam ** 2).sum()), float(lam.sum()),
                     math.sqrt(max(comm, 0.0))])


def exact(case, seed):
    n, r, kind = case["n"], case["r"], case["kind"]
    if kind in ("rk4", "ab3") and n >= 21:
        return None
    if kind == "gram":
        blocks = [x.to(torch.complex128) for x in _blocks(case, seed)]
        return torch.cat([x.mH @ blocks[-1] for x in blocks])
    if kind == "batch":
        out = []
        for t, (nt, rt, kt) in enumerate(_members(case)):
            made = _one(case, nt, rt, seed + 7919 * t)
            H = _hamiltonian(made, nt)
            V, lam = _start(made[3], made[4])
            V, mu = _evolve(H, V, lam, kt, case["model"], case["dt"], "rk4", case["steps"])
            out.append({"V": _aligned(made[4].to(torch.complex128), V), "line": _measured(H, nt, V, lam),
                        "ritz": mu.cpu().numpy()})
        return out
    made = _one(case, n, r, seed)
    H = _hamiltonian(made, n)
    if kind == "hv":
        return H(made[4].to(torch.complex128))
    V, lam = _start(made[3], made[4])
    if kind == "rhs":
        Z, W, G = _rhs(H, V, lam, case["kappa"], case["model"])
        z = (made[4].to(torch.complex128).conj() * V).sum(0)
        z = z.conj() / z.abs()
        return {"Z": Z * z, "W": W * z, "G": (z.conj()[:, None] * G * z).cpu().numpy()}
    if kind in ("rk4", "ab3"):
        V, mu = _evolve(H, V, lam, case["kappa"], case["model"], case["dt"], kind, case["steps"])
        return {"V": _aligned(made[4].to(torch.complex128), V), "line": _measured(H, n, V, lam),
                "ritz": mu.cpu().numpy(), "lam": lam.cpu().numpy(), "t": case["dt"] * case["steps"]}
    R = []
    A = (V * lam.sqrt()).reshape((2,) * n + (r,))
    for i in range(n):
        for j in range(i + 1, n):
            a = A.movedim((i, j), (0, 1)).reshape(4, -1)
            R.append((a @ a.mH).cpu().numpy())
    R = np.array(R)
    T = R.reshape(-1, 2, 2, 2, 2).transpose(0, 1, 4, 3, 2).reshape(-1, 4, 4)
    negativity = np.array([-min(0.0, float(np.minimum(np.linalg.eigvalsh(t), 0.0).sum())) for t in T])
    yy = np.fliplr(np.diag([-1.0, 1.0, 1.0, -1.0]))
    s = [np.sort(np.sqrt(np.maximum(np.linalg.eigvals(x @ yy @ x.conj() @ yy).real, 0.0)))[::-1] for x in R]
    concurrence = np.array([max(0.0, x[0] - x[1] - x[2] - x[3]) for x in s])
    return {"line": _measured(H, n, V, lam), "lam": lam.cpu().numpy(), "R": R, "concurrence": concurrence,
            "negativity": negativity}
