"""What the performance of this library is measured on: propagations of the
kinds its users run, each through the public entry points of
paper_1102_5071_gb300, over the range of sizes, number formats and operator
kinds that those entry points take.

A case is a plain dict; its "kind" says which program it stands for:

  chain     Propagator.propagate of a driven XXZ chain (fixed point, complex64
            or complex128 vectors, Krylov or Chebyshev stage exponentials)
  atom      Propagator.propagate of the radial grid atom in a laser field
            (banded operators)
  csr       Propagator.propagate of a general sparse Hermitian model
  batch     BatchPropagator.propagate of many chains of uneven size
  gradient  Propagator.fidelity_grad: the gradient of the final-state fidelity
            with respect to a piecewise-constant drive (forward and backward)

Every pass starts from the same state (copied on the device into the vector
that the library propagates in place) and returns the whole final state, or
the loss and the gradient.
"""

import math

import numpy as np
import torch

import paper_1102_5071_gb300 as P

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # The smallest system: 8 spins from the Neel state at a tight
        # tolerance, one long call.  A chain of tiny dependent steps: latency.
        dict(name="chain8", kind="chain", N=8, precision="fx", expm="krylov", order=4, dt=0.01, nsteps=100, tol=1e-12,
             state="neel", fields="uniform"),
        # A mid-size chain of an odd length, as parameter scans run them: a few
        # thousand amplitudes, too large for one SM and too small for the chip.
        dict(name="chain13", kind="chain", N=13, precision="fx", expm="krylov", order=6, dt=0.02, nsteps=10, tol=1e-10,
             state="random", fields="uniform"),
        # The ordinary production run: 20 spins, order 6, default format.
        dict(name="chain20", kind="chain", N=20, precision="fx", expm="krylov", order=6, dt=0.02, nsteps=4, tol=1e-10,
             state="random", fields="uniform"),
        # The same run in mixed precision.
        dict(name="chain20_c64", kind="chain", N=20, precision="c64", expm="krylov", order=6, dt=0.02, nsteps=4,
             tol=1e-10, state="random", fields="uniform"),
        # A long chain of odd length in the default format: vectors of 128 MiB.
        dict(name="chain23", kind="chain", N=23, precision="fx", expm="krylov", order=4, dt=0.02, nsteps=1, tol=1e-10,
             state="random", fields="uniform"),
        # The largest: 24 spins in mixed precision, the Krylov basis in HBM.
        dict(name="chain24_c64", kind="chain", N=24, precision="c64", expm="krylov", order=4, dt=0.02, nsteps=2,
             tol=1e-10, state="random", fields="uniform"),
        # complex128 throughout, the plain form the others are compared with.
        dict(name="chain18_f64", kind="chain", N=18, precision="f64", expm="krylov", order=4, dt=0.01, nsteps=4,
             tol=1e-10, state="random", fields="uniform"),
        # Chebyshev stage exponentials of the production chain.
        dict(name="chain20_cheb", kind="chain", N=20, precision="fx", expm="chebyshev", order=6, dt=0.02, nsteps=4,
             tol=1e-12, state="random", fields="uniform"),
        # The grid atom at its full size at the pulse maximum: stiff, many
        # substeps of large Krylov spaces (a shorter step than a whole pulse's).
        dict(name="atom", kind="atom", Nr=2000, L=100, precision="fx", dt=0.01, nsteps=1, tol=1e-10),
        # A general sparse model with random couplings, an odd dimension.
        dict(name="csr", kind="csr", dim=60001, per_row=6, complex=True, precision="fx", order=4, dt=0.05, nsteps=3,
             tol=1e-10),
        # A sweep over disorder and drives: 256 chains of 10 to 16 spins at once.
        dict(name="batch_c64", kind="batch", n=256, n_lo=10, n_hi=16, precision="c64", order=6, dt=0.02, nsteps=2,
             tol=1e-10),
        # One gradient of a pulse optimisation.
        dict(name="gradient16", kind="gradient", N=16, nseg=16, nsteps=32, dt=0.01, tol=1e-10),
    ]


def draw(rng):
    kind = rng.choices(["chain", "atom", "csr", "batch", "gradient"], [11, 2, 2, 3, 2])[0]
    if kind == "chain":
        precision, expm = rng.choices([("fx", "krylov"), ("c64", "krylov"), ("f64", "krylov"), ("fx", "chebyshev")],
                                      [5, 3, 2, 2])[0]
        N = rng.randint(6, {"fx": 23, "c64": 24, "f64": 20}[precision])
        order = rng.choice([2, 4, 6, 8])
        # work in units of one stage exponential of the largest size
        most = max(1, min(40, (1 << 25) // ((1 << N) * {2: 1, 4: 2, 6: 5, 8: 11}[order])))
        return dict(kind="chain", N=N, precision=precision, expm=expm, order=order,
                    dt=rng.choice([0.005, 0.01, 0.02, 0.05]) if order > 2 else rng.choice([0.001, 0.002, 0.005]),
                    nsteps=rng.randint(1, most), tol=10.0 ** -rng.randint(9, 12),
                    state=rng.choice(["random", "random", "neel"]), fields=rng.choice(["uniform", "uniform", "sites"]))
    if kind == "atom":
        L = int(round(math.exp(rng.uniform(math.log(8), math.log(100)))))
        return dict(kind="atom", Nr=int(round(math.exp(rng.uniform(math.log(200), math.log(2000))))), L=L,
                    precision=rng.choice(["fx", "fx", "c64"]), dt=rng.choice([0.002, 0.005, 0.01]), nsteps=1,
                    tol=10.0 ** -rng.randint(9, 11))
    if kind == "csr":
        return dict(kind="csr", dim=int(round(math.exp(rng.uniform(math.log(500), math.log(120000))))),
                    per_row=rng.randint(2, 8), complex=rng.random() < 0.5, precision=rng.choice(["fx", "fx", "c64", "f64"]),
                    order=rng.choice([4, 6]), dt=rng.choice([0.02, 0.05]), nsteps=rng.randint(1, 4),
                    tol=10.0 ** -rng.randint(9, 11))
    if kind == "batch":
        lo = rng.randint(6, 12)
        return dict(kind="batch", n=int(round(math.exp(rng.uniform(math.log(16), math.log(256))))), n_lo=lo,
                    n_hi=rng.randint(lo, 16), precision=rng.choice(["c64", "f64"]), order=rng.choice([4, 6]),
                    dt=rng.choice([0.01, 0.02]), nsteps=rng.randint(1, 3), tol=10.0 ** -rng.randint(9, 11))
    nseg = rng.randint(3, 16)
    return dict(kind="gradient", N=rng.randint(8, 17), nseg=nseg, nsteps=nseg * rng.randint(1, 2), dt=0.01, tol=1e-10)


# ---------------------------------------------------------------- inputs, from the seed alone
def _rng(seed, stream):
    return np.random.default_rng([seed & 0x7FFFFFFF, stream])


def _random_state(dim, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed & 0x7FFFFFFF)
    v = torch.complex(torch.randn(dim, generator=g, device=DEV, dtype=torch.float64),
                      torch.randn(dim, generator=g, device=DEV, dtype=torch.float64))
    return v / torch.linalg.vector_norm(v)


def _neel(N):
    v = torch.zeros(1 << N, dtype=torch.complex128, device=DEV)
    v[sum(1 << i for i in range(1, N, 2))] = 1.0
    return v


def _chain_data(case, seed):
    """Couplings, fields and drive of the chain: J = 1, Delta = 0.5, h_i ~ U[-1, 1], drive A cos(omega t) on
    sum_i a_i X_i with a_i = 1 or, for site-dependent fields, ~ U[0.5, 1.5]."""
    r, N = _rng(seed, 1), case["N"]
    h = r.uniform(-1.0, 1.0, N)
    a = np.ones(N) if case.get("fields", "uniform") == "uniform" else r.uniform(0.5, 1.5, N)
    return dict(J=1.0, Delta=0.5, h=h, a=a, A=r.uniform(0.8, 1.2), omega=r.uniform(1.8, 2.2))


def _chain_state(case, seed):
    return _neel(case["N"]) if case["state"] == "neel" else _random_state(1 << case["N"], seed)


ATOM = dict(dr=0.1, E0=0.05, omega=0.057, Tp=1000.0, t0=500.0)


def _atom_data(case):
    """Stored diagonals of H0 = -1/2 d^2/dr^2 + l(l+1)/(2 r^2) - 1/r and of the dipole operator (index l Nr + j)."""
    Nr, L, dr = case["Nr"], case["L"], ATOM["dr"]
    j, lq = np.tile(np.arange(Nr), L), np.repeat(np.arange(L), Nr).astype(float)
    r = (j + 1) * dr
    off = -0.5 / dr ** 2
    H0 = np.stack([1.0 / dr ** 2 + lq * (lq + 1) / (2.0 * r ** 2) - 1.0 / r, np.where(j < Nr - 1, off, 0.0),
                   np.where(j > 0, off, 0.0)])
    up = np.where(lq < L - 1, r * (lq + 1) / np.sqrt((2 * lq + 1) * (2 * lq + 3)), 0.0)
    dn = np.where(lq > 0, r * lq / np.sqrt(np.maximum((2 * lq - 1) * (2 * lq + 1), 1.0)), 0.0)
    return (np.array([0, 1, -1]), H0), (np.array([Nr, -Nr]), np.stack([up, dn]))


def _atom_drive(t):
    return ATOM["E0"] * math.sin(math.pi * t / ATOM["Tp"]) ** 2 * math.cos(ATOM["omega"] * t)


def _atom_state(case, seed):
    """A bound wave packet: r^(l+1) e^(-r/(l+1)) in the lowest angular momenta with seeded complex weights."""
    r_, Nr, L = _rng(seed, 2), case["Nr"], case["L"]
    r = torch.arange(1, Nr + 1, device=DEV, dtype=torch.float64) * ATOM["dr"]
    psi = torch.zeros(L, Nr, dtype=torch.complex128, device=DEV)
    for l in range(min(L, 8)):
        g = (l + 1) * torch.log(r) - r / (l + 1)
        g = torch.exp(g - g.max())
        w = complex(r_.normal(), r_.normal()) * 0.5 ** l
        psi[l] = w * g / torch.linalg.vector_norm(g)
    return (psi / torch.linalg.vector_norm(psi)).reshape(-1)


def _csr_data(dim, per_row, cplx, band, r):
    """(row_ptr, col, values) of a random Hermitian matrix: a real diagonal and per_row couplings to later rows."""
    rows = np.repeat(np.arange(dim), per_row)
    span = np.minimum(band, dim - 1 - rows) if band else dim - 1 - rows
    cols = rows + 1 + np.floor(r.random(rows.size) * np.maximum(span, 1)).astype(np.int64)
    ok = cols < dim
    rows, cols = rows[ok], cols[ok]
    key = np.unique(rows * dim + cols)
    rows, cols = key // dim, key % dim
    v = r.uniform(-1, 1, rows.size) + (1j * r.uniform(-1, 1, rows.size) if cplx else 0.0)
    d = np.arange(dim)
    R, C = np.concatenate([d, rows, cols]), np.concatenate([d, cols, rows])
    V = np.concatenate([r.uniform(-1, 1, dim) + 0j, v, np.conj(v)])
    order = np.argsort(R * dim + C, kind="stable")
    R, C, V = R[order], C[order], V[order]
    ptr = np.zeros(dim + 1, dtype=np.int64)
    np.cumsum(np.bincount(R, minlength=dim), out=ptr[1:])
    return ptr, C.astype(np.int32), V if cplx else V.real.copy()


def _csr_ops(case, seed):
    r = _rng(seed, 3)
    return (_csr_data(case["dim"], case["per_row"], case["complex"], 0, r),
            _csr_data(case["dim"], max(1, case["per_row"] // 2), False, 40, r))


def _csr_drive(t):
    return 0.8 * math.cos(1.3 * t)


def _batch_data(case, seed):
    """Lengths uniform in n_lo .. n_hi (part of the case), fields and drives from the seed."""
    r = _rng(seed, 4)
    out = []
    for N in _rng(case["n"], 6).integers(case["n_lo"], case["n_hi"] + 1, case["n"]):
        N = int(N)
        out.append(dict(N=N, h=r.uniform(-1, 1, N), A=r.uniform(0.5, 2.0), omega=r.uniform(1.0, 3.0)))
    return out


def _batch_states(chains, seed):
    """One buffer of all states, each normalised."""
    flat = _random_state(sum(1 << c["N"] for c in chains), seed)
    pos = 0
    for c in chains:
        v = flat[pos:pos + (1 << c["N"])]
        v /= torch.linalg.vector_norm(v)
        pos += 1 << c["N"]
    return flat


def _gradient_data(case, seed):
    r, N = _rng(seed, 5), case["N"]
    return dict(J=1.0, Delta=0.5, h=r.uniform(-1, 1, N), a=np.ones(N), omega=2.0, amps=r.uniform(-1, 1, case["nseg"]))


def _gradient_states(case, seed):
    """The initial state and a target that the pulse already reaches in part."""
    psi0 = _random_state(1 << case["N"], seed)
    phi = psi0 + _random_state(1 << case["N"], seed + 1)
    return psi0, phi / torch.linalg.vector_norm(phi)


# ---------------------------------------------------------------- the program
def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        c = _chain_data(case, seed)
        prop = P.Propagator(P.XXZChain(case["N"], c["J"], c["Delta"], c["h"]), [P.XField(case["N"], c["a"])],
                            [lambda t: c["A"] * math.cos(c["omega"] * t)], precision=case["precision"],
                            expm=case["expm"], m_max=16)
        psi0 = _chain_state(case, seed)
        return dict(kind=kind, prop=prop, psi0=psi0, psi=torch.empty_like(psi0), t0=0.0, case=case)
    if kind == "atom":
        H0, V = _atom_data(case)
        prop = P.Propagator(P.DIA(*H0), [P.DIA(*V)], [_atom_drive], precision=case["precision"], m_max=64,
                            max_substeps=100000)
        psi0 = _atom_state(case, seed)
        return dict(kind=kind, prop=prop, psi0=psi0, psi=torch.empty_like(psi0), t0=ATOM["t0"],
                    case=dict(case, order=4))
    if kind == "csr":
        H0, V = _csr_ops(case, seed)
        prop = P.Propagator(P.CSR(*H0), [P.CSR(*V)], [_csr_drive], precision=case["precision"], m_max=24)
        psi0 = _random_state(case["dim"], seed)
        return dict(kind=kind, prop=prop, psi0=psi0, psi=torch.empty_like(psi0), t0=0.0, case=case)
    if kind == "batch":
        chains = _batch_data(case, seed)
        prop = P.BatchPropagator([P.Chain(c["N"], 1.0, 0.5, c["h"], np.ones(c["N"]), A=c["A"], omega=c["omega"])
                                  for c in chains], m_max=16, precision=case["precision"])
        psi0 = _batch_states(chains, seed)
        psi = torch.empty_like(psi0)
        views, pos = [], 0
        for c in chains:
            views.append(psi[pos:pos + (1 << c["N"])])
            pos += 1 << c["N"]
        return dict(kind=kind, prop=prop, psi0=psi0, psi=psi, views=views, t0=0.0, case=case)
    g = _gradient_data(case, seed)
    prop = P.Propagator(P.XXZChain(case["N"], g["J"], g["Delta"], g["h"]), [P.XField(case["N"], g["a"])],
                        [lambda t: 0.0], m_max=16)
    psi0, phi = _gradient_states(case, seed)
    return dict(kind=kind, prop=prop, psi0=psi0, phi=phi, amps=g["amps"], omega=g["omega"], case=case)


def run(state):
    c, prop = state["case"], state["prop"]
    if state["kind"] == "gradient":
        loss, grad, _ = prop.fidelity_grad(state["psi0"], state["phi"], 0.0, c["dt"], c["nsteps"], state["amps"],
                                           state["omega"], order=4, tol=c["tol"])
        return dict(loss=loss, grad=grad)
    state["psi"].copy_(state["psi0"])
    prop.propagate(state["views"] if state["kind"] == "batch" else state["psi"], state["t0"], c["dt"], c["nsteps"],
                   order=c["order"], tol=c["tol"])
    return state["psi"]


# ---------------------------------------------------------------- what a pass cannot do without
_STAGES = {2: 1, 4: 2, 6: 5, 8: 11}


def work(case):
    """Bytes: per operator application the applied vector, the one before it and the result once, per stage
    exponential each basis vector once, and the stored operator once per application.  Operations: real additions
    and multiplications of those.  The number of applications per exponential is a nominal one (it is decided at
    run time from the tolerance)."""
    kind = case["kind"]
    if kind == "batch":
        sizes = np.arange(case["n_lo"], case["n_hi"] + 1)
        el = case["n"] * float(np.mean(2.0 ** sizes))
        n, napp = float(np.mean(sizes)), 7.0 * case["nsteps"] * _STAGES[case["order"]]
        vb, per, extra, vecs = (8 if case["precision"] == "c64" else 16), 2 * 1.5 * n + 24, 0.0, 4.2
    elif kind == "gradient":
        el, n, napp = float(1 << case["N"]), case["N"], 7.0 * case["nsteps"] * 2 * 3
        vb, per, extra, vecs = 16, 2 * 1.5 * n + 24, 0.0, 4.2
    elif kind == "chain":
        el, n = float(1 << case["N"]), case["N"]
        napp = (7.0 if case["N"] > 8 else 8.0) * case["nsteps"] * _STAGES[case["order"]]
        vb, per, extra = (8 if case["precision"] == "c64" else 16), 2 * 1.5 * n + 24, 0.0
        vecs = 5.0 if case["expm"] == "chebyshev" else 4.2
    elif kind == "atom":
        el = float(case["Nr"] * case["L"])
        lam = 0.5 * (case["L"] - 1) * case["L"] / ATOM["dr"] ** 2 + 200.0  # spread of the spectrum
        napp = case["nsteps"] * case["dt"] * lam * 0.75 + 20.0
        vb = 8 if case["precision"] == "c64" else 16
        per, extra, vecs = 44.0, 5.0 * (4 if case["precision"] == "c64" else 8), 4.0
    else:
        el, napp = float(case["dim"]), 9.0 * case["nsteps"] * _STAGES[case["order"]]
        vb = 8 if case["precision"] == "c64" else 16
        nnz = 1 + 2 * case["per_row"] + 1 + 2 * max(1, case["per_row"] // 2)
        per = (8.0 if case["complex"] else 4.0) * nnz + 24
        extra, vecs = nnz * (4 + vb / (2 if not case["complex"] else 1)), 4.2
    return {"bytes": el * (napp * (vecs * vb + extra) + 32.0), "flops": el * napp * per}


# ---------------------------------------------------------------- the same results in 64 bits, in plain torch
class _ChainH:
    """c0 H0 + c1 sum_i a_i X_i of B chains of N sites on vectors of shape (B, 2^N)."""

    def __init__(self, N, h, a):
        h = torch.as_tensor(np.atleast_2d(h), device=DEV)
        x = torch.arange(1 << N, device=DEV)
        s = [1.0 - 2.0 * ((x >> i) & 1).double() for i in range(N)]
        self.N, self.a, self.dim = N, [float(v) for v in a], 1 << N
        self.diag = sum(0.5 * s[i] * s[i + 1] for i in range(N - 1)) + torch.zeros(1, 1, device=DEV, dtype=torch.float64)
        for i in range(N):
            self.diag = self.diag + h[:, i:i + 1] * s[i]
        ph = np.abs(np.asarray(h.cpu())).sum(1).max()
        self.r0, self.r1 = 2.5 * (N - 1) + ph, sum(abs(v) for v in self.a)

    def x(self, v):
        out = torch.zeros_like(v)
        for i in range(self.N):
            out += self.a[i] * v.view(v.shape[0], -1, 2, 1 << i).flip(2).reshape(v.shape)
        return out

    def h0(self, v):
        out = self.diag * v
        for i in range(self.N - 1):
            o, w = out.view(v.shape[0], -1, 2, 2, 1 << i), v.view(v.shape[0], -1, 2, 2, 1 << i)
            o[:, :, 0, 1] += 2.0 * w[:, :, 1, 0]
            o[:, :, 1, 0] += 2.0 * w[:, :, 0, 1]
        return out

    def __call__(self, c0, c1, v):
        return c0 * self.h0(v) + c1 * self.x(v)


def _taylor(H, c0, c1, tau, v, bound):
    """exp(-i tau H) v by the Taylor series in substeps of norm at most 2."""
    S = max(1, int(math.ceil(bound * abs(tau) / 2.0)))
    z = bound * abs(tau) / S
    terms = next(n for n in range(4, 80) if z ** n / math.factorial(n) < 1e-18)
    for _ in range(S):
        t = v
        for n in range(1, terms):
            t = H(c0, c1, t) * (-1j * tau / S / n)
            v = v + t
    return v


def _steps(case, drive, t0, expo, v):
    """The steps of the run: orders 2 and 4 as they are (midpoint; two exponentials on two Gauss points), higher
    orders as so many fourth-order steps that their error is far below the run's own."""
    dt, n = case["dt"], case["nsteps"]
    if case["order"] == 2:
        for k in range(n):
            v = expo(1.0, drive(t0 + (k + 0.5) * dt), dt, v)
        return v
    sub = 1 if case["order"] == 4 else max(1, int(math.ceil(dt / 0.0025)))
    q, d = math.sqrt(3.0) / 6.0, dt / sub
    for k in range(n * sub):
        f1, f2 = drive(t0 + (k + 0.5 - q) * d), drive(t0 + (k + 0.5 + q) * d)
        v = expo(0.5, (0.25 + q) * f1 + (0.25 - q) * f2, d, v)
        v = expo(0.5, (0.25 - q) * f1 + (0.25 + q) * f2, d, v)
    return v


def _bessel(z):
    """J_0 .. J_K of z >= 0 until they are below 1e-18 (Miller's backward recurrence)."""
    top = int(z + 20.0 * max(z, 1.0) ** (1.0 / 3.0) + 60)
    j = np.zeros(top + 2)
    j[top] = 1e-250
    for n in range(top, 0, -1):
        j[n - 1] = 2.0 * n / z * j[n] - j[n + 1]
        if abs(j[n - 1]) > 1e200:
            j *= 1e-200
    j /= j[0] + 2.0 * j[2::2].sum()
    return j[:np.nonzero(np.abs(j) > 1e-18)[0][-1] + 1]


def _exact_atom(case, seed):
    (o0, v0), (o1, v1) = _atom_data(case)
    dim = case["Nr"] * case["L"]
    lo = float((v0[0] - np.abs(v0[1]) - np.abs(v0[2]) - 0.05 * v1.sum(0)).min())
    hi = float((v0[0] + np.abs(v0[1]) + np.abs(v0[2]) + 0.05 * v1.sum(0)).max())
    ops = [(int(o), torch.as_tensor(v, device=DEV), k) for k, (oo, vv) in enumerate(((o0, v0), (o1, v1)))
           for o, v in zip(oo, vv)]

    def expo(c0, c1, tau, v):
        mid, half = 0.5 * c0 * (lo + hi), 0.5 * c0 * (hi - lo) + abs(c1) * float(v1.sum(0).max())
        rows = {}
        for o, d, k in ops:  # the stage's diagonals, scaled to [-1, 1]
            rows[o] = rows.get(o, 0.0) + (c0, c1)[k] * d / half
        rows[0] = rows[0] - mid / half

        def A(w):
            out = rows[0] * w
            for o, d in rows.items():
                if o > 0:
                    out[:dim - o] += d[:dim - o] * w[o:]
                elif o < 0:
                    out[-o:] += d[-o:] * w[:o]
            return out

        J = _bessel(half * tau)
        a, b = v, A(v)
        acc = J[0] * a + 2.0 * J[1] * (-1j) * b
        for n in range(2, len(J)):
            a, b = b, 2.0 * A(b) - a
            acc += (2.0 * J[n] * (-1j) ** (n % 4)) * b
        return acc * complex(math.cos(mid * tau), -math.sin(mid * tau))

    return _steps(dict(case, order=4), _atom_drive, ATOM["t0"], expo, _atom_state(case, seed))


def _exact_csr(case, seed):
    mats = []
    for ptr, col, val in _csr_ops(case, seed):
        bound = float(np.add.reduceat(np.abs(val), ptr[:-1]).max())
        rows = torch.as_tensor(np.repeat(np.arange(case["dim"]), np.diff(ptr)), device=DEV)
        mats.append((rows, torch.as_tensor(col.astype(np.int64), device=DEV),
                     torch.as_tensor(val.astype(np.complex128), device=DEV), bound))

    def H(c0, c1, v):
        out = torch.zeros_like(v)
        for c, (rows, col, val, _) in zip((c0, c1), mats):
            out.index_add_(0, rows, (c * val) * v[col])
        return out

    def expo(c0, c1, tau, v):
        return _taylor(H, c0, c1, tau, v, abs(c0) * mats[0][3] + abs(c1) * mats[1][3])

    return _steps(case, _csr_drive, 0.0, expo, _random_state(case["dim"], seed))


def _exact_gradient(case, seed):
    g = _gradient_data(case, seed)
    H = _ChainH(case["N"], g["h"], g["a"])
    amps = torch.tensor(g["amps"], device=DEV, requires_grad=True)
    v, phi = (s[None] for s in _gradient_states(case, seed))
    per, bound = case["nsteps"] // case["nseg"], H.r0 + H.r1

    class Apply(torch.autograd.Function):  # c0 H0 v + c1 X v of the real symmetric H0, X
        @staticmethod
        def forward(ctx, c1, v):
            xv = H.x(v)
            ctx.save_for_backward(c1, xv)
            return 0.5 * H.h0(v) + c1 * xv

        @staticmethod
        def backward(ctx, gout):
            c1, xv = ctx.saved_tensors
            return (gout.conj() * xv).real.sum(), 0.5 * H.h0(gout) + c1 * H.x(gout)

    for k in range(case["nsteps"]):
        t, dt, q = k * case["dt"], case["dt"], math.sqrt(3.0) / 6.0
        f1, f2 = math.cos(g["omega"] * (t + (0.5 - q) * dt)), math.cos(g["omega"] * (t + (0.5 + q) * dt))
        for w1, w2 in ((0.25 + q, 0.25 - q), (0.25 - q, 0.25 + q)):
            c1 = amps[min(k // per, case["nseg"] - 1)] * (w1 * f1 + w2 * f2)
            v = _taylor(lambda c0, c, u: Apply.apply(c, u), 0.5, c1, dt, v, bound)
    ov = (phi.conj() * v).sum()
    loss = 1.0 - (ov.real ** 2 + ov.imag ** 2)
    loss.backward()
    return dict(loss=float(loss.detach()), grad=amps.grad.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "atom":
        return _exact_atom(case, seed)
    if kind == "csr":
        return _exact_csr(case, seed)
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "chain":
        c = _chain_data(case, seed)
        H = _ChainH(case["N"], c["h"], c["a"])

        def expo(c0, c1, tau, v):
            return _taylor(H, c0, c1, tau, v, abs(c0) * H.r0 + abs(c1) * H.r1)

        return _steps(case, lambda t: c["A"] * math.cos(c["omega"] * t), 0.0, expo,
                      _chain_state(case, seed)[None]).reshape(-1)
    chains = _batch_data(case, seed)
    out = _batch_states(chains, seed)
    offs = np.concatenate([[0], np.cumsum([1 << c["N"] for c in chains])])
    for N in sorted({c["N"] for c in chains}):  # the chains of one size together
        idx = [i for i, c in enumerate(chains) if c["N"] == N]
        H = _ChainH(N, np.stack([chains[i]["h"] for i in idx]), np.ones(N))
        A, w = np.array([chains[i]["A"] for i in idx]), np.array([chains[i]["omega"] for i in idx])

        def expo(c0, c1, tau, v):
            return _taylor(H, c0, torch.as_tensor(c1, device=DEV)[:, None], tau, v,
                           abs(c0) * H.r0 + float(np.abs(c1).max()) * H.r1)

        v = torch.stack([out[offs[i]:offs[i + 1]] for i in idx])
        v = _steps(case, lambda t: A * np.cos(w * t), 0.0, expo, v)
        for k, i in enumerate(idx):
            out[offs[i]:offs[i + 1]] = v[k]
    return out
