"""What a user has this framework do, as timed cases through its public entry points.

A case is a dict of plain values with a "kind":

  apply   y = H psi on a batch of states (syk_apply_H), both vector types, both parity sectors
  expmv   e^{zH} psi, real or imaginary time (syk_expmv)
  G       the two-point function G(t) on a time grid (syk_correlator_G)
  otoc    the regularized OTOC F(t) on a time grid (syk_otoc)
  batch   OTOCs of many coupling draws, sizes and temperatures in one call (syk_otoc_batch)
  grad    F~(t) with its derivatives by every coupling and by beta (syk_otoc_grad)
  eigs    the lowest levels of one sector (syk_lowest_eigenvalues)

Couplings and states are drawn from the seed with the distributions of the method: J_ijkl
normal with variance 6/N^3, amplitudes with standard-normal real and imaginary parts.  A curve
computed with complex64 vectors is returned as complex64, the precision it carries; complex128
results stay complex128.
"""
import itertools
import math

import numpy as np
import torch

from paper_2002_05725_gb300 import syk

C64, C128 = "complex64", "complex128"


def listed():
    return [
        # one matvec of a small sector: the smallest call, launch latency counts
        {"name": "apply_n20_b8_c64", "kind": "apply", "N": 20, "B": 8, "dtype": C64, "parity": 0},
        # a state count that is no power of two, odd sector
        {"name": "apply_n34_b6_c64", "kind": "apply", "N": 34, "B": 6, "dtype": C64, "parity": 1},
        # the benchmark's matvec: 16 random states of one draw at N = 40
        {"name": "apply_n40_b16_c64", "kind": "apply", "N": 40, "B": 16, "dtype": C64, "parity": 0},
        # one state of a large system, as towards N = 60
        {"name": "apply_n48_b1_c64", "kind": "apply", "N": 48, "B": 1, "dtype": C64, "parity": 0},
        # the complex128 reference precision
        {"name": "apply_n36_b16_c128", "kind": "apply", "N": 36, "B": 16, "dtype": C128, "parity": 0},
        # real-time evolution of the N = 32 workload's 16 states to the scrambling time
        {"name": "expmv_n32_b16_c64", "kind": "expmv", "N": 32, "B": 16, "dtype": C64, "parity": 0,
         "zr": 0.0, "zi": -5.0, "m": 40, "tol": 1e-7},
        # thermal factor e^{-beta H/4} at beta = 10 in reference precision
        {"name": "expmv_n28_b8_c128", "kind": "expmv", "N": 28, "B": 8, "dtype": C128, "parity": 1,
         "zr": -2.5, "zi": 0.0, "m": 40, "tol": 1e-12},
        # the plain method's check workload: N = 12, t in [0, 20] by 0.1, Krylov dimension 30
        {"name": "G_n12_t201_c128", "kind": "G", "N": 12, "B": 1, "dtype": C128, "beta": 5.0, "nt": 201,
         "tmax": 20.0, "m": 30, "tol": 1e-12},
        # OTOC curve of 16 states at N = 32, beta J = 10, on a coarse grid to t = 12
        {"name": "otoc_n32_b16_c64", "kind": "otoc", "N": 32, "B": 16, "dtype": C64, "beta": 10.0, "nt": 11,
         "tmax": 12.0, "m": 40, "tol": 1e-7},
        # disorder average: mixed sizes, beta J in {1, 3, 10}, 8 states per draw
        {"name": "batch_n20_28_c64", "kind": "batch", "Nmin": 20, "Nmax": 28, "Nstep": 4, "draws": 2, "B": 8,
         "dtype": C64, "nt": 11, "tmax": 12.0, "m": 40, "tol": 1e-7},
        # gradient of F~(t* = 5) at beta J = 5 by all couplings
        {"name": "grad_n28_b8_c64", "kind": "grad", "N": 28, "B": 8, "dtype": C64, "beta": 5.0, "t": 5.0, "m": 40,
         "tol": 1e-7, "quad_dz": 0.2},
        # the lowest 20 levels, for the spectral window of the finite-size rescaling
        {"name": "eigs_n28_k20_c128", "kind": "eigs", "N": 28, "k": 20, "dtype": C128, "parity": 0, "tol": 1e-8},
    ]


def _masks(N):
    """X-masks of H: one for each choice of 4, 2 or 0 spins."""
    n = N // 2
    return math.comb(n, 4) + math.comb(n, 2) + 1


def _nnz(N):
    return _masks(N) << (N // 2 - 1)


def _even(rng, lo, hi):
    return 2 * rng.randint(lo // 2, hi // 2)


def _states(rng, hi):
    """A state count up to hi: half of the time any, else a power of two."""
    if rng.random() < 0.5:
        return rng.randint(1, hi)
    return 1 << rng.randint(0, hi.bit_length() - 1)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "expmv", "expmv", "G", "otoc", "batch", "grad", "eigs"])
    while True:
        if kind == "apply":
            dtype = rng.choice([C64, C64, C128])
            c = {"kind": kind, "N": _even(rng, 12, 48), "B": _states(rng, 20), "dtype": dtype, "parity": rng.randint(0, 1)}
            # odd state counts run at a lower rate than powers of two: keep a pass below 0.1 s
            if _nnz(c["N"]) * c["B"] * (8 if dtype == C128 else 1) <= 1.2e10 or (c["B"] == 1 and dtype == C64):
                return c
        elif kind == "expmv":
            dtype = rng.choice([C64, C128])
            imag = rng.random() < 0.5
            size = math.exp(rng.uniform(math.log(0.1), math.log(6.0)))
            c = {"kind": kind, "N": _even(rng, 12, 36), "B": _states(rng, 16), "dtype": dtype,
                 "parity": rng.randint(0, 1), "zr": -round(size, 3) if imag else 0.0,
                 "zi": 0.0 if imag else -round(size, 3), "m": rng.choice([20, 30, 40]),
                 "tol": 1e-7 if dtype == C64 else 1e-12}
            if _nnz(c["N"]) * c["B"] * (8 if dtype == C128 else 1) <= 1.5e9:
                return c
        elif kind == "G":
            c = {"kind": kind, "N": _even(rng, 10, 26), "B": _states(rng, 8), "dtype": rng.choice([C64, C128]),
                 "beta": rng.choice([0.0, 1.0, 5.0, 10.0]), "nt": rng.randint(5, 201), "m": 30}
            c.update(tmax=round(0.1 * (c["nt"] - 1), 3), tol=1e-7 if c["dtype"] == C64 else 1e-12)
            if _nnz(c["N"]) * c["B"] * c["nt"] * (8 if c["dtype"] == C128 else 1) <= 2e9:
                return c
        elif kind == "otoc":
            c = {"kind": kind, "N": _even(rng, 12, 34), "B": _states(rng, 16), "dtype": rng.choice([C64, C64, C128]),
                 "beta": rng.choice([1.0, 3.0, 10.0]), "nt": rng.randint(3, 12), "tmax": round(rng.uniform(2.0, 12.0), 2),
                 "m": 40}
            c["tol"] = 1e-7 if c["dtype"] == C64 else 1e-12
            if _nnz(c["N"]) * c["B"] * c["nt"] * (8 if c["dtype"] == C128 else 1) <= 1.6e10:
                return c
        elif kind == "batch":
            lo = 4 * rng.randint(4, 6)
            c = {"kind": kind, "Nmin": lo, "Nmax": lo + 4 * rng.randint(0, 1), "Nstep": 4, "draws": rng.randint(1, 4),
                 "B": rng.choice([2, 4, 8, 8, 6]), "dtype": C64, "nt": rng.randint(4, 11),
                 "tmax": round(rng.uniform(4.0, 12.0), 2), "m": 40, "tol": 1e-7}
            if c["Nmax"] <= 24 or (c["Nmax"] == 28 and c["draws"] <= 2):
                return c
        elif kind == "grad":
            c = {"kind": kind, "N": _even(rng, 12, 28), "B": _states(rng, 8), "dtype": rng.choice([C64, C128]),
                 "beta": rng.choice([1.0, 5.0]), "t": round(rng.uniform(1.0, 5.0), 2), "m": 40,
                 "quad_dz": rng.choice([0.25, 0.5])}
            c["tol"] = 1e-7 if c["dtype"] == C64 else 1e-12
            if c["N"] <= 24 or c["dtype"] == C64:
                return c
        else:
            return {"kind": kind, "N": _even(rng, 18, 30), "k": rng.randint(4, 20), "dtype": C128,
                    "parity": rng.randint(0, 1), "tol": 1e-8}


# ---------------------------------------------------------------- inputs
def _couplings(N, rng):
    return rng.normal(0.0, math.sqrt(6.0 / N ** 3), size=math.comb(N, 4))


def _vectors(N, B, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    real = torch.float32 if dtype == C64 else torch.float64
    v = torch.randn((1 << (N // 2 - 1), B, 2), generator=g, device="cuda", dtype=real)
    return torch.view_as_complex(v)


def _sizes(c):
    """(N, beta) of each item of a batch case."""
    return [(N, beta) for N in range(c["Nmin"], c["Nmax"] + 1, c["Nstep"]) for _ in range(c["draws"])
            for beta in (1.0, 3.0, 10.0)]


def _inputs(case, seed):
    """[(J, psi)] of a case: one for each Hamiltonian and batch of states it names."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        sizes = [N for N, _ in _sizes(case)]
    else:
        sizes = [case["N"]]
    return [(_couplings(N, rng), _vectors(N, case.get("B", 1), case["dtype"], seed * 1000 + 7 * k))
            for k, N in enumerate(sizes)]


def _times(case):
    return np.linspace(0.0, case["tmax"], case["nt"])


def prepare(case, seed):
    ins = _inputs(case, seed)
    if case["kind"] == "batch":
        # the term set of a draw is shared by nothing here: one for each item
        sizes = _sizes(case)
        items = [(syk.syk_build_terms(N, J), beta, psi) for (N, beta), (J, psi) in zip(sizes, ins)]
        return {"case": case, "items": items, "times": _times(case)}
    J, psi = ins[0]
    s = {"case": case, "terms": syk.syk_build_terms(case["N"], J), "psi": psi}
    if case["kind"] == "apply":
        s["out"] = torch.empty_like(psi)
    if case["kind"] == "expmv":
        s["out"] = torch.empty_like(psi)
        code = syk.SYK_C64 if case["dtype"] == C64 else syk.SYK_C128
        nbytes = syk.syk_workspace_bytes(case["N"], code, case["m"], case["B"])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    if case["kind"] in ("G", "otoc"):
        s["times"] = _times(case)
    return s


def _as(case, *arrays):
    """Results of complex64 vectors in single precision; reference results as they are."""
    if case["dtype"] == C128:
        return list(arrays)
    return [a.astype(np.complex64 if np.iscomplexobj(a) else np.float32) for a in arrays]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "apply":
        return [syk.syk_apply_H(state["terms"], c["parity"], state["psi"], out=state["out"])]
    if kind == "expmv":
        y, _ = syk.syk_expmv(state["terms"], c["parity"], complex(c["zr"], c["zi"]), state["psi"],
                             krylov_dim=c["m"], tol=c["tol"], out=state["out"], workspace=state["ws"])
        return [y]
    if kind == "G":
        G, Z = syk.syk_correlator_G(state["terms"], c["beta"], 0, state["times"], state["psi"], krylov_dim=c["m"],
                                    tol=c["tol"])
        return _as(c, G, Z)
    if kind == "otoc":
        return _as(c, syk.syk_otoc(state["terms"], c["beta"], 0, 1, state["times"], state["psi"], krylov_dim=c["m"],
                                   tol=c["tol"]))
    if kind == "batch":
        return _as(c, *syk.syk_otoc_batch(state["items"], 0, 1, state["times"], krylov_dim=c["m"], tol=c["tol"]))
    if kind == "grad":
        return _as(c, *syk.syk_otoc_grad(state["terms"], c["beta"], 0, 1, c["t"], state["psi"], krylov_dim=c["m"],
                                         tol=c["tol"], quad_dz=c["quad_dz"]))
    ev, _, _ = syk.syk_lowest_eigenvalues(state["terms"], c["k"], state["psi"], parity=c["parity"], max_steps=2048,
                                          tol=c["tol"])
    return [ev]


# ---------------------------------------------------------------- work
def _krylov_dim(N, z, tol):
    """Vectors the Lanczos approximation of e^{zH} needs: the smallest k with
    (e rho |z| / 2k)^k <= tol, rho = twice the RMS level 2 sqrt(C(N,4) 6/N^3 / 16)."""
    rt = abs(z) * 2.0 * math.sqrt(math.comb(N, 4) * 6.0 / N ** 3 / 16.0)
    if rt == 0.0:
        return 0
    k = 1
    while k * math.log(math.e * rt / (2 * k)) > math.log(tol):
        k += 1
    return k


def _chain_applies(case, N, beta):
    """Matvecs of one state's OTOC chain, or G chain, on the case's grid."""
    t = _times(case)
    d = lambda z: _krylov_dim(N, z, case["tol"])  # noqa: E731
    if case["kind"] == "G":
        return d(beta / 2) + 2 * sum(d(b - a) for a, b in zip(t[:-1], t[1:]))
    back = sum(2 * d(complex(-beta / 4, x)) for x in t)
    return d(beta / 8) + d(beta / 4) + 2 * sum(d(b - a) for a, b in zip(t[:-1], t[1:])) + back


def work(case):
    kind, size = case["kind"], 8 if case["dtype"] == C64 else 16
    dim = lambda N: 1 << (N // 2 - 1)  # noqa: E731
    if kind == "batch":
        nb = sum(8 * math.comb(N, 4) + dim(N) * case["B"] * size + 16 * case["nt"] * case["B"] for N, _ in _sizes(case))
        fl = sum(8.0 * _nnz(N) * case["B"] * _chain_applies(case, N, beta) for N, beta in _sizes(case))
        return {"bytes": nb, "flops": fl}
    N, B = case["N"], case.get("B", 1)
    vec = dim(N) * B * size
    coup = 8 * math.comb(N, 4)
    apply = 8.0 * _nnz(N) * B
    if kind == "apply":
        return {"bytes": coup + 2 * vec, "flops": apply}
    if kind == "expmv":
        return {"bytes": coup + 2 * vec, "flops": apply * _krylov_dim(N, complex(case["zr"], case["zi"]), case["tol"])}
    if kind in ("G", "otoc"):
        return {"bytes": coup + vec + 16 * case["nt"] * B, "flops": apply * _chain_applies(case, N, case["beta"])}
    if kind == "grad":
        # forward and adjoint evolutions of the two chains, and one inner product per term at
        # each of the 4-point Gauss-Legendre nodes
        rho = 3.0 * math.sqrt(math.comb(N, 4) * 6.0 / N ** 3 / 16.0)
        total = case["beta"] * 3.0 / 8.0 + 4.0 * case["t"]
        nodes = 4 * math.ceil(total * rho / case["quad_dz"])
        return {"bytes": coup + vec + 16 * math.comb(N, 4) * B,
                "flops": 2 * apply * _krylov_dim(N, total, case["tol"]) + nodes * 8.0 * _nnz(N) * B}
    # Lanczos with about 8 vectors per level, each orthogonalised against the ones before it
    steps = min(dim(N), 8 * case["k"])
    return {"bytes": coup + vec + 8 * case["k"], "flops": steps * apply + 8.0 * steps * steps * dim(N)}


# ---------------------------------------------------------------- exact values in 64 bits
class _Sector:
    """H of one coupling draw in one parity sector, in complex128 on the GPU.

    Majorana a on spin k = a // 2 is the Z string below k times X_k (even a) or Y_k (odd a),
    over sqrt 2; a basis state of sector p is the low n - 1 bits of its spin index."""

    def __init__(self, N, J, parity):
        self.N, self.n, self.p = N, N // 2, parity
        self.D = 1 << (self.n - 1)
        x = torch.arange(self.D, device="cuda", dtype=torch.int32)
        self.xc = x.long()
        par = x
        for s in (16, 8, 4, 2, 1):
            par = par ^ (par >> s)
        self.x = x | (((par & 1) ^ parity) << (self.n - 1))
        q = np.array(list(itertools.combinations(range(N), 4)), dtype=np.int64)
        self.J = J
        m = np.zeros(len(q), dtype=np.int64)
        z = np.zeros(len(q), dtype=np.int64)
        ph = np.zeros(len(q), dtype=np.int64)
        pc = lambda v: sum((v >> b) & 1 for b in range(self.n))  # noqa: E731
        for col in range(4):
            k, odd = q[:, col] // 2, q[:, col] & 1
            mk, zk = np.int64(1) << k, (np.int64(1) << k) - 1 + (odd << k)
            ph += odd + 2 * pc(z & mk)
            m ^= mk
            z ^= zk
        # (term psi)[x] = (i^ph / 4) (-1)^{|z & (x ^ m)|} psi[x ^ m]
        self.w = J * (1j ** (ph % 4)) / 4.0 * (1 - 2 * (pc(z & m) & 1))
        self.m, self.z = m, z

    def _sign(self, z):
        v = self.x & int(z)
        for s in (16, 8, 4, 2, 1):
            v = v ^ (v >> s)
        return 1.0 - 2.0 * (v & 1).double()

    def groups(self):
        """(compact flip, coefficient over the sector) of every X-mask."""
        order = np.argsort(self.m, kind="stable")
        cuts = np.flatnonzero(np.diff(self.m[order])) + 1
        for idx in np.split(order, cuts):
            m = int(self.m[idx[0]])
            if bin(m).count("1") == 4:
                sup = [b for b in range(self.n) if (m >> b) & 1]
                z0 = int(self.z[idx[0]]) & ~m
                s = sum((((self.z[idx] >> b) & 1) << o) for o, b in enumerate(sup))
                tab = np.zeros(16, dtype=np.complex128)
                for u in range(16):
                    v = s & u
                    tab[u] = np.sum(self.w[idx] * (1 - 2 * ((v ^ (v >> 1) ^ (v >> 2) ^ (v >> 3)) & 1)))
                u = sum((((self.x >> b) & 1) << o) for o, b in enumerate(sup))
                c = torch.from_numpy(tab).cuda()[u.long()] * self._sign(z0)
            else:
                c = torch.zeros(self.D, dtype=torch.complex128, device="cuda")
                for t in idx:
                    c += complex(self.w[t]) * self._sign(self.z[t])
            yield m & (self.D - 1), c

    def apply(self, v):
        y = torch.zeros_like(v)
        for flip, c in self.groups():
            y += c[:, None] * v[self.xc ^ flip]
        return y

    def keep(self):
        """The groups, kept for many applications."""
        g = list(self.groups())
        step = max(1, (1 << 22) // self.D)
        self.kept = [(torch.stack([self.xc ^ f for f, _ in g[k:k + step]]), torch.stack([c for _, c in g[k:k + step]]))
                     for k in range(0, len(g), step)]
        return self

    def kept_apply(self, v):
        y = torch.zeros_like(v)
        for at, c in self.kept:
            for b in range(v.shape[1]):
                y[:, b] += (c * v[:, b][at]).sum(0)
        return y

    def expmv(self, z, v):
        """Taylor series in steps of |z| |H| <= 1.5 (|H| at most 0.06 N here)."""
        steps = max(1, math.ceil(abs(z) * 0.06 * self.N / 1.5))
        for _ in range(steps):
            term, out = v, v.clone()
            for k in range(1, 26):
                term = self.kept_apply(term) * (z / steps / k)
                out += term
            v = out
        return v

    def dense(self):
        h = torch.zeros((self.D, self.D), dtype=torch.complex128, device="cuda")
        for flip, c in self.groups():
            h[self.xc, self.xc ^ flip] += c
        return h

    def chi(self, a, v):
        """chi_a psi; psi in this sector, the result in the other one."""
        k = a // 2
        x = self.x
        below = x & ((1 << k) - 1)
        for s in (16, 8, 4, 2, 1):
            below = below ^ (below >> s)
        f = (1.0 - 2.0 * (below & 1).double()).to(torch.complex128)
        if a & 1:
            f = f * 1j * (1.0 - 2.0 * ((x >> k) & 1).double())
        out = torch.empty_like(v)
        out[(x ^ (1 << k)).long() & (self.D - 1)] = v * f[:, None] / math.sqrt(2.0)
        return out


class _Spectral:
    """Both sectors of a draw by full diagonalisation."""

    def __init__(self, N, J):
        self.s = [_Sector(N, J, p) for p in (0, 1)]
        self.eig = [torch.linalg.eigh(s.dense()) for s in self.s]

    def exp(self, z, v, p):
        e, q = self.eig[p]
        return q @ (torch.exp(z * e)[:, None] * (q.mH @ v))


def _dot(a, b):
    return (a.conj() * b).sum(0)


def _exact_otoc(N, J, beta, times, psi):
    S = _Spectral(N, J)
    phi = S.exp(-beta / 8, psi, 0)
    a0 = S.exp(-beta / 4, S.s[0].chi(1, phi), 1)
    out = []
    for t in times:
        p = S.s[0].chi(0, S.exp(-1j * t, phi, 0))
        q = S.s[1].chi(0, S.exp(-1j * t, a0, 1))
        back = complex(-beta / 4, t)
        out.append(_dot(S.exp(back, p, 1), S.s[0].chi(1, S.exp(back, q, 0))))
    return torch.stack(out).cpu().numpy()


def _exact_grad(case, J, psi):
    """F~(t), its derivatives by J and beta, by automatic differentiation of dense exponentials."""
    N, t = case["N"], case["t"]
    S = [_Sector(N, J, p) for p in (0, 1)]
    D, T = S[0].D, len(J)
    Jt = torch.tensor(J, device="cuda", requires_grad=True)
    beta = torch.tensor(float(case["beta"]), dtype=torch.float64, device="cuda", requires_grad=True)
    hams = []
    for s in S:
        w = np.where(J != 0.0, s.w / np.where(J != 0.0, J, 1.0), 0.0)  # the term without its coupling
        rows = s.xc.repeat(T)
        cols = (s.xc[None, :] ^ torch.from_numpy(s.m & (D - 1)).cuda()[:, None]).reshape(-1)
        sign = torch.stack([s._sign(z) for z in s.z])
        vals = (torch.from_numpy(w).cuda() * Jt)[:, None] * sign
        hams.append(torch.zeros(D * D, dtype=torch.complex128, device="cuda").index_add(0, rows * D + cols, vals.reshape(-1))
                    .reshape(D, D))
    ex = lambda z, p: torch.linalg.matrix_exp(z * hams[p])  # noqa: E731
    chi = [[S[p].chi(a, torch.eye(D, dtype=torch.complex128, device="cuda")) for a in (0, 1)] for p in (0, 1)]
    phi = ex(-beta / 8, 0) @ psi
    a0 = ex(-beta / 4, 1) @ (chi[0][1] @ phi)
    F = []
    for tt in (t, 0.0):
        p = chi[0][0] @ (ex(-1j * tt, 0) @ phi)
        q = chi[1][0] @ (ex(-1j * tt, 1) @ a0)
        F.append(_dot(ex(-beta / 4 + 1j * tt, 1) @ p, chi[0][1] @ (ex(-beta / 4 + 1j * tt, 0) @ q)))
    Ft = F[0] / F[1]
    B = psi.shape[1]
    dJ = np.zeros((T, B), dtype=np.complex128)
    db = np.zeros(B, dtype=np.complex128)
    for b in range(B):
        for part, unit in ((Ft[b].real, 1.0), (Ft[b].imag, 1j)):
            gJ, gb = torch.autograd.grad(part, (Jt, beta), retain_graph=True)
            dJ[:, b] += unit * gJ.cpu().numpy()
            db[b] += unit * float(gb)
    return [Ft.detach().cpu().numpy(), dJ, db]


def exact(case, seed):
    ins = _inputs(case, seed)
    kind = case["kind"]
    J, psi = ins[0]
    psi = psi.to(torch.complex128)
    if kind == "apply":
        return [_Sector(case["N"], J, case["parity"]).apply(psi)]
    if kind == "expmv":
        N = case["N"]
        steps = max(1, math.ceil(abs(complex(case["zr"], case["zi"])) * 0.06 * N / 1.5))
        if _nnz(N) > 1.0e8 or steps * _nnz(N) * case["B"] > 1.5e10:  # a longer series than 20 seconds allow
            return None
        return [_Sector(N, J, case["parity"]).keep().expmv(complex(case["zr"], case["zi"]), psi)]
    if kind == "G":
        if case["N"] > 24:
            return None
        S = _Spectral(case["N"], J)
        phi = S.exp(-case["beta"] / 2, psi, 0)
        Z = _dot(phi, phi).real
        b0 = S.s[0].chi(0, phi)
        G = [_dot(S.exp(-1j * t, phi, 0), S.s[1].chi(0, S.exp(-1j * t, b0, 1))) / Z for t in _times(case)]
        return [torch.stack(G).cpu().numpy(), Z.cpu().numpy()]
    if kind == "otoc":
        return [_exact_otoc(case["N"], J, case["beta"], _times(case), psi)] if case["N"] <= 24 else None
    if kind == "batch":
        items = list(zip(_sizes(case), ins))
        small = 24 if sum(N == 24 for (N, _), _ in items) <= 6 else 20
        return [_exact_otoc(N, Jk, beta, _times(case), v.to(torch.complex128)) if N <= small else None
                for (N, beta), (Jk, v) in items]
    if kind == "grad":
        return _exact_grad(case, J, psi) if case["N"] <= 16 else None
    if case["N"] > 24:
        return None
    ev = torch.linalg.eigvalsh(_Sector(case["N"], J, case["parity"]).dense()).cpu().numpy()
    distinct = [ev[0]]
    for v in ev[1:]:
        if v - distinct[-1] > 1e-7:
            distinct.append(v)
    return [np.array(distinct[:case["k"]])]
