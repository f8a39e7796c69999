"""The calls that a user of this library makes, as measurable cases.

A case is a dict of plain values.  ``kind`` says which entry point it goes
through, ``precision`` the arithmetic the caller asks for, ``N`` and ``L`` the
ribbon (dimer lines, unit cells), ``nE`` energies spread over [``lo``, ``hi``]
eV, ``W`` the Anderson disorder in eV and ``p`` the edge roughness.  The sizes
are those of the standard workloads and the tests (N = 11, 101, 245, 501 and
the uneven batch N = 51 .. 401), shortened along the ribbon to calls of at most
about a second: the work per unit cell does not depend on the length.

Disorder and energies come from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

T_HOP = -2.7
ETA = 1e-8
PREC = {"fp64": 0, "mixed": 1, "mixed_tc": 2, "fp64_tc": 3}


def _lib():
    from paper_1107_5300_gb300 import rgf
    return rgf


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: T of one narrow ribbon at one energy, numpy in and out
        dict(name="host_n11_one_energy", kind="host", precision="fp64", N=11, L=50, nE=1,
             lo=0.4, hi=0.4, W=0.1, p=0.0),
        # a conductance curve of the narrow ribbon, 201 energies, plain binary64
        dict(name="host_n11_curve", kind="host", precision="fp64", N=11, L=50, nE=201,
             lo=-1.0, hi=1.0, W=0.1, p=0.0),
        # the 30 nm ribbon: a prepared batch of 69 energies replayed as a graph,
        # the charge-neutrality point and its neighbours among them
        dict(name="graph_n245", kind="graph", precision="mixed_tc", N=245, L=320, nE=69,
             lo=-0.5, hi=0.5, W=0.25, p=0.0),
        # the same ribbon when the caller wants binary64 storage
        dict(name="dev_n245_fp64tc", kind="dev", precision="fp64_tc", N=245, L=96, nE=32,
             lo=-0.5, hi=0.5, W=0.25, p=0.0),
        # plain binary64 over an energy window, device buffers
        dict(name="dev_n101_fp64", kind="dev", precision="fp64", N=101, L=200, nE=64,
             lo=-0.8, hi=0.8, W=0.15, p=0.0),
        # a caller that may not allocate: double-float on the pipes, rough edges
        dict(name="noalloc_n123_mixed", kind="noalloc", precision="mixed", N=123, L=150, nE=24,
             lo=-0.7, hi=0.9, W=0.1, p=0.05),
        # many ribbons of different width and length in one call
        dict(name="batch_uneven", kind="batch", precision="mixed_tc", N=51, Nhi=401, L=20, Lhi=200,
             nE=192, lo=-1.0, hi=1.0, W=0.1, p=0.05),
        # a wide ribbon with rough edges (columns of 251 orbitals, several tensor tiles)
        dict(name="dev_n501_wide", kind="dev", precision="mixed_tc", N=501, L=40, nE=32,
             lo=-0.3, hi=0.3, W=0.1, p=0.02),
        # one chain, cut into as many domains as there are multiprocessors to run them
        dict(name="one_chain_domains", kind="domains", precision="mixed_tc", N=245, L=1200, nE=1,
             lo=0.37, hi=0.37, W=0.1, p=0.0),
        # training step: forward and backward through autograd (weighted sum over energies)
        dict(name="autograd_n101", kind="autograd", precision="mixed_tc", N=101, L=60, nE=64,
             lo=0.15, hi=0.8, W=0.15, p=0.0),
        # sensitivity maps per energy, binary64, rough edges, numpy in and out
        dict(name="grad_n61_fp64", kind="grad", precision="fp64", N=61, L=40, nE=48,
             lo=-0.8, hi=0.8, W=0.15, p=0.05),
        # local density of states maps
        dict(name="ldos_n151", kind="ldos", precision="fp64_tc", N=151, L=32, nE=40,
             lo=0.1, hi=0.9, W=0.1, p=0.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["host", "graph", "dev", "dev", "noalloc", "batch", "domains", "autograd",
                       "grad", "ldos"])
    W = round(rng.uniform(0.05, 0.25), 3)
    p = rng.choice([0.0, 0.0, 0.02, 0.05])
    prec = rng.choice(["mixed_tc", "mixed_tc", "mixed_tc", "mixed", "fp64_tc", "fp64"])
    if kind == "host":
        return dict(kind=kind, precision=rng.choice(["fp64", "mixed_tc"]), N=_logint(rng, 11, 64),
                    L=_logint(rng, 10, 200), nE=_logint(rng, 8, 256), lo=-1.0, hi=1.0, W=W, p=p)
    if kind in ("graph", "dev"):
        N, nE = _logint(rng, 51, 401), _logint(rng, 16, 128)
        return dict(kind=kind, precision=prec, N=N, L=_length(rng, N, nE, prec, 1.0), nE=nE,
                    lo=-0.7, hi=0.7, W=W, p=p)
    if kind == "noalloc":
        N = _logint(rng, 24, 245)
        nE = min(_logint(rng, 8, 64), int(21 * (245 / N) ** 2))
        return dict(kind=kind, precision=prec, N=N, L=_length(rng, N, nE, prec, 1.0), nE=nE,
                    lo=-0.9, hi=0.9, W=W, p=p)
    if kind == "batch":
        Nlo = rng.randint(31, 101)
        return dict(kind=kind, precision="mixed_tc", N=Nlo, Nhi=rng.randint(151, 401), L=10,
                    Lhi=rng.randint(40, 200), nE=rng.randint(48, 192), lo=-1.0, hi=1.0, W=0.1, p=0.05)
    if kind == "domains":
        return dict(kind=kind, precision=rng.choice(["mixed_tc", "fp64_tc"]), N=rng.randint(101, 301),
                    L=_logint(rng, 150, 1200), nE=rng.randint(1, 4), lo=0.3, hi=0.6, W=0.1, p=0.0)
    N, nE = _logint(rng, 31, 151), _logint(rng, 16, 128)
    gp = rng.choice(["mixed_tc", "fp64_tc", "fp64"])
    return dict(kind=kind, precision=gp, N=N, L=_length(rng, N, nE, gp, 9.0, 64), nE=nE,
                lo=0.15, hi=0.85, W=round(min(W, 0.15), 3), p=p)


def _length(rng, N, nE, prec, per_cell, most=400):
    """A length whose call stays below the largest listed one (about a second)."""
    cell = 1.2e-3 * ((N + 40) / 285.0) ** 2.6 * {"mixed_tc": 1.0, "mixed": 1.5, "fp64_tc": 2.2, "fp64": 5.0}[prec]
    rounds = math.ceil(2 * nE / 152)
    hi = max(6, min(most, int(0.6 / (cell * rounds * per_cell))))
    return _logint(rng, max(4, hi // 12), hi)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _disorder(rng, N, L, W, p):
    eps = rng.uniform(-W, W, (L, 2 * N))
    rem = np.zeros((L, 2 * N), dtype=np.uint8)
    if p > 0:
        for row in (0, N - 1):
            rem[:, 2 * row:2 * row + 2] = rng.random((L, 2)) < p
    return eps, rem


def _inputs(case, seed):
    """(list of (N, L, eps, removed or None), energies): one ribbon, or one per
    chain of the uneven batch."""
    rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 7])
    nE, p = case["nE"], case["p"]
    if case["kind"] == "batch":
        ribs = []
        for _ in range(nE):
            N, L = int(rng.integers(case["N"], case["Nhi"] + 1)), int(rng.integers(case["L"], case["Lhi"] + 1))
            eps, rem = _disorder(rng, N, L, case["W"], p)
            ribs.append((N, L, eps, rem))
        E = rng.uniform(case["lo"], case["hi"], nE)
    else:
        eps, rem = _disorder(rng, case["N"], case["L"], case["W"], p)
        ribs = [(case["N"], case["L"], eps, rem if p > 0 else None)]
        E = np.linspace(case["lo"], case["hi"], nE)
        if case["kind"] == "graph" and nE > 16:
            E[-5:] = (0.0, 1e-3, -1e-3, 5e-3, -5e-3)     # around the charge-neutrality point
    return ribs, E


class _State:
    pass


def prepare(case, seed):
    rgf = _lib()
    s = _State()
    s.case, s.kind, s.prec, s.n = dict(case), case["kind"], PREC[case["precision"]], case["nE"]
    ribs, E = _inputs(case, seed)
    s.E = E
    N, L, eps, rem = ribs[0]
    s.N, s.L = N, L
    if s.kind in ("graph", "dev", "batch", "noalloc", "autograd"):
        s.Ed = torch.from_numpy(E).cuda()
        s.T = torch.empty(s.n, dtype=torch.float64, device="cuda")
        s.st = torch.empty(s.n, dtype=torch.int32, device="cuda")
    if s.kind == "batch":
        s.ribs = [rgf.Ribbon(n, l, T_HOP, onsite=e, removed=r) for n, l, e, r in ribs]
    elif s.kind in ("noalloc", "autograd"):
        s.eps = torch.from_numpy(eps).cuda()
        s.rem = torch.from_numpy(rem).cuda() if rem is not None else None
        if s.kind == "autograd":
            s.eps.requires_grad_(True)
            s.w = torch.from_numpy(np.random.default_rng([int(seed) & 0xFFFFFFFF, 8]).uniform(0.5, 1.5, s.n)).cuda()
    else:
        s.ribs = [rgf.Ribbon(N, L, T_HOP, onsite=eps, removed=rem)] * s.n
    if s.kind == "graph":
        s.batch = rgf.Batch(s.ribs, s.Ed.data_ptr(), s.n, s.T.data_ptr(), s.st.data_ptr(), ETA, ETA, s.prec)
    return s


def run(s):
    rgf = _lib()
    if s.kind == "host":
        return rgf.conductance(s.ribs, s.E, ETA, ETA, s.prec)
    if s.kind == "domains":
        rgf.set_domains(0)
        try:
            return rgf.conductance(s.ribs, s.E, ETA, ETA, s.prec)
        finally:
            rgf.set_domains(2)
    if s.kind == "grad":
        return rgf.conductance_grad(s.ribs, s.E, ETA, ETA, s.prec)
    if s.kind == "ldos":
        return rgf.ldos(s.ribs, s.E, ETA, ETA, s.prec)
    stream = torch.cuda.current_stream().cuda_stream
    if s.kind == "graph":
        s.batch.launch(stream)
        return s.T, s.st
    if s.kind in ("dev", "batch"):
        rgf.conductance_dev(s.ribs, s.Ed.data_ptr(), s.n, s.T.data_ptr(), s.st.data_ptr(), ETA, ETA, s.prec, stream)
        return s.T, s.st
    if s.kind == "noalloc":
        rgf.conductance_noalloc(s.N, s.L, T_HOP, s.eps.data_ptr(), s.rem.data_ptr() if s.rem is not None else 0,
                                s.Ed.data_ptr(), s.n, s.T.data_ptr(), s.st.data_ptr(), ETA, ETA, s.prec, stream)
        return s.T, s.st
    from paper_1107_5300_gb300 import autograd
    T = autograd.conductance(s.eps, s.Ed, s.N, removed=s.rem, precision=s.prec)
    (g,) = torch.autograd.grad((T * s.w).sum(), s.eps)
    return T.detach(), g


def _step_flops(N):
    """Real operations of one unit cell of one chain: two slice inverses and two
    corner products of ceil(N/2) and floor(N/2) orbitals (columns joined by
    single bonds fold into their neighbours)."""
    a, b = (N + 1) // 2, N // 2
    return 8.0 * (a ** 3 + a ** 3 + b ** 3 + a * b * b)


def work(case):
    ribs, E = _inputs(case, 1)
    if case["kind"] == "batch":
        cells = [(n, l, 1) for n, l, _, _ in ribs]
    else:
        cells = [(case["N"], case["L"], case["nE"])]
    flops = sum(k * l * _step_flops(n) for n, l, k in cells)
    sites = sum(l * 2 * n for n, l, _, _ in ribs)
    by = sites * (8 + (1 if case["p"] > 0 else 0)) + case["nE"] * 20
    if case["kind"] in ("grad", "ldos"):
        by += case["nE"] * sites * 8
        flops *= 3.0
    elif case["kind"] == "autograd":
        by += sites * 8
        flops *= 4.0
    return {"bytes": float(by), "flops": float(flops)}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, column by column along the ribbon
# ---------------------------------------------------------------------------

class _Plain:
    """One ribbon at a list of energies, complex128: the columns x = 0, a,
    1.5 a, 2.5 a of every cell (entry p of column c is orbital 4 p + c), removed
    atoms as isolated unit entries, the leads mode by mode in closed form."""

    def __init__(self, N, L, eps, rem, E, dev):
        f = dict(dtype=torch.complex128, device=dev)
        self.N, self.L, self.n = N, L, 4 * L
        self.K = ((N + 1) // 2, (N + 1) // 2, N // 2, N // 2)
        self.z = torch.tensor(np.asarray(E) + 1j * ETA, **f)
        e = torch.tensor(eps, dtype=torch.float64, device=dev)
        k = torch.ones_like(e) if rem is None else (torch.tensor(rem, device=dev) == 0).double()
        self.eps = [e[:, c::4].contiguous() for c in range(4)]
        self.keep = [k[:, c::4].contiguous() for c in range(4)]
        KL, KR = self.K[0], self.K[2]
        S = torch.zeros(KL, KR, dtype=torch.float64, device=dev)      # rows 2p with rows 2q + 1
        for q in range(KR):
            S[q, q] = 1.0
            if q + 1 < KL:
                S[q + 1, q] = 1.0
        I = (torch.eye(KL, dtype=torch.float64, device=dev), torch.eye(KR, dtype=torch.float64, device=dev))
        self.bond = (S.T.contiguous(), I[0], S, I[1])       # [c]: column c - 1 (rows) to column c
        zc, modes = self.z[:, None], []
        p = torch.arange(1, KL + 1, dtype=torch.float64, device=dev)
        tau = 2 * T_HOP * torch.cos(math.pi * p / (N + 1))
        # g = 1 / (z - t^2 / (z - tau^2 g)):  tau^2 z g^2 - (z^2 - t^2 + tau^2) g + z = 0
        b = zc * zc - T_HOP ** 2 + tau * tau
        sq = torch.sqrt(b * b - 4 * tau * tau * zc * zc)
        big = torch.where((b.conj() * sq).real >= 0, b + sq, b - sq)
        small, large = 2 * zc / big, big / (2 * tau * tau * zc)
        # the decaying solution: |g tau / t-chain| < 1, i.e. the one with Im g < 0
        # where they differ, else the smaller transfer
        lam = lambda g: (g * T_HOP * tau / (zc - tau * tau * g)).abs()
        self.g = torch.where(lam(small) < lam(large), small, large)
        self.w = tau * tau * self.g
        self.U = []
        for K, par in ((KL, 0), (KR, 1)):
            r = (2 * torch.arange(K, dtype=torch.float64, device=dev) + par + 1)[:, None]
            u = torch.sin(math.pi * r * torch.arange(1, K + 1, dtype=torch.float64, device=dev)[None] / (N + 1))
            self.U.append((u / u.norm(dim=0)).to(torch.complex128))

    def W(self, k):
        """Coupling of column k - 1 (rows) to column k."""
        a, b = k - 1, k
        m = self.keep[a & 3][a >> 2][:, None] * self.bond[b & 3] * self.keep[b & 3][b >> 2][None]
        return (T_HOP * m).to(torch.complex128)

    def D(self, k):
        """Diagonal z - eps of column k (1 at removed atoms), per energy."""
        c, n = k & 3, k >> 2
        keep = self.keep[c][n]
        return torch.where(keep[None] > 0, self.z[:, None] - self.eps[c][n][None], torch.ones_like(self.z)[:, None])

    def sigma(self, side):
        U = self.U[side]
        k = 0 if side == 0 else self.n - 1
        keep = self.keep[k & 3][k >> 2]
        return (U * self.w[:, None, :U.shape[0]]) @ U.T * (keep[:, None] * keep[None])

    def gamma(self, side):
        return -2.0 * self.w[:, :self.U[side].shape[0]].imag

    def transmission(self):
        clean = bool((self.keep[0][0] > 0).all())
        U = self.U[0]
        if clean:
            A = (U.T * self.D(0)[:, None, :]) @ U - torch.diag_embed(self.w[:, :U.shape[0]])
            P = torch.linalg.inv(A) @ U.T
            g = U @ P
        else:
            g = torch.linalg.inv(torch.diag_embed(self.D(0)) - self.sigma(0))
            P = U.T @ g
        for k in range(1, self.n):
            Wk = self.W(k)
            A = torch.diag_embed(self.D(k)) - Wk.T @ g @ Wk
            if k < self.n - 1:
                g = torch.linalg.inv(A)
                P = P @ Wk @ g
        V = self.U[1]
        if bool((self.keep[3][-1] > 0).all()):
            A = V.T @ A @ V - torch.diag_embed(self.w[:, :V.shape[0]])
            P = P @ Wk @ V @ torch.linalg.inv(A)
        else:
            P = P @ Wk @ torch.linalg.inv(A - self.sigma(1)) @ V
        return torch.einsum("ep,epq,eq->e", self.gamma(0), P.abs() ** 2, self.gamma(1))

    def two_sided(self, want):
        """(T, dT/d eps or the local density of states) for every energy."""
        n, nE = self.n, self.z.numel()
        Sl, Sr = self.sigma(0), self.sigma(1)
        A = lambda k: torch.diag_embed(self.D(k)) - (Sl if k == 0 else 0) - (Sr if k == n - 1 else 0)
        gr, Qr = [None] * n, [None] * n
        for k in range(n - 1, -1, -1):
            M = A(k)
            if k < n - 1:
                Wn = self.W(k + 1)
                M = M - Wn @ gr[k + 1] @ Wn.T
            gr[k] = torch.linalg.inv(M)
            Qr[k] = gr[k] if k == n - 1 else gr[k] @ Wn @ Qr[k + 1]
        cl = lambda x: x.conj().transpose(1, 2)
        Gl, Gr = 1j * (Sl - cl(Sl)), 1j * (Sr - cl(Sr))
        Mb = Gr @ cl(Qr[0]) @ Gl
        T = torch.einsum("eij,eji->e", Gl @ Qr[0] @ Gr, cl(Qr[0])).real
        out = torch.zeros(nE, self.L, 2 * self.N, dtype=torch.float64, device=self.z.device)
        gl = Pl = None
        for k in range(n):
            B = A(k)
            if k > 0:
                Wk = self.W(k)
                B = B - Wk.T @ gl @ Wk
            full = B
            if k < n - 1:
                Wn = self.W(k + 1)
                full = B - Wn @ gr[k + 1] @ Wn.T
            G = torch.linalg.inv(full)
            if want == "ldos":
                d = -torch.diagonal(G, dim1=1, dim2=2).imag / math.pi
            else:
                G1 = G if k == 0 else Pl @ Wk @ G
                GL = G if k == n - 1 else G @ Wn @ Qr[k + 1]
                d = 2.0 * torch.einsum("eib,ebi->ei", GL @ Mb, G1).real
            out[:, k >> 2, (k & 3)::4] = d * self.keep[k & 3][k >> 2]
            gl = torch.linalg.inv(B)
            Pl = gl if k == 0 else Pl @ Wk @ gl
        return T, out


def exact(case, seed):
    # column inversions of every energy; what would take too long is left out
    if case["kind"] == "batch" or case["N"] > 320 or case["nE"] * case["L"] * (case["N"] / 245.0) ** 2.5 > 2400:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    ribs, E = _inputs(case, seed)
    N, L, eps, rem = ribs[0]
    m = _Plain(N, L, eps, rem, E, dev)
    if case["kind"] in ("autograd", "grad", "ldos"):
        # T of the autograd call comes from the forward sweep
        T, out = m.two_sided("ldos" if case["kind"] == "ldos" else "grad")
        if case["kind"] == "autograd":
            w = torch.tensor(np.random.default_rng([int(seed) & 0xFFFFFFFF, 8]).uniform(0.5, 1.5, E.size), device=dev)
            return T, torch.einsum("e,eln->ln", w, out)
        return T.cpu().numpy(), out.cpu().numpy(), None
    T = m.transmission()
    return (T.cpu().numpy() if case["kind"] in ("host", "domains") else T), None
