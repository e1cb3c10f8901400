"""The calls that a user of this library makes, as cases with sizes, inputs and exact values.

The time axis: a contour Green's function of nk problems (k-points, or independent clusters) is
stepped from slice to slice.  One step at slice n reads the whole history 0..n-1, so the cases go
from the first steps of a small run (launches and latency count) to the last steps of the largest
one (the history no longer fits any cache).  Kinds of calls:

  step    Context.dyson_timestep: one Dyson time step.  `shared`: one local self-energy for all
          problems (the second-Born chain and lattice) or one per problem (momentum-dependent GW,
          clusters); `precision` is the entry point's option (fp64, f32c, df64).
  vie2    Context.vie2_timestep: one step of the bosonic susceptibility equation of GW.
  run2b   Context.run_2b: a whole self-consistent second-Born run, Matsubara set-up included
          (`model`: the Hubbard chain in k-space, or the Hubbard dimer in real space).
  batch   Batch.step: one step of an uneven batch of embedded clusters, nf = 1, 2, 4, 8.
  grad    adjoint.densities and its backward: the gradient of a final-time observable with
          respect to the driving field.

Inputs are smooth functions of the times with a few spectral modes per problem, as Green's
functions and self-energies are: G^R of size one on the diagonal, G^< of the occupation's size,
decaying and oscillating away from it.
"""
import math
from fractions import Fraction
from functools import lru_cache

import numpy as np
import torch

import paper_1911_01211_gb300 as ng
from paper_1911_01211_gb300 import adjoint
from paper_1911_01211_gb300 import workloads as wl

C128 = torch.complex128
PRECISION = {"fp64": ng.NG_FP64, "f32c": ng.NG_F32C, "df64": ng.NG_DF64}


def step(name, nk, n, ntau, h=0.02, beta=10.0, nf=1, k=5, shared=True, precision="fp64"):
    return {"name": name, "kind": "step", "nk": nk, "n": n, "ntau": ntau, "h": h, "beta": beta, "nf": nf, "k": k,
            "shared": shared, "precision": precision}


def listed():
    return [
        # the Hubbard chain benchmark (512 k-points, ntau = 800), late in the run: the largest call
        step("chain_late", 512, 1600, 800, h=0.01),
        # the same run near its beginning
        step("chain_early", 512, 240, 800, h=0.01),
        # a lattice whose sizes are multiples of nothing, a lower order of the quadrature
        step("ragged", 251, 777, 401, k=4, beta=7.5),
        # the first steps of a small run: a few microseconds of work
        step("small", 64, 40, 100, h=0.05, beta=5.0),
        # the two faster precision modes of the chain
        step("chain_f32c", 512, 1000, 800, h=0.01, precision="f32c"),
        step("lattice_df64", 256, 900, 400, precision="df64"),
        # the Dyson step of the momentum-dependent GW chain: a self-energy of its own per k-point
        step("gw_dyson", 128, 1250, 400, shared=False),
        # and the bosonic equation of its susceptibility
        {"name": "gw_chi", "kind": "vie2", "nk": 128, "n": 1250, "ntau": 400, "h": 0.02, "beta": 10.0, "nf": 1, "k": 5},
        # a whole run of the Hubbard dimer after an interaction quench: one problem, 2 x 2 blocks
        {"name": "dimer_run", "kind": "run2b", "model": "dimer", "nk": 1, "n": 200, "ntau": 200, "h": 0.02, "beta": 20.0},
        # a whole run of a small chain, set-up included
        {"name": "chain_run", "kind": "run2b", "model": "chain", "nk": 128, "n": 160, "ntau": 200, "h": 0.02, "beta": 10.0},
        # a step of independent embedded clusters of 1, 2, 4 and 8 orbitals
        {"name": "clusters", "kind": "batch", "nk": 16, "n": 500, "ntau": 300, "h": 0.02, "beta": 12.0},
        # the gradient with respect to a field on an 8 x 8 lattice, forward and backward
        {"name": "gradient", "kind": "grad", "nk": 64, "n": 100, "ntau": 80, "h": 0.04, "beta": 5.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: kinds in about the proportion of the listed ones."""
    most, room = _bytes_step(listed()[0]), _footprint(listed()[0])
    while True:
        kind = rng.choice(["step"] * 5 + ["f32c", "df64", "perk", "vie2", "dimer", "chain", "batch", "grad"])
        h, beta = round(rng.uniform(0.01, 0.05), 4), round(rng.uniform(3.0, 15.0), 2)
        if kind in ("step", "f32c", "df64", "perk", "vie2"):
            c = step("", _log(rng, 16, 640), _log(rng, 24, 2000), _log(rng, 40, 900), h=h, beta=beta,
                     k=rng.choice([3, 4, 5, 5, 5]), shared=kind != "perk",
                     precision=kind if kind in ("f32c", "df64") else "fp64")
            if kind == "vie2":
                c = {x: c[x] for x in c if x not in ("shared", "precision")} | {"kind": "vie2"}
            if _bytes_step(c) > most or _footprint(c) > room:
                continue
        elif kind == "dimer":
            c = {"kind": "run2b", "model": "dimer", "nk": 1, "n": _log(rng, 30, 240), "ntau": _log(rng, 50, 240), "h": h,
                 "beta": beta}
        elif kind == "chain":
            c = {"kind": "run2b", "model": "chain", "nk": _log(rng, 16, 160), "n": _log(rng, 20, 180),
                 "ntau": _log(rng, 50, 220), "h": h, "beta": beta}
        elif kind == "batch":
            c = {"kind": "batch", "nk": rng.randint(4, 16), "n": _log(rng, 40, 500), "ntau": _log(rng, 50, 300), "h": h,
                 "beta": beta}
        else:
            L = rng.choice([4, 6, 8])
            c = {"kind": "grad", "nk": L * L, "n": _log(rng, 20, 100), "ntau": _log(rng, 30, 80), "h": h, "beta": beta}
        c.pop("name", None)
        return c


# ------------------------------------------------------------------------------------------------
# work
# ------------------------------------------------------------------------------------------------
def _elements(n, T):
    """Stored history of one problem at slice n: two triangles and the left-mixing rows."""
    return n * (n + 1) + n * (T + 1)


def _bytes_step(c):
    dd = c.get("nf", 1) ** 2
    return 16.0 * dd * c["nk"] * (_elements(c["n"], c["ntau"]) + (2 * c["n"] + c["ntau"] + 3))


def _footprint(c):
    full = 16.0 * c.get("nf", 1) ** 2 * c["nk"] * _elements(c["n"] + 1, c["ntau"])
    extra = {"f32c": 0.5, "df64": 1.0}.get(c.get("precision"), 0.0)
    return full * (4 if c["kind"] == "vie2" else 1 if c.get("shared", True) else 2) + extra * full


def _cmacs(n, T):
    """Complex multiply-adds of one step and problem: ret and les history, the les sources, tv."""
    return n * n / 2.0 + n * (T + 1) + n * n + n * n / 2.0 + n * (T + 1)


def work(case):
    n, T, nk = case["n"], case["ntau"], case["nk"]
    if case["kind"] in ("step", "vie2"):
        return {"bytes": _bytes_step(case), "flops": 8.0 * case["nf"] ** 3 * nk * _cmacs(n, T)}
    if case["kind"] == "batch":
        b = f = 0.0
        for d, N, _ in _cluster_sizes(case):
            b += 16.0 * d * d * (_elements(n, T) + 2 * n + T + 3)
            f += 8.0 * d ** 3 * _cmacs(n, T)
        return {"bytes": b, "flops": f}
    # whole runs: three corrector passes a slice, each over the history of that slice; the gradient
    # walks back through the same sums with twice the multiply-adds
    nf = 2 if case.get("model") == "dimer" else 1
    times = 3.0 * (3.0 if case["kind"] == "grad" else 1.0)
    b = sum(16.0 * nf * nf * nk * _elements(i, T) for i in range(6, n + 1)) * times
    f = sum(8.0 * nf ** 3 * nk * _cmacs(i, T) for i in range(6, n + 1)) * times
    f += 8.0 / 3.0 * nk * ((T + 1) * nf) ** 3
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _fill(H, g, gen, scale, gamma, upto):
    """Slices 0..upto of a contour function with two decaying modes per problem and element."""
    n, T, d, nb = g.nt, g.ntau, g.nf, H.ldk
    dev = "cuda"
    P = 2

    def rnd(*shape):
        return torch.rand(shape, generator=gen, device=dev, dtype=torch.float64)

    e = 4.0 * rnd(P, 1, 1, nb) - 2.0                            # mode energies
    ga = gamma * (0.5 + rnd(P, 1, 1, nb))                       # decay rates
    A = torch.complex(rnd(P, d, d, nb) - 0.5, rnd(P, d, d, nb) - 0.5)
    A = 0.5 * scale * (A + A.transpose(1, 2).conj()) * 0.5      # hermitian amplitudes
    A = A + scale * 0.5 * torch.eye(d, device=dev, dtype=torch.float64).reshape(1, d, d, 1)
    f = 1.0 / (1.0 + torch.exp(g.beta * e))
    t = g.h * torch.arange(n + 1, device=dev, dtype=torch.float64).reshape(-1, 1, 1, 1)
    tau = (g.beta / T) * torch.arange(T + 1, device=dev, dtype=torch.float64).reshape(-1, 1, 1, 1)
    down = [torch.exp(torch.complex(-ga[p] * t, -e[p] * t)) for p in range(P)]     # e^{(-i e - g) t}
    up = [torch.exp(torch.complex(ga[p] * t, e[p] * t)) for p in range(P)]         # e^{(i e + g) t}
    lup = [torch.exp(torch.complex(ga[p] * t, -e[p] * t)) for p in range(P)]       # e^{(-i e + g) t}
    ldn = [torch.exp(torch.complex(-ga[p] * t, e[p] * t)) for p in range(P)]
    mt = [(torch.exp(e[p] * tau - torch.log1p(torch.exp(g.beta * e[p])))).to(C128) for p in range(P)]
    for j in range(upto + 1):
        a = ng.tri(j)
        r, l = H.ret[a:a + j + 1], H.les[a:a + j + 1]
        torch.mul(up[0][:j + 1], -1j * A[0] * down[0][j], out=r)
        r.addcmul_(up[1][:j + 1], -1j * A[1] * down[1][j])
        torch.mul(lup[0][:j + 1], 1j * f[0] * A[0] * ldn[0][j], out=l)
        l.addcmul_(lup[1][:j + 1], 1j * f[1] * A[1] * ldn[1][j])
        v = H.tv[j * (T + 1):(j + 1) * (T + 1)]
        torch.mul(mt[0], 1j * A[0] * down[0][j], out=v)
        v.addcmul_(mt[1], 1j * A[1] * down[1][j])
    H.mat.copy_(-sum((A[p] * torch.exp(-e[p] * tau - torch.log1p(torch.exp(-g.beta * e[p])))).to(C128) for p in range(P)))


def _zero_slice(H, g, n):
    H.ret[ng.tri(n):ng.tri(n + 1)] = 0
    H.les[ng.tri(n):ng.tri(n + 1)] = 0
    H.tv[n * (g.ntau + 1):(n + 1) * (g.ntau + 1)] = 0


def _eps(g, gen):
    d, nb = g.nf, g.nbatch
    a = torch.complex(torch.randn((d, d, nb), generator=gen, device="cuda", dtype=torch.float64),
                      torch.randn((d, d, nb), generator=gen, device="cuda", dtype=torch.float64))
    a = 0.5 * (a + a.transpose(0, 1).conj())
    t = g.h * torch.arange(-1, g.nt + 1, device="cuda", dtype=torch.float64).reshape(-1, 1, 1, 1)
    return ng.Func(g, values=(a[None] * (1.0 + 0.2 * torch.sin(2.0 * t))).contiguous())


def _cluster_sizes(case):
    """(nf, nt, index) of the batch's problems: the four orbital counts in turn, the fewest at nf = 8;
    every problem is still running at slice n."""
    dims = (1, 2, 4, 8, 1, 2, 4, 1, 2, 4, 1, 2, 1, 2, 4, 1)
    return [(dims[i % 16], case["n"] + 3 * i, i) for i in range(case["nk"])]


def _step_problem(case, seed, nf, nk, nt, shared, sig=-1):
    gen = _gen(seed)
    g = ng.Grid(nt=nt, ntau=case["ntau"], nf=nf, nbatch=nk, korder=case.get("k", 5), h=case["h"], beta=case["beta"],
                mu=0.0 if sig == 1 else 0.1, sig=sig)
    G = ng.Herm(g, zero=False)
    _fill(G, g, gen, 1.0, 0.15, case["n"] - 1)
    for n in range(case["n"], nt + 1):
        _zero_slice(G, g, n)
    S = ng.Herm(g, ldk=1 if shared else None, zero=False)
    _fill(S, g, gen, 0.3, 0.8, nt)
    return g, G, S, gen


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "step":
        g, G, S, gen = _step_problem(case, seed, case["nf"], case["nk"], n, case["shared"])
        return {"kind": kind, "g": g, "G": G, "S": S, "eps": _eps(g, gen), "ctx": ng.Context(g.korder), "n": n,
                "precision": PRECISION[case["precision"]]}
    if kind == "vie2":
        g, G, F, gen = _step_problem(case, seed, case["nf"], case["nk"], n, False, sig=1)
        Fcc, Q = ng.Herm(g, zero=False), ng.Herm(g, zero=False)
        _fill(Fcc, g, gen, 0.3, 0.8, n)
        _fill(Q, g, gen, 1.0, 0.3, n)
        return {"kind": kind, "g": g, "G": G, "F": F, "Fcc": Fcc, "Q": Q, "ctx": ng.Context(g.korder), "n": n}
    if kind == "batch":
        probs = []
        for d, nt, i in _cluster_sizes(case):
            g, G, S, gen = _step_problem(case, seed * 64 + i, d, 1, nt, True)
            probs.append((g, G, S, _eps(g, gen)))
        ctx = ng.Context(5)
        return {"kind": kind, "ctx": ctx, "batch": ctx.batch(*[[p[q] for p in probs] for q in range(4)]), "n": n,
                "probs": probs}
    rng = np.random.default_rng(seed)
    if kind == "grad":
        L = int(round(math.sqrt(case["nk"])))
        t = case["h"] * np.arange(-1, n + 1)
        A = np.where(t > 0, wl.pulse_A(t, A0=rng.uniform(0.3, 0.6), omega=rng.uniform(1.5, 2.5), t0=0.5 * t[-1],
                                       sigma=0.2 * t[-1]), 0.0)
        w = wl.square_kspace(L=L, nt=n, ntau=case["ntau"], beta=case["beta"], h=case["h"], A=A)
        g = ng.Grid(nt=n, ntau=w.ntau, nf=1, nbatch=w.nbatch, korder=5, h=w.h, beta=w.beta)
        eps0 = torch.from_numpy(w.eps0[:, 0, 0, :].real.copy()).cuda()
        return {"kind": kind, "g": g, "ctx": ng.Context(5), "eps0": eps0, "U": torch.from_numpy(np.asarray(w.U, float)).cuda()}
    if case["model"] == "dimer":
        w = wl.hubbard_dimer(nt=n, ntau=case["ntau"], beta=case["beta"], h=case["h"], J=rng.uniform(0.8, 1.2),
                             U0=rng.uniform(0.5, 1.0), U1=rng.uniform(1.2, 1.8))
    else:
        w = wl.chain_kspace(nk=case["nk"], nt=n, ntau=case["ntau"], beta=case["beta"], h=case["h"],
                            U=rng.uniform(0.8, 1.6), A0=rng.uniform(0.3, 0.6), t0=0.4 * n * case["h"], sigma=0.5)
    g = ng.Grid(nt=w.nt, ntau=w.ntau, nf=w.nf, nbatch=w.nbatch, korder=w.korder, h=w.h, beta=w.beta)
    U = ng.Func(g, values=torch.from_numpy(np.asarray(w.U, complex).reshape(-1, 1, 1, 1)), scalar=True) \
        if w.nf == 1 else ng.Func(g, scalar=True)
    U.val[:, 0, 0, 0] = torch.from_numpy(np.asarray(w.U, complex)).cuda()
    return {"kind": kind, "g": g, "G": ng.Herm(g), "Gloc": ng.Herm(g, ldk=1), "S": ng.Herm(g, ldk=1),
            "eps0": ng.Func(g, values=torch.from_numpy(w.eps0)), "mf": ng.Func(g), "U": U, "ctx": ng.Context(w.korder),
            "corrector": w.corrector, "nbar": w.nbar}


def _slice(G, g, n):
    T1 = g.ntau + 1
    return {"ret": G.ret[ng.tri(n):ng.tri(n + 1)], "les": G.les[ng.tri(n):ng.tri(n + 1)], "tv": G.tv[n * T1:(n + 1) * T1]}


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "step":
        ctx.dyson_timestep(s["g"], s["n"], s["G"], s["S"], s["eps"], precision=s["precision"])
        return _slice(s["G"], s["g"], s["n"])
    if kind == "vie2":
        ctx.vie2_timestep(s["g"], s["n"], s["G"], s["F"], s["Fcc"], s["Q"])
        return _slice(s["G"], s["g"], s["n"])
    if kind == "batch":
        s["batch"].step(s["n"])
        return [_slice(p[1], p[0], s["n"]) for p in s["probs"]]
    if kind == "grad":
        eps0 = s["eps0"].clone().requires_grad_(True)
        rho = adjoint.densities(eps0, ctx, s["g"], s["U"])
        (s["eps0"][-1] * rho[-1].real).mean().backward()
        return {"rho": rho.detach(), "grad": eps0.grad}
    g = s["g"]
    ctx.run_2b(g, s["G"], s["Gloc"], s["S"], s["eps0"], s["mf"], s["U"], corrector=s["corrector"], nbar=s["nbar"])
    return {"Gloc": list(s["Gloc"].tensors().values()), "Sigma": list(s["S"].tensors().values()), "mf": s["mf"].val,
            "last": _slice(s["G"], g, g.nt)}


# ------------------------------------------------------------------------------------------------
# exact values: the discretised equations of one step, in plain torch
# ------------------------------------------------------------------------------------------------
class _W:
    """Quadrature weights of order k: exact rationals, then 64 bits."""

    def __init__(self, k):
        self.k = k
        V = [[Fraction(j) ** a for a in range(k + 1)] for j in range(k + 1)]
        n = k + 1
        M = [V[i] + [Fraction(int(i == j)) for j in range(n)] for i in range(n)]
        for c in range(n):
            p = next(r for r in range(c, n) if M[r][c] != 0)
            M[c], M[p] = M[p], M[c]
            M[c] = [x / M[c][c] for x in M[c]]
            for r in range(n):
                if r != c:
                    M[r] = [x - M[r][c] * y for x, y in zip(M[r], M[c])]
        P = self.P = [row[n:] for row in M]
        self.D = [[float(sum((P[a][l] * a * Fraction(m) ** (a - 1) for a in range(1, n)), Fraction(0))) for l in range(n)]
                  for m in range(n)]
        self.a = [-x for x in self.D[0]]
        G = [Fraction(1)]
        c = [Fraction((-1) ** i, i + 1) for i in range(n + 1)]
        for i in range(1, n + 1):
            G.append(-sum((c[j] * G[i - j] for j in range(1, i + 1)), Fraction(0)))
        self.G = [abs(x) for x in G]

    @lru_cache(maxsize=None)
    def w(self, n):
        """Gregory row w_{n,0..max(n,k)} on the GPU."""
        k = self.k
        if n <= k:
            row = [sum((self.P[a][l] * Fraction(n) ** (a + 1) / (a + 1) for a in range(k + 1)), Fraction(0))
                   for l in range(k + 1)]
        else:
            row = [Fraction(1)] * (n + 1)
            for p in range(k + 1):
                for q in range(p + 1):
                    x = self.G[p + 1] * (-1) ** q * math.comb(p, q)
                    row[n - q] -= x
                    row[q] -= x
        return torch.tensor([float(x) for x in row], dtype=torch.float64, device="cuda")

    @lru_cache(maxsize=None)
    def R(self, m):
        """R[r][s] = int_0^m P_r(m - x) P_s(x) dx."""
        n = self.k + 1
        B = [[Fraction(m) ** (a + b + 1) * Fraction(math.factorial(a) * math.factorial(b), math.factorial(a + b + 1))
              for b in range(n)] for a in range(n)]
        return [[float(sum((self.P[a][r] * self.P[b][s] * B[a][b] for a in range(n) for b in range(n)), Fraction(0)))
                 for s in range(n)] for r in range(n)]


def _mm(x, y):
    """Products of d x d blocks [..., d, d, nk]."""
    if x.shape[-2] == 1:
        return x * y
    return torch.einsum("...abk,...bck->...ack", *torch.broadcast_tensors(x, y))


def _dg(x):
    return x.transpose(-3, -2).conj()


def _inv(x):
    return torch.linalg.inv(x.permute(2, 0, 1)).permute(1, 2, 0)


def _solve(A, B):
    """sum_l A[m][l] X[l] = B[m] of blocks, per problem."""
    n, d, nb = len(B), B[0].shape[0], B[0].shape[-1]
    M = torch.stack([torch.stack(r) for r in A]).permute(4, 0, 2, 1, 3).reshape(nb, n * d, n * d)
    Y = torch.stack(B).permute(3, 0, 1, 2).reshape(nb, n * d, d)
    return torch.linalg.solve(M, Y).reshape(nb, n, d, d).permute(1, 2, 3, 0)


def _wsum(w, x, y):
    """sum_j w_j x_j y_j of blocks."""
    return _mm(w.reshape(-1, 1, 1, 1) * x, y).sum(0)


class _Sums:
    """The history sums of slice n with the row vectors of S (retarded row, lesser column of Scc,
    left-mixing row), one row of G at a time."""

    def __init__(self, W, g, G, S, Scc, n):
        k, T, d, nb = g.korder, g.ntau, g.nf, g.nbatch
        T1 = T + 1
        self.sr, self.sl = S.ret[ng.tri(n):ng.tri(n + 1)], Scc.les[ng.tri(n):ng.tri(n + 1)]
        self.st = S.tv[n * T1:(n + 1) * T1]
        z = dict(dtype=C128, device="cuda")
        self.ret, self.tv = torch.zeros((n + 1, d, d, nb), **z), torch.zeros((T1, d, d, nb), **z)
        self.c1, self.c3, self.hist = (torch.zeros((n + 1, d, d, nb), **z) for _ in range(3))
        wn, wT = W.w(n), W.w(T)
        full = torch.ones(n + 1, dtype=torch.float64, device="cuda")
        stc = _dg(self.st.flip(0))                       # [Sigma^tv(n, T-j)]^dagger
        for j in range(n):
            row, col = G.ret[ng.tri(j):ng.tri(j + 1)], G.les[ng.tri(j):ng.tri(j + 1)]
            tv = G.tv[j * T1:(j + 1) * T1]
            # weight w_{n-m, j-m} of row j in column m: one but near either end
            w = full[:j + 1].clone()
            for m in range(max(0, n - 2 * k - 1), j + 1):
                if n - m > k:
                    w[m] = W.w(n - m)[j - m]
            om = W.w(4 * k + 4)
            lim = max(0, n - 2 * k - 1)                  # columns m < lim have rows longer than 2k+1
            if lim:
                if j >= n - k:
                    w[:min(lim, j + 1)] = om[n - j]
                lo = max(0, j - k)
                for m in range(lo, min(lim, j + 1)):
                    w[m] = om[j - m]
            self.ret[:j + 1] += _mm(self.sr[j] * w.reshape(-1, 1, 1, 1), row)
            self.tv += wn[j] * _mm(self.sr[j], tv)
            if j > k:
                self.c1[j] = _wsum(W.w(j) if j <= 2 * k + 1 else self._greg(om, j, k), row, self.sl[:j + 1])
            else:
                ext = torch.stack([row[l] if l <= j else -_dg(G.ret[ng.tri(l) + j]) for l in range(k + 1)])
                self.c1[j] = _wsum(W.w(j), ext, self.sl[:k + 1])
            self.c3[j] = _wsum(wT, tv, stc)
            self.hist[:j + 1] += _mm(col, wn[j] * _dg(self.sr[j]))
            if j:
                self.hist[j] -= _wsum(wn[:j], _dg(col[:j]), _dg(self.sr[:j]))

    @staticmethod
    def _greg(om, j, k):
        w = torch.ones(j + 1, dtype=torch.float64, device="cuda")
        w[:k + 1] = om[:k + 1]
        w[j - k:] = om[:k + 1].flip(0)
        return w


def _ctv23(W, g, S_tv, mat):
    """C_2 + C_3 of the left-mixing row (without h_tau): the Matsubara convolutions of S^tv(n, .)."""
    k, T = g.korder, g.ntau
    xi = float(g.sig)
    out = torch.zeros((T + 1, g.nf, g.nf, g.nbatch), dtype=C128, device="cuda")
    if S_tv.shape[-1] == 1 and g.nf == 1:                # one shared row: two matrix products
        A2 = torch.zeros((T + 1, T + 1), dtype=C128, device="cuda")
        A3 = torch.zeros_like(A2)
        s, fl = S_tv[:, 0, 0, 0], S_tv[:, 0, 0, 0].flip(0)
        for m in range(T + 1):
            if m > k:
                A2[m, :m + 1] = W.w(m) * fl[T - m:]
            else:
                for r in range(k + 1):
                    A2[m, r] = sum(W.R(m)[r][q] * s[q] for q in range(k + 1))
            if T - m > k:
                A3[m, :T - m + 1] = W.w(T - m) * s[m:]
            else:
                for r in range(k + 1):
                    A3[m, r] = sum(W.R(T - m)[r][q] * s[T - q] for q in range(k + 1))
        M = mat[:, 0, 0, :]
        return (xi * A2 @ M.flip(0) + A3 @ M).reshape(out.shape)
    for m in range(T + 1):
        if m > k:
            out[m] += xi * _wsum(W.w(m), S_tv[:m + 1].flip(0), mat[T - m:].flip(0))
        else:
            for r in range(k + 1):
                out[m] += xi * _mm(sum(W.R(m)[r][q] * S_tv[q] for q in range(k + 1)), mat[T - r])
        if T - m > k:
            out[m] += _wsum(W.w(T - m), S_tv[m:], mat[:T - m + 1])
        else:
            for r in range(k + 1):
                out[m] += _mm(sum(W.R(T - m)[r][q] * S_tv[T - q] for q in range(k + 1)), mat[r])
    return out


def _exact_dyson(g, G, S, eps, n):
    W, k, T, h, d = _W(g.korder), g.korder, g.ntau, g.h, g.nf
    T1, xi, htau = T + 1, float(g.sig), g.beta / g.ntau
    I = torch.eye(d, dtype=C128, device="cuda").reshape(d, d, 1).expand(d, d, g.nbatch)
    s = _Sums(W, g, G, S, S, n)

    def sret(a, b):
        return S.ret[ng.tri(a) + b] if b <= a else -_dg(S.ret[ng.tri(b) + a])

    def p(j):
        return 1j * (eps.val[j + 1] - g.mu * I)

    def M_of(m):
        return W.a[0] / h * I + p(m) + 1j * h * W.w(m)[m] * sret(m, m)

    Mi = _inv(M_of(n))
    R = {"ret": torch.zeros((n + 1, d, d, g.nbatch), dtype=C128, device="cuda")}
    R["les"] = torch.zeros_like(R["ret"])
    bdf = sum(W.a[l] * G.ret[ng.tri(n - l):ng.tri(n - l) + n - k] for l in range(1, k + 1))
    R["ret"][:n - k] = _mm(Mi, -bdf / h - 1j * h * s.ret[:n - k])
    A, B = [], []
    for j in range(1, k + 1):                            # conjugate start-up, transposed blocks
        Mh = [W.D[j][l] / h * I + 1j * h * W.w(j)[l] * sret(n - l, n - j) + (p(n - j) if l == j else 0.0)
              for l in range(k + 1)]
        A.append([x.transpose(0, 1) for x in Mh[1:]])
        B.append((1j * Mh[0]).transpose(0, 1))
    y = _solve(A, B)
    R["ret"][n] = -1j * I
    for l in range(1, k + 1):
        R["ret"][n - l] = y[l - 1].transpose(0, 1)
    bdf = sum(W.a[l] * G.tv[(n - l) * T1:(n - l + 1) * T1] for l in range(1, k + 1))
    R["tv"] = _mm(Mi, -1j * htau * _ctv23(W, g, s.st, G.mat) - bdf / h - 1j * h * s.tv)
    m0 = n - k
    bdf = sum(W.a[l] * G.les[ng.tri(n - l) + 1:ng.tri(n - l) + m0] for l in range(1, k + 1))
    q = 1j * h * s.c1[1:m0] - xi * htau * s.c3[1:m0]
    R["les"][1:m0] = _mm(q - bdf / h + 1j * h * s.hist[1:m0], _dg(Mi))
    R["les"][0] = -_dg(R["tv"][0])
    wn, wT = W.w(n), W.w(T)
    gtd = _dg(R["tv"].flip(0))
    for m in range(m0, n + 1):
        les = torch.stack([S.les[ng.tri(j) + m] if m <= j else -_dg(S.les[ng.tri(m) + j]) for j in range(n + 1)])
        q = -1j * h * _wsum(wn, les, _dg(R["ret"])) + xi * htau * _wsum(wT, S.tv[m * T1:(m + 1) * T1], gtd)
        q = q - sum(W.a[l] * R["les"][m - l] for l in range(1, k + 1)) / h
        q = q - 1j * h * _wsum(W.w(m)[:m], S.ret[ng.tri(m):ng.tri(m) + m], R["les"][:m])
        R["les"][m] = _mm(_inv(M_of(m)), q)
    return R


def _exact_vie2(g, G, F, Fcc, Q, n):
    W, k, T, h, d = _W(g.korder), g.korder, g.ntau, g.h, g.nf
    T1, xi, htau = T + 1, float(g.sig), g.beta / g.ntau
    I = torch.eye(d, dtype=C128, device="cuda").reshape(d, d, 1).expand(d, d, g.nbatch)
    s = _Sums(W, g, G, F, Fcc, n)
    fnn = F.ret[ng.tri(n) + n]
    q = _slice(Q, g, n)
    R = {"ret": torch.zeros((n + 1, d, d, g.nbatch), dtype=C128, device="cuda")}
    R["les"] = torch.zeros_like(R["ret"])
    R["ret"][n] = q["ret"][n]
    for m in range(n):
        L = n - m
        w = W.w(min(L, 4 * k + 4))
        if L > k:
            acc, wd = s.ret[m], (w[-1] if L <= 4 * k + 4 else w[0])
        else:
            acc = 0
            for j in range(1, k + 1):
                a, b = n - j, m
                x = G.ret[ng.tri(a) + b] if b <= a else -_dg(G.ret[ng.tri(b) + a])
                acc = acc + w[j] * _mm(F.ret[ng.tri(n) + n - j], x)
            wd = w[0]
        R["ret"][m] = _mm(_inv(I + h * wd * fnn), q["ret"][m] - h * acc)
    Mi = _inv(I + h * W.w(n)[n] * fnn)
    R["tv"] = _mm(Mi, q["tv"] - htau * _ctv23(W, g, s.st, G.mat) - h * s.tv)
    c = 1j * xi * htau
    R["les"][0] = -_dg(R["tv"][0])
    R["les"][1:n] = _mm(q["les"][1:n] - h * (s.c1[1:n] + s.hist[1:n]) - c * s.c3[1:n], _dg(Mi))
    c1 = _wsum(W.w(n), R["ret"], s.sl)
    c3 = _wsum(W.w(T), R["tv"], _dg(s.st.flip(0)))
    hist = _wsum(W.w(n)[:n], -_dg(R["les"][:n]), _dg(s.sr[:n]))
    R["les"][n] = _mm(q["les"][n] - h * (c1 + hist) - c * c3, _dg(Mi))
    return R


def exact(case, seed):
    """One step follows from its inputs by the sums above.  A whole self-consistent run and its
    gradient have no such value within seconds."""
    if case["kind"] not in ("step", "vie2", "batch"):
        return None
    s = prepare(case, seed)
    if case["kind"] == "step":
        return _exact_dyson(s["g"], s["G"], s["S"], s["eps"], s["n"])
    if case["kind"] == "vie2":
        return _exact_vie2(s["g"], s["G"], s["F"], s["Fcc"], s["Q"], s["n"])
    return [_exact_dyson(g, G, S, e, s["n"]) for g, G, S, e in s["probs"]]
