"""Performance cases of the GFCCSD library, through its public entry points (paper_2010_04768_gb300.gfcc).

Inputs follow the synthetic recipe of the package (orbital energies, Cholesky vectors, amplitudes);
sizes run from the tiny workload (o=4 v=12 L=48) to the medium one (o=40 v=200 L=800), with v about
5 o and L about 4 v as in the named workloads.  exact() states the same quantities as 64-bit torch
expressions written from the equations of the method.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2010_04768_gb300 import gfcc

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64, C128 = torch.float64, torch.complex128


# ------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one operator product on one vector by a caller's own iterative solver: latency of the smallest call
        {"name": "sigma_ip_tiny", "kind": "sigma", "o": 4, "v": 12, "L": 48, "sectors": "IP", "precision": "fp64",
         "n_vec": 1},
        # the tiny workload: 4 frequencies, every orbital, both sectors, plain FP64
        {"name": "solve_fp64_tiny", "kind": "solve", "o": 4, "v": 12, "L": 48, "sectors": "IP+EA",
         "precision": "fp64", "n_omega": 4, "n_orb": 16, "lo": -1.0, "hi": -0.2, "eta": 0.01, "tol": 1e-8},
        # plain FP64 at odd sizes: a small molecule, frequencies and orbitals around the gap, both sectors
        {"name": "solve_fp64_odd", "kind": "solve", "o": 13, "v": 67, "L": 269, "sectors": "IP+EA",
         "precision": "fp64", "n_omega": 1, "n_orb": 7, "lo": -0.7, "hi": 0.4, "eta": 0.01, "tol": 1e-8},
        # mixed precision, ionisation, an odd middle size: two frequencies of a sweep over the valence orbitals
        {"name": "solve_mixed_ip_odd", "kind": "solve", "o": 27, "v": 133, "L": 531, "sectors": "IP",
         "precision": "mixed", "n_omega": 2, "n_orb": 15, "lo": -1.0, "hi": -0.3, "eta": 0.005, "tol": 1e-8},
        # the medium workload's ionisation sector: one frequency, the 40 orbitals nearest the gap
        {"name": "solve_mixed_ip_medium", "kind": "solve", "o": 40, "v": 200, "L": 800, "sectors": "IP",
         "precision": "mixed", "n_omega": 1, "n_orb": 40, "lo": -1.2, "hi": 0.5, "eta": 0.005, "tol": 1e-8},
        # mixed precision, attachment sector (the vvvv contraction carries it)
        {"name": "solve_mixed_ea", "kind": "solve", "o": 20, "v": 100, "L": 400, "sectors": "EA",
         "precision": "mixed", "n_omega": 1, "n_orb": 12, "lo": -0.2, "hi": 0.5, "eta": 0.005, "tol": 1e-8},
        # molecules of uneven size solved together on their own streams
        {"name": "batch_mixed_uneven", "kind": "batch", "o": 10, "step": 3, "molecules": 4, "precision": "mixed",
         "n_omega": 4, "n_orb": 8, "lo": -1.0, "hi": -0.3, "eta": 0.005, "tol": 1e-8},
        # closed-shell spin-adapted ionisation (the medium closed-shell workload, 10 highest occupied orbitals)
        {"name": "closed_shell_medium", "kind": "rhf", "o": 30, "v": 150, "L": 600, "n_omega": 1, "n_orb": 10,
         "lo": -1.2, "hi": -0.2, "eta": 0.005, "tol": 1e-8},
        # ground-state CCSD and Lambda from the Hamiltonian, large contractions on the tensor cores
        {"name": "ccsd_lambda", "kind": "ccsd", "o": 16, "v": 80, "L": 320, "emulate": True, "lambda": True,
         "tol": 1e-8},
        # a new molecule: context set-up, one frequency, context released
        {"name": "setup_and_solve", "kind": "setup", "o": 20, "v": 100, "L": 400, "sectors": "IP+EA",
         "precision": "mixed", "n_omega": 1, "n_orb": 4, "lo": -1.0, "hi": -0.3, "eta": 0.005, "tol": 1e-8},
        # a fine spectrum and its error estimate from a reduced model (three solved frequencies)
        {"name": "mor_spectrum", "kind": "mor", "o": 16, "v": 80, "L": 320, "n_omega": 3, "n_orb": 12, "points": 500,
         "lo": -1.0, "hi": -0.3, "eta": 0.01, "tol": 1e-8},
        # training of the initial-guess model: loss and gradient of one minibatch, forward and backward
        {"name": "mlp_loss_grad", "kind": "mlp", "hidden": 256, "batch": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma", "solve", "solve", "mixed", "mixed", "batch", "rhf", "ccsd", "setup", "mor", "mlp"])
    if kind == "mlp":
        return {"kind": "mlp", "hidden": rng.choice([64, 100, 128, 200, 256]), "batch": _log_int(rng, 16, 1024)}

    def shape(lo, hi):
        o = _log_int(rng, lo, hi)
        v = int(round(o * rng.uniform(4.0, 5.2)))
        return {"o": o, "v": v, "L": int(round(v * rng.uniform(3.5, 4.2)))}

    # around the gap, where GMRES needs few iterations; the valence band (more) only for mixed ionisation
    window = {"lo": -0.7, "hi": 0.4, "eta": rng.choice([0.005, 0.01]), "tol": 1e-8}
    band = rng.choice([window, dict(window, lo=-1.0, hi=-0.3)])
    if kind == "sigma":
        return {"kind": "sigma", **shape(3, 14), "sectors": rng.choice(["IP", "EA"]), "precision": "fp64",
                "n_vec": _log_int(rng, 1, 8)}
    if kind == "solve":
        return {"kind": "solve", **shape(3, 12), "sectors": rng.choice(["IP", "EA", "IP+EA"]), "precision": "fp64",
                "n_omega": rng.randint(1, 4), "n_orb": rng.randint(2, 10), **dict(window, eta=0.01)}
    if kind == "mixed":
        sector = rng.choice(["IP", "IP", "EA"])
        return {"kind": "solve", **shape(8, 32 if sector == "IP" else 18), "sectors": sector, "precision": "mixed",
                "n_omega": rng.randint(1, 3), "n_orb": rng.randint(3, 14), **(band if sector == "IP" else window)}
    if kind == "batch":
        return {"kind": "batch", "o": rng.randint(8, 12), "step": rng.randint(1, 3), "molecules": rng.randint(2, 4),
                "precision": "mixed", "n_omega": rng.randint(1, 5), "n_orb": rng.randint(3, 8), **band}
    if kind == "rhf":
        return {"kind": "rhf", **shape(5, 26), "n_omega": rng.randint(1, 2), "n_orb": rng.randint(2, 8),
                **dict(window, lo=-1.0, hi=-0.2, eta=0.01)}
    if kind == "ccsd":
        emulate = rng.random() < 0.5
        return {"kind": "ccsd", **shape(4, 16 if emulate else 8), "emulate": emulate, "lambda": rng.random() < 0.7,
                "tol": 1e-8}
    if kind == "setup":
        return {"kind": "setup", **shape(5, 18), "sectors": rng.choice(["IP", "EA", "IP+EA"]), "precision": "mixed",
                "n_omega": 1, "n_orb": rng.randint(2, 5), **window}
    return {"kind": "mor", **shape(5, 16), "n_omega": rng.randint(2, 4), "n_orb": rng.randint(3, 10),
            "points": _log_int(rng, 60, 600), **dict(window, lo=-1.0, hi=-0.3, eta=0.01)}


# ------------------------------------------------------------------------------------------- inputs
def _antisym(g):
    return 0.5 * (g - g.transpose(0, 1) - g.transpose(2, 3) + g.transpose(0, 1).transpose(2, 3))


def _problem(o, v, L, seed, kind="spin"):
    """Host inputs by the package's recipe.  kind: spin orbitals with T, "closed" shell, or no T ("bare")."""
    gen = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 7919 * o + 31 * v + L)
    n = o + v

    def normal(*s):
        return torch.randn(*s, generator=gen, device=DEV, dtype=F64)

    eps = torch.cat([torch.sort(-1.5 + 1.2 * torch.rand(o, generator=gen, device=DEV, dtype=F64)).values,
                     torch.sort(0.1 + 1.9 * torch.rand(v, generator=gen, device=DEV, dtype=F64)).values])
    width = 1.0 / math.sqrt(o * v) if kind != "closed" else 1.0 / math.sqrt(4 * o * v)
    chol = torch.triu(normal(L, n, n))
    chol = chol + torch.triu(chol, 1).transpose(1, 2)
    chol *= width * torch.exp(-torch.arange(L, device=DEV, dtype=F64) / 12.0)[:, None, None]
    t1, t2 = torch.zeros(o, v, dtype=F64, device=DEV), None
    if kind != "bare":
        t1 = 0.01 * normal(o, v)
        g = 0.02 * normal(o, o, v, v)
        t2 = _antisym(g) if kind == "spin" else 0.5 * (g + g.permute(1, 0, 3, 2))
    cpu = [None if x is None else x.contiguous().cpu().numpy() for x in (torch.diag(eps), chol, t1, t2)]
    return SimpleNamespace(o=o, v=v, L=L, fock=cpu[0], chol=cpu[1], t1=cpu[2], t2=cpu[3], lam1=None, lam2=None)


def _orbitals(p, case):
    """The orbitals nearest the gap (both sectors, attachment) or the highest occupied ones, over the first
    virtual ones where there are not enough."""
    eps, k = np.diag(p.fock), min(case["n_orb"], p.o + p.v)
    if case.get("sectors", "IP") == "IP" and case["hi"] <= 0.0:
        lo = max(0, p.o - k)
        return np.arange(lo, lo + k, dtype=np.int32)
    mid = 0.5 * (eps[p.o - 1] + eps[p.o])
    return np.sort(np.argsort(np.abs(eps - mid), kind="stable")[:k]).astype(np.int32)


def _omegas(case, seed, count=None):
    """Frequencies of the window, spread evenly, the whole set shifted by the seed."""
    k = count or case["n_omega"]
    shift = np.random.default_rng(int(seed) + 17).uniform(0.1, 0.9)
    return case["lo"] + (case["hi"] - case["lo"]) * (np.arange(k) + shift) / k


def _molecules(case):
    return [(o, 5 * o, 20 * o) for o in range(case["o"], case["o"] + case["step"] * case["molecules"], case["step"])]


def _mlp_inputs(case, seed):
    rng = np.random.default_rng(int(seed) + 5)
    h, nb = case["hidden"], case["batch"]
    w = np.concatenate([rng.standard_normal(h * 27) * math.sqrt(2 / 27), np.zeros(h),
                        rng.standard_normal(h * h) * math.sqrt(2 / h), np.zeros(h),
                        rng.standard_normal(16 * h) * 0.1 / math.sqrt(h), np.zeros(16), np.zeros(27), np.ones(27)])
    F = rng.standard_normal((nb, 27))
    U = rng.standard_normal((nb, 9, 32)) + 1j * rng.standard_normal((nb, 9, 32))
    U[:, 1:] = 0.5 * U[:, 1:] + 0.5 * U[:, :1]       # neighbours resemble the right-hand side
    return w, F, U.conj() @ U.transpose(0, 2, 1)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        w, F, gram = _mlp_inputs(case, seed)
        model = gfcc.MLP(w, hidden=case["hidden"])
        model.set_params(w)
        return SimpleNamespace(case=case, model=model, F=F, gram=gram)
    if kind == "batch":
        ps = [_problem(*m, seed) for m in _molecules(case)]
        ctxs = [gfcc.GFCC(p, sectors="IP", precision=case["precision"]) for p in ps]
        reqs = [(_omegas(case, seed), case["eta"], _orbitals(p, case), case["tol"]) for p in ps]
        return SimpleNamespace(case=case, ctxs=ctxs, reqs=reqs)
    p = _problem(case["o"], case["v"], case["L"], seed, {"ccsd": "bare", "rhf": "closed"}.get(kind, "spin"))
    s = SimpleNamespace(case=case, p=p)
    if kind == "ccsd":
        return s
    if kind == "sigma":
        s.ctx = gfcc.GFCC(p, sectors=case["sectors"], precision=case["precision"])
        s.X = _vectors(case, seed)
        return s
    s.omegas, s.orbitals = _omegas(case, seed), _orbitals(p, case)
    if kind == "solve":
        s.ctx = gfcc.GFCC(p, sectors=case["sectors"], precision=case["precision"])
    elif kind == "rhf":
        s.ctx = gfcc.GFCC(p, sectors="IP", closed_shell=True)
    elif kind == "mor":
        s.ctx = gfcc.GFCC(p, sectors="IP", precision="mixed")
        s.mor = gfcc.MOR(s.ctx, "IP")
        s.mor.expand(s.omegas, case["eta"], s.orbitals, case["tol"])
        s.fine = _omegas(case, seed, case["points"])
    return s


def _dim(case):
    o, v = case["o"], case["v"]
    return o + o * (o - 1) // 2 * v if case["sectors"] == "IP" else v + o * (v * (v - 1) // 2)


def _vectors(case, seed):
    rng = np.random.default_rng(int(seed) + 3)
    n = (case["n_vec"], _dim(case))
    return rng.standard_normal(n) + 1j * rng.standard_normal(n)


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "sigma":
        return s.ctx.sigma(case["sectors"], s.X, case["precision"])
    if kind in ("solve", "rhf"):
        return s.ctx.solve(s.omegas, case["eta"], s.orbitals, case["tol"])
    if kind == "batch":
        return gfcc.solve_batch(s.ctxs, s.reqs)
    if kind == "setup":
        ctx = gfcc.GFCC(s.p, sectors=case["sectors"], precision=case["precision"])
        out = ctx.solve(s.omegas, case["eta"], s.orbitals, case["tol"])
        ctx.close()
        return out
    if kind == "mor":
        return s.mor.green(s.fine, case["eta"], s.orbitals, residuals=True)
    if kind == "mlp":
        return s.model.loss_grad(s.F, s.gram)
    t1, t2, l1, l2, info, code = gfcc.ccsd(s.p.fock, s.p.chol, s.p.o, tol=case["tol"], want_lambda=case["lambda"],
                                           emulate=case["emulate"])
    out = {"t1": t1, "t2": t2, "e_corr": info["e_corr"], "code": code}
    if case["lambda"]:
        out.update(l1=l1, l2=l2)
    return out


# ------------------------------------------------------------------------------------------- work
# operator products per solved system: the iterations that diagonally preconditioned GMRES needs to 1e-8 on
# these inputs in 64 bits, about 20
ITERATIONS = 20


def _sigma_flops(o, v, sector):
    """Multiplications and additions of one operator product with a complex vector."""
    if sector == "IP":
        return 2.0 * (2 * o**3 * v**2 + 0.5 * o**4 * v + 3 * o**2 * v**2 + 4 * o**3 * v)
    return 2.0 * (2 * o**2 * v**3 + 0.5 * o * v**4 + 3 * o * v**3 + 3 * o**2 * v**2)


def _setup_flops(o, v, L, sectors):
    """Leading terms of the elements of the transformed Hamiltonian: integrals and their products with T2."""
    f = 4.0 * (o * v) ** 2 * L + 2.0 * (o * v) ** 3 + 2.0 * o * v**3 * L
    if "IP" in sectors:
        f += 2.0 * o**4 * v**2 + 4.0 * o**4 * v**2 + 2.0 * o**3 * v**3
    if "EA" in sectors:
        f += v**4 * L + 0.5 * o**2 * v**4 + 2.0 * o**2 * v**4
    return f


def _operator_bytes(o, v, sectors):
    b = 0.0
    if "IP" in sectors:
        b += 8.0 * ((o * v) ** 2 + o**4 + o**2 * v * (o + v) + 2 * o**2 * v**2)
    if "EA" in sectors:
        b += 8.0 * ((o * v) ** 2 + v**4 / 4 + o * v**2 * (o + v) + 2 * o**2 * v**2 + o * v**3)
    return b


def work(case):
    kind = case["kind"]
    if kind == "mlp":
        h, nb = case["hidden"], case["batch"]
        n = 27 * h + h * h + 16 * h
        return {"bytes": 8.0 * (2 * n + nb * (27 + 162)), "flops": 6.0 * nb * n}
    if kind == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        for o, v, _ in _molecules(case):
            w["bytes"] += _operator_bytes(o, v, "IP")
            w["flops"] += case["n_omega"] * case["n_orb"] * ITERATIONS * _sigma_flops(o, v, "IP")
        return w
    o, v, L = case["o"], case["v"], case["L"]
    if kind == "ccsd":
        n, its = o + v, 8 * (2 if case["lambda"] else 1)
        return {"bytes": 8.0 * (L * n * n + (2 if case["lambda"] else 1) * (o * v) ** 2),
                "flops": its * (2.0 * o**2 * v**4 + 2.0 * L * v**4 + 4.0 * (o * v) ** 3)}
    cols = case.get("n_omega", 1) * case.get("n_orb", 1)
    if kind == "rhf":
        f = 2.0 * (6 * o**3 * v**2 + 2 * o**4 * v + 2 * o**2 * v * (v + o) + 2 * o**2 * v**2)
        return {"bytes": 8.0 * (3 * (o * v) ** 2 + o**4 + o**2 * v * (2 * v + 2 * o)), "flops": cols * ITERATIONS * f}
    if kind == "mor":
        m, n, pts = 2 * cols, o + o * (o - 1) // 2 * v, case["points"]
        return {"bytes": 16.0 * m * n + 16.0 * pts * case["n_orb"] ** 2,
                "flops": pts * (8.0 / 3 * m**3 + case["n_orb"] * 8.0 * m * n)}
    sectors = case["sectors"].split("+")
    if kind == "sigma":
        k = case["n_vec"]
        return {"bytes": _operator_bytes(o, v, sectors) + 32.0 * k * _dim(case),
                "flops": k * _sigma_flops(o, v, case["sectors"])}
    flops = cols * ITERATIONS * sum(_sigma_flops(o, v, s) for s in sectors)
    nbytes = _operator_bytes(o, v, sectors) + 16.0 * case["n_omega"] * case["n_orb"] ** 2
    if kind == "setup":
        n = o + v
        flops += _setup_flops(o, v, L, sectors)
        nbytes += 8.0 * (L * n * n + (o * v) ** 2)
    return {"bytes": nbytes, "flops": flops}


# Largest relative difference of G (amplitudes, gradients) to the 64-bit values seen on the listed and drawn
# cases, times about four: iterative solutions stop at relative residuals of 1e-8.
def tolerance(case):
    return {"sigma": {"rel": 2e-15, "max": 2e-14}, "mlp": {"rel": 1e-6, "max": 4e-5}, "mor": {"rel": 2.5e-4, "max": 2.5e-3},
            "ccsd": {"rel": 4e-6, "max": 4e-5}}.get(case["kind"], {"rel": 4e-8, "max": 4e-7})


# ------------------------------------------------------------------------------------------- 64-bit values
def _es(spec, *xs):
    return torch.einsum(spec, *xs)


class _Rotated:
    """T1-rotated Cholesky vectors and Fock matrix; `spin` sums each closed-shell pair twice."""

    def __init__(self, fock, chol, t1, pairs=1.0):
        self.o, self.v = t1.shape
        o, n = self.o, sum(t1.shape)
        X, Y = torch.eye(n, dtype=F64, device=t1.device), torch.eye(n, dtype=F64, device=t1.device)
        X = X - torch.nn.functional.pad(t1.T, (0, self.v, o, 0))
        Y = Y + torch.nn.functional.pad(t1.T, (0, self.v, o, 0))

        def mean_field(C):
            J = _es("kpq,k->pq", C, C[:, :o, :o].diagonal(dim1=1, dim2=2).sum(1))
            return pairs * J - _es("kpj,kjq->pq", C[:, :, :o], C[:, :o, :])

        self.C = X @ chol @ Y
        self.f = X @ (fock - mean_field(chol)) @ Y + mean_field(self.C)

    def block(self, p, r):
        s = {"o": slice(0, self.o), "v": slice(self.o, None)}
        return self.C[:, s[p], s[r]]

    def coulomb(self, blk):
        """(pr|qs) as [p][q][r][s]."""
        p, q, r, s = blk
        return _es("kpr,kqs->pqrs", self.block(p, r), self.block(q, s))

    def eri(self, blk):
        p, q, r, s = blk
        return self.coulomb(blk) - self.coulomb(p + q + s + r).transpose(2, 3)

    def fock(self, blk):
        s = {"o": slice(0, self.o), "v": slice(self.o, None)}
        return self.f[s[blk[0]], s[blk[1]]]


class _Sector:
    """One sector of the spin-orbital problem on unpacked vectors [one | two], rows of a batch."""

    def __init__(self, rot, t1, t2, ip):
        o, v = t1.shape
        self.o, self.v, self.ip, self.t1, self.t2 = o, v, ip, t1, t2
        g = rot.eri("oovv")
        self.g, self.Fov = g, rot.fock("ov")
        self.Foo = rot.fock("oo") + 0.5 * _es("mnef,inef->mi", g, t2)
        self.Fvv = rot.fock("vv") - 0.5 * _es("mnef,mnaf->ae", g, t2)
        self.ring = rot.eri("ovvo") - _es("mnef,jnfb->mbej", g, t2)
        if ip:
            self.ooov = rot.eri("ooov")
            self.oooo = rot.eri("oooo") + 0.5 * _es("mnef,ijef->mnij", g, t2)
            x = _es("mnie,jnbe->mbij", self.ooov, t2)
            self.ovoo = rot.eri("ovoo") - _es("me,ijbe->mbij", self.Fov, t2) + x - x.transpose(2, 3)
            for m in range(o):      # one row of <mb||ef> at a time
                C = rot.C[:, m, o:]
                w = _es("ke,kbf->bef", C, rot.block("v", "v"))
                self.ovoo[m] += 0.5 * _es("bef,ijef->bij", w - w.transpose(1, 2), t2)
            shape = (o, o, v)
            d1 = -self.Foo.diagonal()
            d2 = self.Fvv.diagonal()[None, None, :] + d1[:, None, None] + d1[None, :, None]
        else:
            self.vovv = rot.eri("vovv")
            self.vvvv = rot.eri("vvvv") + 0.5 * _es("mnef,mnab->abef", g, t2)
            x = _es("mbef,miaf->abei", rot.eri("ovvv"), t2)
            self.vvvo = (rot.eri("vvvo") - _es("me,miab->abei", self.Fov, t2)
                         + 0.5 * _es("mnei,mnab->abei", rot.eri("oovo"), t2) - x + x.transpose(0, 1))
            shape = (o, v, v)
            d1 = self.Fvv.diagonal()
            d2 = d1[None, :, None] + d1[None, None, :] - self.Foo.diagonal()[:, None, None]
        self.shape, self.n1, self.diag = shape, d1.numel(), torch.cat([d1, d2.reshape(-1)])

    def split(self, x):
        return x[:, :self.n1], x[:, self.n1:].reshape(-1, *self.shape)

    def real_sigma(self, x):
        a, b = self.split(x)
        if self.ip:
            s1 = -a @ self.Foo - _es("me,cmie->ci", self.Fov, b) + 0.5 * _es("nmie,cmne->ci", self.ooov, b)
            y = _es("maei,cmje->cija", self.ring, b) - _es("mi,cmja->cija", self.Foo, b)
            z = 0.5 * _es("mnef,cmnf->ce", self.g, b)
            s2 = (_es("maji,cm->cija", self.ovoo, a) + b @ self.Fvv.T + y - y.transpose(1, 2)
                  + 0.5 * _es("mnij,cmna->cija", self.oooo, b) + _es("ce,ijae->cija", z, self.t2))
        else:
            s1 = a @ self.Fvv.T + _es("me,cmae->ca", self.Fov, b) + 0.5 * _es("amef,cmef->ca", self.vovv, b)
            y = b @ self.Fvv.T + _es("mbei,cmae->ciab", self.ring, b)
            z = 0.5 * _es("mnef,cnef->cm", self.g, b)
            s2 = (_es("abei,ce->ciab", self.vvvo, a) - _es("mi,cmab->ciab", self.Foo, b) + y - y.transpose(2, 3)
                  + 0.5 * _es("abef,cief->ciab", self.vvvv, b) - _es("cm,miab->ciab", z, self.t2))
        return torch.cat([s1, s2.reshape(len(x), -1)], 1)

    def sigma(self, x):
        r = self.real_sigma(torch.cat([x.real, x.imag]))
        return torch.complex(r[:len(x)], r[len(x):])

    def rhs(self, orbs):
        o, v, rows = self.o, self.v, []
        for p in orbs:
            a = torch.zeros(self.n1, dtype=F64, device=self.t1.device)
            b = torch.zeros(self.shape, dtype=F64, device=self.t1.device)
            if self.ip and p < o:
                a[p] = 1
            elif self.ip:
                a, b = self.t1[:, p - o], self.t2[:, :, p - o]
            elif p >= o:
                a[p - o] = 1
            else:
                a, b = -self.t1[p], -self.t2[p]
            rows.append(torch.cat([a, b.reshape(-1)]))
        return torch.stack(rows)

    def left(self, orbs):
        """Left vectors with Lambda = T^dagger, weighted for the dot product over unpacked pairs."""
        o, v, t1, t2, rows = self.o, self.v, self.t1, self.t2, []
        for q in orbs:
            b = torch.zeros(self.shape, dtype=F64, device=t1.device)
            if self.ip and q >= o:
                a, b = t1[:, q - o], t2[:, :, q - o]
            elif self.ip:
                a = -t1 @ t1[q] - 0.5 * _es("lcd,klcd->k", t2[q], t2)
                a[q] += 1
                b[q] += t1
                b[:, q] -= t1
                b = b - _es("c,ijca->ija", t1[q], t2)
            elif q < o:
                a, b = -t1[q], t2[:, q]
            else:
                e = q - o
                a = -t1[:, e] @ t1 + 0.5 * _es("kld,kldc->c", t2[:, :, e], t2)
                a[e] += 1
                b[:, e] += t1
                b[:, :, e] -= t1
                b = b + _es("k,ikcd->icd", t1[:, e], t2)
            rows.append(torch.cat([a, 0.5 * b.reshape(-1)]))
        return torch.stack(rows)

    def solve(self, omegas, eta, orbs):
        """Solutions [frequency][orbital][unpacked]."""
        z = torch.as_tensor(np.repeat(omegas, len(orbs)), dtype=F64, device=DEV)
        sign = 1.0 if self.ip else -1.0
        z = torch.complex(z, torch.full_like(z, -sign * eta))[:, None]
        b = self.rhs(orbs).to(C128).repeat(len(omegas), 1)
        x = _gmres(lambda x: z * x + sign * self.sigma(x), b, z + sign * self.diag)
        return x.reshape(len(omegas), len(orbs), -1)


class _NotSolved(Exception):
    """The 64-bit solution was not reached within its iterations."""


def _gmres(apply, b, D, tol=3e-12, m=120):
    """Independent right-preconditioned GMRES(m) solves, one for each row of b."""
    x, bn = torch.zeros_like(b), b.norm(dim=1)
    for cycle in range(5):
        r = b - apply(x)
        beta = r.norm(dim=1)
        if bool((beta <= tol * bn).all()):
            break
        if cycle == 4:
            if bool((beta > 1e-10 * bn).any()):
                raise _NotSolved
            break
        V = torch.zeros(m + 1, *b.shape, dtype=C128, device=b.device)
        H = torch.zeros(len(b), m + 1, m, dtype=C128, device=b.device)
        V[0] = r / beta.clamp_min(1e-300)[:, None]
        e1 = torch.zeros(len(b), m + 1, 1, dtype=C128, device=b.device)
        e1[:, 0, 0] = beta.to(C128)
        k = 0
        while k < m:
            w = apply(V[k] / D)
            for _ in range(2):
                h = _es("jbn,bn->bj", V[:k + 1].conj(), w)
                w = w - _es("jbn,bj->bn", V[:k + 1], h)
                H[:, :k + 1, k] += h
            nw = w.norm(dim=1)
            H[:, k + 1, k] = nw
            V[k + 1] = torch.where((nw > 1e-13)[:, None], w / nw.clamp_min(1e-300)[:, None], 0)
            k += 1
            if k % 5 == 0 or k == m:
                Q, R = torch.linalg.qr(H[:, :k + 1, :k], mode="complete")
                if bool(((Q.mH @ e1[:, :k + 1])[:, k, 0].abs() <= tol * bn).all()):
                    break
        y = torch.linalg.pinv(H[:, :k + 1, :k], rtol=1e-15) @ e1[:, :k + 1]
        x = x + _es("jbn,bj->bn", V[:k], y[:, :, 0]) / D
    return x


def _tensors(p):
    return [torch.as_tensor(x, device=DEV) for x in (p.fock, p.chol, p.t1, p.t2)]


def _green(p, case, sectors, omegas, orbs):
    fock, chol, t1, t2 = _tensors(p)
    rot = _Rotated(fock, chol, t1)
    G = 0
    for ip in (True, False):
        if ("IP" if ip else "EA") in sectors:
            s = _Sector(rot, t1, t2, ip)
            g = s.solve(omegas, case["eta"], orbs) @ s.left(orbs).to(C128).T
            G = G + (g if ip else g.transpose(1, 2))
    return G


class _ClosedShell:
    """The spin-summed ionisation operator on [r_i | r_ij^a]."""

    def __init__(self, p):
        fock, chol, t1, t2 = _tensors(p)
        self.o, self.v, self.t1, self.t2 = p.o, p.v, t1, t2
        rot = _Rotated(fock, chol, t1, 2.0)
        u = rot.coulomb("oovv")                                  # [m][n][e][f] = (me|nf)
        self.u2 = 2 * u - u.transpose(2, 3)
        self.Foo = rot.fock("oo") + _es("mnef,inef->mi", self.u2, t2)
        self.Fvv = rot.fock("vv") - _es("mnef,mnaf->ae", self.u2, t2)
        self.Fov = rot.fock("ov")
        self.oooo = rot.coulomb("oooo") + _es("mnef,ijef->mnij", u, t2)
        B = rot.coulomb("ooov")                                  # [m][n][i][e] = (mi|ne)
        c = rot.coulomb("oovo").permute(0, 3, 1, 2)              # [m][i][n][e] = (me|ni)
        self.W = B
        Bm = B.transpose(1, 2)                                   # [m][i][n][e]
        self.maij = (rot.coulomb("ovoo") + _es("me,ijea->maij", self.Fov, t2)
                     + _es("mine,jnae->maij", 2 * Bm - c, t2) - _es("mine,jnea->maij", Bm, t2)
                     - _es("mjne,inea->maij", c, t2))
        for m in range(p.o):
            self.maij[m] += _es("eaf,ijef->aij", _es("ke,kaf->eaf", rot.block("o", "v")[:, m], rot.block("v", "v")), t2)
        self.X = (rot.coulomb("ovvo") + _es("mnef,jnaf->maej", self.u2, t2) - _es("mnef,jnfa->maej", u, t2))
        self.Y = rot.coulomb("ovov") - _es("mnfe,infa->maie", u, t2)
        self.n1 = p.o
        d = self.Foo.diagonal()
        self.diag = torch.cat([-d, (self.Fvv.diagonal() - d[:, None, None] - d[None, :, None]).reshape(-1)])

    def sigma(self, x):
        x = torch.cat([x.real, x.imag])
        a, b = x[:, :self.o], x[:, self.o:].reshape(-1, self.o, self.o, self.v)
        s1 = (-a @ self.Foo + _es("me,cime->ci", self.Fov, 2 * b - b.transpose(1, 2))
              + _es("nmie,cmne->ci", self.W, b) - 2 * _es("mnie,cmne->ci", self.W, b))
        z = _es("mnef,cmnf->ce", self.u2, b)
        s2 = (-_es("maij,cm->cija", self.maij, a) + b @ self.Fvv.T - _es("mi,cmja->cija", self.Foo, b)
              - _es("mj,cima->cija", self.Foo, b) + _es("mnij,cmna->cija", self.oooo, b)
              - _es("maie,cmje->cija", self.Y, b) + 2 * _es("maej,cime->cija", self.X, b)
              - _es("maje,cime->cija", self.Y, b) - _es("maej,cmie->cija", self.X, b)
              - _es("ce,ijea->cija", z, self.t2))
        r = torch.cat([s1, s2.reshape(len(x), -1)], 1)
        return torch.complex(r[:len(x) // 2], r[len(x) // 2:])

    def green(self, omegas, eta, orbs):
        o, t1, t2, rhs, left = self.o, self.t1, self.t2, [], []
        for p in orbs:
            a = torch.zeros(o, dtype=F64, device=DEV)
            b = torch.zeros(o, o, self.v, dtype=F64, device=DEV)
            if p < o:
                a[p] = 1
                rhs.append(torch.cat([a, b.reshape(-1)]))
                a = a - t1 @ t1[p] - _es("lcd,ilcd->i", 2 * t2[p] - t2[p].transpose(1, 2), t2)
                b[p] += 2 * t1
                b[:, p] -= t1
                b = b - _es("c,ijca->ija", t1[p], 2 * t2 - t2.transpose(2, 3))
                left.append(torch.cat([a, b.reshape(-1)]))
            else:
                t = t2[:, :, p - o]
                rhs.append(torch.cat([t1[:, p - o], t.reshape(-1)]))
                left.append(torch.cat([t1[:, p - o], (2 * t - t2[:, :, :, p - o]).reshape(-1)]))
        z = torch.as_tensor(np.repeat(omegas, len(orbs)), dtype=F64, device=DEV)
        z = torch.complex(z, torch.full_like(z, -eta))[:, None]
        b = torch.stack(rhs).to(C128).repeat(len(omegas), 1)
        x = _gmres(lambda x: z * x + self.sigma(x), b, z + self.diag)
        return x.reshape(len(omegas), len(orbs), -1) @ torch.stack(left).to(C128).T


def _ccsd(p, want_lambda):
    """Converged amplitudes and energy; Lambda from the stationary point of E + Lambda Omega (its gradient with
    respect to T by automatic differentiation)."""
    fock, chol = (torch.as_tensor(x, device=DEV) for x in (p.fock, p.chol))
    o, v = p.o, p.v
    e = fock.diagonal()
    D1 = e[:o, None] - e[None, o:]
    D2 = D1[:, None, :, None] + D1[None, :, None, :]
    g0 = _Rotated(fock, chol, torch.zeros(o, v, dtype=F64, device=DEV)).eri("oovv")

    def energy(t1, t2):
        return (fock[:o, o:] * t1).sum() + (g0 * (0.25 * t2 + 0.5 * _es("ia,jb->ijab", t1, t1))).sum()

    def residual(t1, t2):
        r = _Rotated(fock, chol, t1)
        g = r.eri("oovv")
        Fvv = r.fock("vv") - 0.5 * _es("mnef,mnbf->be", g, t2)
        Foo = r.fock("oo") + 0.5 * _es("mnef,jnef->mj", g, t2)
        oooo = r.eri("oooo") + 0.5 * _es("mnef,ijef->mnij", g, t2)
        ring = r.eri("ovvo") - 0.5 * _es("mnef,jnfb->mbej", g, t2)
        r1 = (r.fock("vo").T + _es("me,imae->ia", r.fock("ov"), t2)
              + 0.5 * _es("amef,imef->ia", r.eri("vovv"), t2) + 0.5 * _es("mnei,mnae->ia", r.eri("oovo"), t2))
        x = _es("mbej,imae->ijab", ring, t2)
        y, w = _es("be,ijae->ijab", Fvv, t2), _es("mj,imab->ijab", Foo, t2)
        r2 = (r.eri("vvoo").permute(2, 3, 0, 1) + y - y.transpose(2, 3) - w + w.transpose(0, 1)
              + 0.5 * _es("mnij,mnab->ijab", oooo, t2) + 0.5 * _es("abef,ijef->ijab", r.eri("vvvv"), t2)
              + x - x.transpose(0, 1) - x.transpose(2, 3) + x.transpose(0, 1).transpose(2, 3))
        return r1, r2

    def converge(x, step):
        xs, es = [], []
        for _ in range(100):
            r = step(x)
            if float(r[0].abs().max()) < 1e-12 and float(r[1].abs().max()) < 1e-12:
                break
            d = torch.cat([(r[0] / D1).reshape(-1), (r[1] / D2).reshape(-1)])
            xs, es = (xs + [torch.cat([t.reshape(-1) for t in x]) + d])[-8:], (es + [d])[-8:]
            k = len(es)
            A = torch.full((k + 1, k + 1), -1.0, dtype=F64, device=DEV)
            A[k, k] = 0
            E = torch.stack(es)
            A[:k, :k] = E @ E.T
            scale = A[k - 1, k - 1].clone()
            A[:k, :k] /= scale
            b = torch.zeros(k + 1, dtype=F64, device=DEV)
            b[k] = -1
            c = torch.linalg.lstsq(A.cpu(), b.cpu()[:, None], driver="gelsd").solution[:k, 0].to(DEV)
            flat = (c[:, None] * torch.stack(xs)).sum(0)
            x = (flat[:o * v].reshape(o, v), flat[o * v:].reshape(o, o, v, v))
        return x

    zero = (torch.zeros(o, v, dtype=F64, device=DEV), torch.zeros(o, o, v, v, dtype=F64, device=DEV))
    t1, t2 = converge(zero, lambda x: residual(*x))
    out = {"t1": t1, "t2": t2, "e_corr": float(energy(t1, t2)), "code": None}
    if want_lambda:
        a1, a2 = t1.clone().requires_grad_(), t2.clone().requires_grad_()
        r1, r2 = residual(a1, a2)
        en = energy(a1, a2)

        def step(l):
            g1, g2 = torch.autograd.grad([en, r1, r2], [a1, a2], [torch.ones_like(en), l[0], 0.25 * l[1]],
                                         retain_graph=True)
            return g1, 2.0 * _antisym(g2)           # derivative for one independent element, all four images

        out["l1"], out["l2"] = converge((t1, t2), step)
    return out


def _mor(p, case, seed, orbs):
    fock, chol, t1, t2 = _tensors(p)
    s = _Sector(_Rotated(fock, chol, t1), t1, t2, True)
    w = torch.cat([torch.ones(s.n1, device=DEV, dtype=F64), torch.full((s.diag.numel() - s.n1,), math.sqrt(0.5),
                                                                       device=DEV, dtype=F64)])
    x = s.solve(_omegas(case, seed), case["eta"], orbs).reshape(-1, s.diag.numel()) * w
    S = torch.linalg.qr(torch.cat([x.real, x.imag]).T)[0]       # orthonormal over the packed coordinates
    W = (s.real_sigma((S.T / w)) * w).T
    b, c = (s.rhs(orbs) * w).T, (s.left(orbs) / w).T
    H, bh, ch = (S.T @ W).to(C128), (S.T @ b).to(C128), (S.T @ c).to(C128)
    G, rr = [], []
    for om in _omegas(case, seed, case["points"]):
        z = complex(om, -case["eta"])
        y = torch.linalg.solve(z * torch.eye(len(H), dtype=C128, device=DEV) + H, bh)
        G.append(y.T @ ch)
        res = b - z * (S.to(C128) @ y) - W.to(C128) @ y
        rr.append(res.norm(dim=0) / b.norm(dim=0))
    return torch.stack(G), torch.stack(rr)


def _mlp(case, seed):
    w, F, gram = _mlp_inputs(case, seed)
    h = case["hidden"]
    w, F, gram = (torch.as_tensor(x, device=DEV) for x in (w, F, gram))
    w.requires_grad_()
    sizes = [h * 27, h, h * h, h, 16 * h, 16, 27, 27]
    W1, b1, W2, b2, W3, b3, mu, sd = torch.split(w, sizes)
    x = torch.relu((F - mu.detach()) / sd.detach() @ W1.reshape(h, 27).T + b1)
    y = torch.relu(x @ W2.reshape(h, h).T + b2) @ W3.reshape(16, h).T + b3
    c = torch.complex(y[:, 0::2], y[:, 1::2])
    a = torch.cat([c.sum(1, keepdim=True) - 1, c], 1)
    loss = (_es("si,sij,sj->s", a.conj(), gram, a).real / gram[:, 0, 0].real).mean()
    g, = torch.autograd.grad(loss, w)
    return float(loss.detach()), g


def _np(x):
    if isinstance(x, (list, tuple)):
        return type(x)(_np(y) for y in x)
    if isinstance(x, dict):
        return {k: _np(y) for k, y in x.items()}
    return x.detach().cpu().numpy() if isinstance(x, torch.Tensor) else x


def exact(case, seed):
    try:
        return _exact(case, seed)
    except _NotSolved:
        return None


def _exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _np(_mlp(case, seed))
    if kind == "batch":
        ps = [_problem(*m, seed) for m in _molecules(case)]
        return [_np(_green(p, case, ["IP"], _omegas(case, seed), _orbitals(p, case))) for p in ps], None
    # FP64 units give about 1 TFLOP/s, and several times the stated work is done here
    if work(case)["flops"] > 4e12:
        return None
    p = _problem(case["o"], case["v"], case["L"], seed, {"ccsd": "bare", "rhf": "closed"}.get(kind, "spin"))
    if kind == "ccsd":
        return _np(_ccsd(p, case["lambda"]))
    if kind == "sigma":
        fock, chol, t1, t2 = _tensors(p)
        s = _Sector(_Rotated(fock, chol, t1), t1, t2, case["sectors"] == "IP")
        n1, size = s.n1, p.o if case["sectors"] == "IP" else p.v
        i, j = torch.triu_indices(size, size, 1, device=DEV)
        x = torch.as_tensor(_vectors(case, seed), device=DEV)
        full = torch.zeros(len(x), *s.shape, dtype=C128, device=DEV)
        if s.ip:
            packed = x[:, n1:].reshape(len(x), -1, p.v)
            full[:, i, j], full[:, j, i] = packed, -packed
        else:
            packed = x[:, n1:].reshape(len(x), p.o, -1)
            full[:, :, i, j], full[:, :, j, i] = packed, -packed
        a, b = s.split(s.sigma(torch.cat([x[:, :n1], full.reshape(len(x), -1)], 1)))
        b = b[:, i, j] if s.ip else b[:, :, i, j]
        return _np(torch.cat([a, b.reshape(len(x), -1)], 1))
    orbs = _orbitals(p, case)
    if kind == "mor":
        return _np(_mor(p, case, seed, orbs))
    omegas = _omegas(case, seed)
    if kind == "rhf":
        return _np(_ClosedShell(p).green(omegas, case["eta"], orbs)), None
    return _np(_green(p, case, case["sectors"].split("+"), omegas, orbs)), None
