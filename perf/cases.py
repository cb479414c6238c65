"""Performance cases: the calls a user of this package makes, over the sizes it serves.

Each case is a dict of plain values.  ``prepare`` makes what a program holds before the call
(the model handle, its tables and the input vectors), ``run`` makes one call (or the few calls
that belong together) through the package's public entry points, ``work`` counts the bytes and
operations such a call cannot do without, and ``exact`` computes the same outputs in 64-bit
torch operations that share no code with the package: hops as gathers, one bond at a time.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1307_7542_gb300 import hub
from paper_1307_7542_gb300 import workloads as W

DEV = "cuda"


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # The package's smallest benchmark system, solved to the default tolerance with its
        # ground-state vector: an iteration is far shorter than a kernel launch.
        dict(name="ring8_ground", kind="ground", lattice="ring", M=8, n_up=4, n_dn=4, U=4.0, t=1.0),
        # One product of the same system: the smallest call of the package, all latency.
        dict(name="ring8_apply", kind="apply", lattice="ring", M=8, n_up=4, n_dn=4, U=4.0, t=1.0, vector="normal"),
        # An ordinary ground state: a 12-site ring at half filling (0.85 M states).
        dict(name="ring12_ground", kind="ground", lattice="ring", M=12, n_up=6, n_dn=6, U=4.0, t=1.0),
        # Green's function of the 12-site ring: both start vectors from the ground state, and
        # the coefficients of both continued fractions (two rectangular sectors).
        dict(name="ring12_green", kind="green", lattice="ring", M=12, n_up=6, n_dn=6, U=4.0, t=1.0, steps=32, site=0,
             spin=0),
        # The benchmark lattice: one product, FP64 vectors on the device (165.6 M states).
        dict(name="square4x4_apply", kind="apply", lattice="square4x4", M=16, n_up=8, n_dn=8, U=4.0, t=1.0,
             vector="normal"),
        # The benchmark's Lanczos steps on the same lattice: a fixed number from a given vector.
        dict(name="square4x4_lanczos", kind="lanczos", lattice="square4x4", M=16, n_up=8, n_dn=8, U=4.0, t=1.0,
             steps=12, psi=False),
        # 18 sites: 48620 spin-up strings against 816 spin-down ones, long rows, few of them.
        dict(name="square3x6_apply", kind="apply", lattice="square3x6", M=18, n_up=9, n_dn=3, U=4.0, t=1.0,
             vector="normal"),
        # Disordered 3x4 lattice (every t, U and site energy its own): ground-state energy and
        # its 41 derivatives, forward and backward through autograd.
        dict(name="disordered3x4_energy_grad", kind="energy_grad", lattice="disordered3x4", M=12, n_up=6, n_dn=6),
        # The same lattice: a differentiable product, forward and backward.
        dict(name="disordered3x4_vjp", kind="vjp", lattice="disordered3x4", M=12, n_up=6, n_dn=6),
        # An impurity solver's batch: all 81 sectors of the 8-site star for 64 parameter sets.
        dict(name="aim_batch", kind="batch", lattice="star", M=8, sets=64),
        # The benchmark lattice in the zero-momentum sector of its two translations (10.6 M
        # entries): Lanczos steps and the vector they give.
        dict(name="torus4x4_momentum", kind="momentum", lattice="square4x4", M=16, n_up=8, n_dn=8, U=4.0, t=1.0,
             chi0=1, chi1=1, steps=16, psi=True),
        # A product on host buffers (page-locked numpy-style vectors in and out).
        dict(name="square4x4_host", kind="host", lattice="square4x4", M=16, n_up=6, n_dn=6, U=4.0, t=1.0),
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "lanczos", "lanczos", "ground", "green", "momentum", "energy_grad",
                       "vjp", "batch", "host"])
    U = rng.choice([0.0, 1.0, 2.0, 4.0, 8.0, round(rng.uniform(0.5, 12.0), 3)])
    t = rng.choice([1.0, 1.0, 1.0, -1.0, round(rng.uniform(0.3, 2.5), 3)])
    if kind in ("energy_grad", "vjp"):
        return dict(kind=kind, lattice="disordered3x4", M=12, n_up=rng.randint(4, 7), n_dn=rng.randint(3, 7),
                    draw=rng.randrange(1, 1000))
    if kind == "batch":
        return dict(kind=kind, lattice="star", M=rng.choice([5, 6, 7, 8]), sets=rng.randint(1, 64))
    if kind == "momentum":
        lattice, M = rng.choice([("ring", 10), ("ring", 12), ("ring", 14), ("ring", 16), ("square3x4", 12),
                                 ("square4x4", 16)])
        n = M // 2 - (rng.randint(1, 2) if lattice == "square4x4" else rng.randint(0, 2))
        return dict(kind=kind, lattice=lattice, M=M, n_up=n, n_dn=n - rng.randint(0, 1), U=U, t=t, chi0=1, chi1=1,
                    steps=rng.randint(1, 16), psi=rng.random() < 0.5)
    # a size between a few thousand and 10^8 states, spread over its logarithm: the sector of
    # the right size nearest the target among the package's lattices
    top = {"apply": 1.5e8, "lanczos": 1.2e8, "ground": 9e5, "green": 5e6, "host": 5e7}[kind]
    low = 3e3 if kind in ("apply", "ground") else (3e4 if kind == "host" else 3e5)
    target = math.exp(rng.uniform(math.log(low), math.log(top)))
    best = []
    for lattice, M in (("ring", 8), ("ring", 9), ("ring", 10), ("ring", 11), ("ring", 12), ("ring", 13), ("ring", 14),
                       ("ring", 16), ("square3x4", 12), ("square3x4open", 12), ("square4x4", 16), ("square3x6", 18)):
        for nu in range(1, M):
            for nd in range(1, M):
                d = math.comb(M, nu) * math.comb(M, nd)
                if 0.6 * target < d < min(1.4 * target, top):
                    best.append((lattice, M, nu, nd))
    lattice, M, nu, nd = rng.choice(best)
    c = dict(kind=kind, lattice=lattice, M=M, n_up=nu, n_dn=nd, U=U, t=t)
    if kind == "apply":
        c["vector"] = rng.choice(["normal", "normal", "ground"]) if target < 2e7 else "normal"
    if kind == "lanczos":
        c.update(steps=rng.randint(1, 12), psi=rng.random() < 0.4)
    if kind == "green":
        c.update(steps=rng.randint(8, 24), site=rng.randrange(M), spin=rng.randrange(2))
    return c


# ------------------------------------------------------------------- inputs, from the seed

def _bonds(case):
    lat, M = case["lattice"], case["M"]
    if lat == "ring":
        return W.ring_bonds(M)
    if lat == "star":
        return W.star_bonds(M - 1)
    size = lat[len("square"):] if lat.startswith("square") else "3x4open"
    return W.square_bonds(int(size[0]), int(size[2]), periodic=not size.endswith("open"))


def _params(case, seed):
    """(bonds, t, U, eps) of a case."""
    b, M = _bonds(case), case["M"]
    if case["lattice"] == "disordered3x4":
        w = W.disordered3x4(3 * (seed + case.get("draw", 0)))
        return b, w["t"], w["U"], w["eps"]
    return b, np.full(len(b), case["t"]), np.full(M, case["U"]), np.zeros(M)


def _normal(seed, n, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000 * seed + salt)
    return torch.randn(n, dtype=torch.float64, device=DEV, generator=g)


def _star_sets(case, seed):
    """Parameter sets and jobs of the impurity star: every sector of every set."""
    ps = [W.aim_star(p, n_bath=case["M"] - 1, seed=seed + 1) for p in range(case["sets"])]
    t, U, eps = (np.stack([p[k] for p in ps]) for k in ("t", "U", "eps"))
    sectors = [(a, b) for a in range(case["M"] + 1) for b in range(case["M"] + 1)]
    jobs = [(a, b, p) for p in range(case["sets"]) for a, b in sectors]
    nu, nd, jp = (np.array([j[k] for j in jobs], dtype=np.int32) for k in range(3))
    return t, U, eps, sectors, nu, nd, jp


def _translations(case):
    """Site permutations of the case's lattice: T of the ring, or both translations of the torus."""
    M = case["M"]
    if case["lattice"] == "ring":
        return np.array([[(i + M - 1) % M for i in range(M)]], dtype=np.int32), [case["chi0"]]
    Lx, Ly = int(case["lattice"][6]), int(case["lattice"][8])
    px = [(s % Lx + 1) % Lx + Lx * (s // Lx) for s in range(M)]
    py = [s % Lx + Lx * ((s // Lx + 1) % Ly) for s in range(M)]
    return np.array([px, py], dtype=np.int32), [case["chi0"], case["chi1"]]


def _start_vector(case, seed, ref=None):
    """The vector a case's call starts from: random normal numbers, or an approximate ground
    state (a short Lanczos run from random numbers: entries over many orders of magnitude)."""
    D = math.comb(case["M"], case["n_up"]) * math.comb(case["M"], case["n_dn"])
    x = _normal(seed, D)
    if case.get("vector") == "ground" or case["kind"] == "green":
        r = ref or Reference(case["M"], case["n_up"], case["n_dn"], *_params(case, seed))
        x = r.lanczos(x, 40, psi=True)[2]
    return x


def prepare(case, seed):
    kind, M = case["kind"], case["M"]
    if kind == "batch":
        t, U, eps, _, nu, nd, jp = _star_sets(case, seed)
        return dict(case=case, bonds=_bonds(case), t=t, U=U, eps=eps, nu=nu, nd=nd, jp=jp)
    b, t, U, eps = _params(case, seed)
    m = hub.Hubbard(M, case["n_up"], case["n_dn"], b, t, U, eps)
    s = dict(case=case, m=m)
    if kind == "momentum":
        perms, chars = _translations(case)
        m.set_translations(perms, chars)
        s["x"] = _normal(seed, m.D)
    elif kind == "host":
        s["x"] = _normal(seed, m.D).cpu().pin_memory()
        s["y"] = torch.empty(m.D, dtype=torch.float64, pin_memory=True)
    else:
        s["x"] = _start_vector(case, seed)
    if kind == "apply":
        s["y"] = torch.empty_like(s["x"])
    if kind == "green":
        d = (1, 0) if case["spin"] == 0 else (0, 1)
        for key, sg in (("plus", 1), ("minus", -1)):
            s[key] = hub.Hubbard(M, case["n_up"] + sg * d[0], case["n_dn"] + sg * d[1], b, t, U, eps)
            s["v_" + key] = torch.empty(s[key].D, dtype=torch.float64, device=DEV)
    if kind in ("vjp", "energy_grad"):
        s["theta"] = [torch.tensor(p, dtype=torch.float64) for p in (t, U, eps)]
    if kind == "vjp":
        s["ybar"] = _normal(seed, m.D, salt=1)
    return s


# -------------------------------------------------------------------------------- one pass

def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "batch":
        return dict(E0=hub.hub_batch_ground(c["M"], s["bonds"], s["t"], s["U"], s["eps"], s["nu"], s["nd"], s["jp"])[0])
    m = s["m"]
    if kind == "apply":
        return m.apply(s["x"], s["y"])
    if kind == "host":
        return m.apply_host(s["x"], s["y"])
    if kind == "ground":
        r = m.ground(s["x"], want_psi=True)
        return dict(E0=np.float64(r["E0"]), psi=r["psi"])
    if kind in ("lanczos", "momentum"):
        r = m.ground(s["x"], maxit=c["steps"], tol=0.0, want_psi=c["psi"])
        a, b = hub.hub_lanczos_coeffs(m.h, cap=c["steps"])
        return dict(E0=np.float64(r["E0"]), alpha=a, beta=b, psi=r["psi"])
    if kind == "green":
        out = {}
        for key, create in (("plus", True), ("minus", False)):
            hub.hub_ladder(m.h, s[key].h, c["site"], c["spin"], create, s["x"], s["v_" + key])
            a, b, n2 = hub.hub_green_coeffs(s[key].h, s["v_" + key], c["steps"])
            out[key] = dict(v=s["v_" + key], alpha=a, beta=b, norm2=n2)
        return out
    th = [p.clone().requires_grad_(True) for p in s["theta"]]
    if kind == "energy_grad":
        E = hub.ground_energy(m, *th, x0=s["x"])
        E.backward()
        return dict(E=E.detach(), dt=th[0].grad, dU=th[1].grad, deps=th[2].grad)
    x = s["x"].detach().requires_grad_(True)
    y = hub.apply_fn(m, x, *th)
    y.backward(s["ybar"])
    return dict(y=y.detach(), dx=x.grad, dt=th[0].grad, dU=th[1].grad, deps=th[2].grad)


# ------------------------------------------------------------- what a pass cannot do without

def _size(case):
    """(states, multiply-adds of one product)."""
    M, nu, nd = case["M"], case["n_up"], case["n_dn"]
    nb = len(_bonds(case))
    cu, cd = math.comb(M, nu), math.comb(M, nd)

    def nnz(n):
        return 2 * nb * math.comb(M - 2, n - 1) if 0 < n < M else 0
    return cu * cd, nnz(nu) * cd + nnz(nd) * cu + cu * cd


def work(case):
    """Bytes: a product reads x and writes y once (8 bytes an entry each); a Lanczos step cannot
    keep its vectors on the chip, so it reads two and writes one; a gradient reads its vectors
    once.  Operations: two per multiply-add of the product, six per entry of a Lanczos step.
    Ground states to a tolerance count 50 steps (the order of what they take)."""
    kind = case["kind"]
    if kind == "batch":
        by = fl = 0.0
        for a in range(case["M"] + 1):
            for b in range(case["M"] + 1):
                D, mac = _size(dict(case, n_up=a, n_dn=b))
                by += 8.0 * case["sets"]
                fl += case["sets"] * min(D, 30) * (2.0 * mac + 6.0 * D)
        return dict(bytes=by, flops=fl)
    D, mac = _size(case)
    if kind == "green":
        d = (1, 0) if case["spin"] == 0 else (0, 1)
        by, fl = 16.0 * D, 0.0
        for sg in (1, -1):
            D2, mac2 = _size(dict(case, n_up=case["n_up"] + sg * d[0], n_dn=case["n_dn"] + sg * d[1]))
            by += case["steps"] * 24.0 * D2
            fl += case["steps"] * (2.0 * mac2 + 6.0 * D2)
        return dict(bytes=by, flops=fl)
    if kind == "momentum":
        g = case["M"]
        D, mac = D / g, mac / g
    if kind in ("apply", "host"):
        return dict(bytes=16.0 * D, flops=2.0 * mac)
    if kind == "vjp":
        return dict(bytes=32.0 * D, flops=6.0 * mac)
    steps = case.get("steps", 50)
    passes = 2 if kind in ("ground", "energy_grad") or case.get("psi") else 1
    return dict(bytes=passes * steps * 24.0 * D, flops=passes * steps * (2.0 * mac + 6.0 * D))


# ------------------------------------------------------- the same in plain 64-bit arithmetic

class Reference:
    """H on a sector as gathers in torch FP64: vectors are count_dn x count_up matrices of the
    ascending spin strings, site i is bit i, hops carry the sign of the electrons between."""

    def __init__(self, M, n_up, n_dn, bonds, t, U, eps):
        self.M, self.bonds = M, np.asarray(bonds).reshape(-1, 2)
        self.t, self.U, self.eps = (np.asarray(v, dtype=np.float64) for v in (t, U, eps))
        self.s = [self._strings(M, n) for n in (n_up, n_dn)]
        self.shape = (len(self.s[1]), len(self.s[0]))
        self.hops = [self._hops(s) for s in self.s]
        self.bits = [torch.tensor((s[:, None] >> np.arange(M)) & 1, dtype=torch.float64, device=DEV) for s in self.s]

    @staticmethod
    def _strings(M, n):
        v = np.arange(1 << M, dtype=np.int64)
        return v[sum((v >> i) & 1 for i in range(M)) == n]

    def _hops(self, s):
        """Per bond: target rows, source rows and the signed element of dH/d(-t)."""
        out = []
        for i, j in self.bonds:
            lo, hi = min(int(i), int(j)), max(int(i), int(j))
            ok = np.nonzero(((s >> lo) ^ (s >> hi)) & 1)[0]
            src = np.searchsorted(s, s[ok] ^ ((1 << lo) | (1 << hi)))
            between = (s[ok] >> (lo + 1)) & ((1 << (hi - lo - 1)) - 1)
            par = sum((between >> k) & 1 for k in range(self.M)) & 1
            out.append((torch.tensor(ok, device=DEV), torch.tensor(src, device=DEV),
                        torch.tensor(1.0 - 2.0 * par, device=DEV)))
        return out

    def diag(self):
        d = (self.bits[1] * torch.tensor(self.U, device=DEV)) @ self.bits[0].T
        e = [b @ torch.tensor(self.eps, device=DEV) for b in self.bits]
        return d + e[0][None, :] + e[1][:, None]

    def apply(self, x):
        X = x.view(self.shape)
        Y = self.diag() * X
        for b, tb in enumerate(self.t):
            dst, src, sg = self.hops[0][b]
            if len(dst):
                Y.index_add_(1, dst, X.index_select(1, src) * (-tb * sg)[None, :])
            dst, src, sg = self.hops[1][b]
            if len(dst):
                Y.index_add_(0, dst, X.index_select(0, src) * (-tb * sg)[:, None])
        return Y.reshape(-1)

    def lanczos(self, x0, steps, psi=False):
        """alpha, beta and, for the lowest eigenvector of T, the vector it stands for."""
        al, be = [], []
        q, qp, Q = x0 / x0.norm(), None, []
        for _ in range(steps):
            if psi:
                Q.append(q)
            w = self.apply(q)
            if qp is not None:
                w -= be[-1] * qp
            a = torch.dot(q, w)
            w -= a * q
            b = w.norm()
            al.append(float(a))
            be.append(float(b))
            if be[-1] <= 1e-12 * max(1.0, abs(al[-1])):
                break
            qp, q = q, w / b
        T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
        ev, vec = np.linalg.eigh(T)
        if not psi:
            return np.array(al), np.array(be), None, np.float64(ev[0])
        v = vec[:, 0] * (1.0 if vec[0, 0] > 0 else -1.0)
        p = sum(float(c) * u for c, u in zip(v, Q))
        return np.array(al), np.array(be), p / p.norm(), np.float64(ev[0])

    def ground(self, x0, steps=160):
        """Converged ground state (full re-orthogonalisation), its sign that of <x0, psi> > 0."""
        n = x0.numel()
        steps = min(steps, n)
        Q = torch.empty(steps, n, dtype=torch.float64, device=DEV)
        al, be = [], []
        q = x0 / x0.norm()
        for j in range(steps):
            Q[j] = q
            w = self.apply(q)
            al.append(float(torch.dot(q, w)))
            for _ in range(2):
                w -= Q[: j + 1].T @ (Q[: j + 1] @ w)
            b = float(w.norm())
            be.append(b)
            if b < 1e-9:
                break
            q = w / b
        k = len(al)
        ev, vec = np.linalg.eigh(np.diag(al) + np.diag(be[: k - 1], 1) + np.diag(be[: k - 1], -1))
        v = vec[:, 0] * (1.0 if vec[0, 0] > 0 else -1.0)
        p = torch.tensor(v, device=DEV) @ Q[:k]
        return np.float64(ev[0]), p / p.norm()

    def form(self, a, b):
        """a^T (dH/dtheta) b for every t, U and eps."""
        A, B = a.view(self.shape), b.view(self.shape)
        dt = np.empty(len(self.t))
        for k in range(len(self.t)):
            v = 0.0
            dst, src, sg = self.hops[0][k]
            if len(dst):
                v += float((A.index_select(1, dst) * B.index_select(1, src) * sg[None, :]).sum())
            dst, src, sg = self.hops[1][k]
            if len(dst):
                v += float((A.index_select(0, dst) * B.index_select(0, src) * sg[:, None]).sum())
            dt[k] = -v
        P = A * B
        both = torch.einsum("di,du,ui->i", self.bits[1], P, self.bits[0])
        one = self.bits[0].T @ P.sum(0) + self.bits[1].T @ P.sum(1)
        return dt, both.cpu().numpy(), one.cpu().numpy()


def _exact_green(case, seed):
    M, nu, nd = case["M"], case["n_up"], case["n_dn"]
    par = _params(case, seed)
    r = Reference(M, nu, nd, *par)
    X = _start_vector(case, seed, r).view(r.shape)
    p, spin, out = case["site"], case["spin"], {}
    for key, sg in (("plus", 1), ("minus", -1)):
        to = Reference(M, nu + (sg if spin == 0 else 0), nd + (sg if spin == 1 else 0), *par)
        s = to.s[spin]
        ok = np.nonzero(((s >> p) & 1) == (1 if sg > 0 else 0))[0]
        src = np.searchsorted(r.s[spin], s[ok] ^ (1 << p))
        below = s[ok] & ((1 << p) - 1)
        par_ = (sum((below >> k) & 1 for k in range(M)) + (nu if spin == 1 else 0)) & 1
        sign = torch.tensor(1.0 - 2.0 * par_, device=DEV)
        V = torch.zeros(to.shape, dtype=torch.float64, device=DEV)
        dst, src = torch.tensor(ok, device=DEV), torch.tensor(src, device=DEV)
        if spin == 0:
            V[:, dst] = X[:, src] * sign[None, :]
        else:
            V[dst, :] = X[src, :] * sign[:, None]
        v = V.reshape(-1)
        a, b, _, _ = to.lanczos(v, case["steps"])
        out[key] = dict(v=v, alpha=a, beta=b, norm2=float(torch.dot(v, v)))
    return out


def _act(perm, s):
    """Image of the spin strings s under a site permutation and the sign of reordering."""
    M = len(perm)
    img = np.zeros_like(s)
    inv = np.zeros_like(s)
    for i in range(M):
        img |= ((s >> i) & 1) << perm[i]
        for j in range(i + 1, M):
            if perm[j] < perm[i]:
                inv += ((s >> i) & (s >> j)) & 1
    return img, 1 - 2 * (inv & 1)


def _group(case):
    """Elements (breadth-first from the identity over the generators) and their characters."""
    perms, chars = _translations(case)
    ident = tuple(range(case["M"]))
    elems, chi = [ident], [1]
    k = 0
    while k < len(elems):
        for p, c in zip(perms, chars):
            e = tuple(int(p[i]) for i in elems[k])
            if e not in elems:
                elems.append(e)
                chi.append(chi[k] * c)
        k += 1
    return elems, chi


def _exact_momentum(case, seed):
    """The row form (up representatives x down strings in orbit order) spread over the full
    sector, where the Lanczos steps run; the vector is read back at the representatives."""
    r = Reference(case["M"], case["n_up"], case["n_dn"], *_params(case, seed))
    elems, chi = _group(case)
    su, sd = r.s
    acts = [[_act(e, s) for e in elems] for s in (su, sd)]
    up = np.stack([a[0] for a in acts[0]])
    reps = np.nonzero(up.min(0) == su)[0]
    stab = (up[:, reps] == su[reps][None, :]).sum(0)
    P = len(elems) / stab
    # columns: each down representative followed by its new images in element order
    dn = np.stack([a[0] for a in acts[1]])
    dsg = np.stack([a[1] for a in acts[1]])
    cols, csign = [], []
    for j in np.nonzero(dn.min(0) == sd)[0]:
        seen = set()
        for e in range(len(elems)):
            if int(dn[e, j]) not in seen:
                seen.add(int(dn[e, j]))
                cols.append(int(dn[e, j]))
                csign.append(int(dsg[e, j]))
    cidx = np.searchsorted(sd, np.array(cols))
    csg = torch.tensor(csign, dtype=torch.float64, device=DEV)
    sqP = torch.tensor(np.sqrt(P), device=DEV)
    X = _normal(seed, len(reps) * len(cols)).view(len(reps), len(cols))
    part = torch.zeros(r.shape[0], len(reps), dtype=torch.float64, device=DEV)   # Psi(R_i, d), one term per string
    part[torch.tensor(cidx, device=DEV)] = (X * csg[None, :] / sqP[:, None]).T
    part = part / torch.tensor(stab.astype(np.float64), device=DEV)[None, :]
    Psi = torch.zeros(r.shape, dtype=torch.float64, device=DEV)
    for e in range(len(elems)):
        ui = torch.tensor(np.searchsorted(su, up[e, reps]), device=DEV)
        di = torch.tensor(np.searchsorted(sd, dn[e]), device=DEV)
        sg = torch.tensor(acts[0][e][1][reps].astype(np.float64) * chi[e], device=DEV)[None, :] * \
            torch.tensor(dsg[e].astype(np.float64), device=DEV)[:, None]
        moved = torch.empty_like(part)
        moved[di] = part * sg
        Psi.index_add_(1, ui, moved)
    a, b, p, E = r.lanczos(Psi.reshape(-1), case["steps"], psi=case["psi"])
    if p is not None:
        rows = p.view(r.shape)[:, torch.tensor(reps, device=DEV)].T[:, torch.tensor(cidx, device=DEV)]
        p = (rows * csg[None, :] * sqP[:, None]).reshape(-1)
    return dict(E0=E, alpha=a, beta=b, psi=p)


def _exact_batch(case, seed):
    """Lowest eigenvalue of every job: dense for small sectors, else Lanczos with full
    re-orthogonalisation for all parameter sets of a sector together."""
    t, U, eps, sectors, *_ = _star_sets(case, seed)
    n = case["sets"]
    E = np.empty((n, len(sectors)))
    tt, UU, ee = (torch.tensor(v, device=DEV) for v in (t, U, eps))
    for k, (a, b) in enumerate(sectors):
        r = Reference(case["M"], a, b, _bonds(case), t[0], U[0], eps[0])
        D = r.shape[0] * r.shape[1]
        diag = torch.einsum("pi,di,ui->pdu", UU, r.bits[1], r.bits[0])
        diag += (ee @ r.bits[0].T)[:, None, :] + (ee @ r.bits[1].T)[:, :, None]

        def apply(X):
            Y = diag * X
            for bond in range(t.shape[1]):
                dst, src, sg = r.hops[0][bond]
                if len(dst):
                    Y.index_add_(2, dst, X.index_select(2, src) * (-tt[:, bond, None, None] * sg[None, None, :]))
                dst, src, sg = r.hops[1][bond]
                if len(dst):
                    Y.index_add_(1, dst, X.index_select(1, src) * (-tt[:, bond, None, None] * sg[None, :, None]))
            return Y
        if D <= 200:
            eye = torch.eye(D, dtype=torch.float64, device=DEV)
            H = torch.stack([apply(eye[i].view(1, *r.shape).expand(n, *r.shape)).reshape(n, D) for i in range(D)], 1)
            E[:, k] = torch.linalg.eigvalsh(H)[:, 0].cpu().numpy()
            continue
        steps = 110
        Q = torch.empty(n, steps, D, dtype=torch.float64, device=DEV)
        al, be = (torch.zeros(n, steps, dtype=torch.float64, device=DEV) for _ in range(2))
        q = _normal(seed, n * D, salt=2).view(n, D)
        q = q / q.norm(dim=1, keepdim=True)
        for j in range(steps):
            Q[:, j] = q
            w = apply(q.view(n, *r.shape)).reshape(n, D)
            al[:, j] = (q * w).sum(1)
            for _ in range(2):
                w = w - torch.einsum("pjd,pj->pd", Q[:, : j + 1], torch.einsum("pjd,pd->pj", Q[:, : j + 1], w))
            be[:, j] = w.norm(dim=1)
            q = w / be[:, j, None]
        T = torch.diag_embed(al) + torch.diag_embed(be[:, :-1], 1) + torch.diag_embed(be[:, :-1], -1)
        E[:, k] = torch.linalg.eigvalsh(T)[:, 0].cpu().numpy()
    return dict(E0=E.reshape(-1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "green":
        return _exact_green(case, seed)
    if kind == "momentum":
        return _exact_momentum(case, seed)
    r = Reference(case["M"], case["n_up"], case["n_dn"], *_params(case, seed))
    x = _start_vector(case, seed, r)
    if kind in ("apply", "host"):
        return r.apply(x)
    if kind == "lanczos":
        a, b, p, E = r.lanczos(x, case["steps"], psi=case["psi"])
        return dict(E0=E, alpha=a, beta=b, psi=p)
    if kind == "vjp":
        ybar = _normal(seed, x.numel(), salt=1)
        dt, dU, de = r.form(ybar, x)
        return dict(y=r.apply(x), dx=r.apply(ybar), dt=dt, dU=dU, deps=de)
    E, psi = r.ground(x)
    if kind == "ground":
        return dict(E0=E, psi=psi)
    dt, dU, de = r.form(psi, psi)
    return dict(E=E, dt=dt, dU=dU, deps=de)
