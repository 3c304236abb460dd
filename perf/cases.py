"""The work this library is asked to do, as timed cases.

Operator applications and solves through the public entry points, with the
inputs on the GPU as a program that calls them keeps them: links
exp(i eps A) with Gaussian traceless Hermitian A, Gaussian or point sources,
antiperiodic in t.  ``exact`` restates every operator in plain torch on
complex128 from its definition.

Results come back from the library in FP64 containers whatever precision
computed them; an operator result is returned here in the type that holds
the precision it was computed in.
"""

from __future__ import annotations

import math
from ctypes import byref, c_void_p

import torch

from paper_2303_05883_gb300 import _abi, api

BC = (1, 1, 1, -1)
DEV = "cuda"


def listed():
    return [
        # The smallest call: one application of the Wilson operator, in the
        # precision the methods take by default, on a lattice that fits in L2.
        dict(name="wilson_D_f64_8x8x8x8", what="mult", kind="wilson", op="D", prec="f64", x=8, y=8, z=8, t=8,
             nrhs=1, Ls=0, par=0.12),
        # A residual or a source as a program computes it: the full clover
        # operator in FP64 on a mid-size lattice.
        dict(name="clover_D_f64_24x24x24x48", what="mult", kind="clover", op="D", prec="f64", x=24, y=24, z=24, t=48,
             nrhs=1, Ls=0, par=0.125),
        # The even-odd operator on fields kept in the GPU layout, as a power
        # iteration or a polynomial filter applies it: the largest single
        # right-hand side in FP32.
        dict(name="clover_Dhat_f32_32x32x32x64", what="resident", kind="clover", op="Dhat", prec="f32", x=32, y=32,
             z=32, t=64, nrhs=1, Ls=0, par=0.125, applies=4),
        # The same on the twelve spin-colour columns of a propagator, 16-bit storage.
        dict(name="clover_Dhat_f16_24x24x24x48_12rhs", what="resident", kind="clover", op="Dhat", prec="f16", x=24,
             y=24, z=24, t=48, nrhs=12, Ls=0, par=0.125, applies=4),
        # The adjoint of the Moebius Schur operator (normal equations written by the caller).
        dict(name="mobius_Dhat_dag_f32_16x16x16x32_Ls16", what="mult", kind="mobius", op="Dhat_dag", prec="f32", x=16,
             y=16, z=16, t=32, nrhs=1, Ls=16, par=0.01),
        # The staggered operator in the default precision.
        dict(name="staggered_D_f64_32x32x32x32", what="mult", kind="staggered", op="D", prec="f64", x=32, y=32, z=32,
             t=32, nrhs=1, Ls=0, par=0.05),
        # The smallest solve, to near FP64 accuracy.
        dict(name="wilson_solve_f32_8x8x8x8", what="solve", kind="wilson", prec="f32", x=8, y=8, z=8, t=8, nrhs=1,
             Ls=0, par=0.12, tol=1e-12, source="gaussian"),
        # The headline solve: one right-hand side, FP32 inside FP64.
        dict(name="clover_solve_f32_32x32x32x64", what="solve", kind="clover", prec="f32", x=32, y=32, z=32, t=64,
             nrhs=1, Ls=0, par=0.125, tol=1e-12, source="gaussian"),
        # A propagator: twelve point sources with 16-bit inner storage.
        dict(name="clover_solve_f16_24x24x24x48_12rhs", what="solve", kind="clover", prec="f16", x=24, y=24, z=24,
             t=48, nrhs=12, Ls=0, par=0.125, tol=1e-12, source="point"),
        # Moebius domain wall: CG on the normal equations.
        dict(name="mobius_solve_f32_16x16x16x32_Ls16", what="solve", kind="mobius", prec="f32", x=16, y=16, z=16,
             t=32, nrhs=1, Ls=16, par=0.01, tol=1e-12, source="gaussian"),
        # Staggered CG.
        dict(name="staggered_solve_f32_48x48x48x48", what="solve", kind="staggered", prec="f32", x=48, y=48, z=48,
             t=48, nrhs=1, Ls=0, par=0.05, tol=1e-12, source="gaussian"),
        # The multigrid solver near the critical kappa, its hierarchy kept between solves.
        dict(name="multigrid_solve_16x16x16x32", what="mg", kind="clover", prec="f32", x=16, y=16, z=16, t=32, nrhs=1,
             Ls=0, par=0.1275, tol=1e-12, source="gaussian"),
    ]


def _extents(rng, lo, hi, step=2):
    """Four even extents with a volume spread evenly on a log scale over [lo, hi]."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = v ** 0.25
        d = [max(step, int(round(side * rng.uniform(0.7, 1.4) / step)) * step) for _ in range(3)]
        d.append(max(step, int(round(v / (d[0] * d[1] * d[2]) / step)) * step))
        if lo <= math.prod(d) <= hi and max(d) <= 96:
            return d


def draw(rng):
    what = rng.choice(["mult"] * 5 + ["resident"] * 2 + ["solve"] * 4 + ["mg"])
    nrhs = rng.choice([1, 1, 1, 2, 3, 4, 5, 7, 8, 11, 12])
    if what == "mg":
        d = [8 * rng.randint(1, 3) for _ in range(3)] + [8 * rng.randint(2, 5)]
        return dict(what=what, kind="clover", prec="f32", x=d[0], y=d[1], z=d[2], t=d[3], nrhs=1, Ls=0, par=0.1275,
                    tol=1e-12, source="gaussian")
    kinds = ["wilson", "clover", "clover", "clover"] if what == "resident" else ["wilson", "clover", "clover",
                                                                                "mobius", "staggered"]
    kind = rng.choice(kinds)
    Ls = rng.choice([4, 8, 10, 12, 16]) if kind == "mobius" else 0
    par = {"wilson": rng.choice([0.115, 0.12]), "clover": rng.choice([0.115, 0.12, 0.125]),
           "mobius": rng.choice([0.01, 0.05]), "staggered": rng.choice([0.05, 0.1])}[kind]
    if kind == "mobius":
        nrhs = 1 if nrhs < 8 else 2
    wc = kind in ("wilson", "clover")
    if what == "solve":
        prec = rng.choice(["f32", "f32", "f16", "bf16"]) if wc else "f32"
        d = _extents(rng, 8 ** 4, (24 ** 3 * 48 if wc or kind == "staggered" else 14 ** 3 * 28) // max(1, nrhs // 2))
        return dict(what=what, kind=kind, prec=prec, x=d[0], y=d[1], z=d[2], t=d[3], nrhs=nrhs, Ls=Ls, par=par,
                    tol=1e-12, source="point" if wc and nrhs > 6 else "gaussian")
    if what == "resident":
        prec = rng.choice(["f32", "f16", "bf16"])
        d = _extents(rng, 8 ** 4, 32 ** 3 * 64 // nrhs)
        return dict(what=what, kind=kind, op=rng.choice(["Dhat", "Dhat", "D"]), prec=prec, x=d[0], y=d[1], z=d[2],
                    t=d[3], nrhs=nrhs, Ls=0, par=par, applies=4)
    prec = rng.choice(["f64", "f64", "f32"] + (["f16", "bf16"] if wc else []))
    op = rng.choice(["D", "D", "Deo", "Dhat"] + (["Dhat_dag"] if kind == "mobius" else []))
    d = _extents(rng, 6 ** 4, 32 ** 3 * 64 // (nrhs * max(1, Ls)))
    return dict(what=what, kind=kind, op=op, prec=prec, x=d[0], y=d[1], z=d[2], t=d[3], nrhs=nrhs, Ls=Ls, par=par)


# ------------------------------------------------------------------ inputs


def _dims(c):
    return (c["x"], c["y"], c["z"], c["t"])


def _volume(c):
    return math.prod(_dims(c))


def _gauge(c, seed):
    """Links (4, V, 3, 3) complex128: exp(0.2 i A), made unitary in FP64."""
    V = _volume(c)
    g = torch.Generator(device=DEV).manual_seed(2 * seed + 1)
    w = torch.randn((4 * V, 8), generator=g, device=DEV) * 0.1  # eps / 2 times the Gell-Mann coefficients
    q = 1 / math.sqrt(3)
    zero = torch.zeros_like(w[:, 0])
    re = torch.stack([w[:, 2] + q * w[:, 7], w[:, 0], w[:, 3], w[:, 0], q * w[:, 7] - w[:, 2], w[:, 5], w[:, 3],
                      w[:, 5], -2 * q * w[:, 7]], 1)
    im = torch.stack([zero, -w[:, 1], -w[:, 4], w[:, 1], zero, -w[:, 6], w[:, 4], w[:, 6], zero], 1)
    X = torch.complex(-im, re).reshape(-1, 3, 3)  # i eps A
    E = torch.eye(3, dtype=X.dtype, device=DEV) + X / 8
    for k in range(7, 0, -1):
        E = torch.eye(3, dtype=X.dtype, device=DEV) + (X @ E) / k
    E = E.to(torch.complex128)
    r1 = E[:, 0] / torch.linalg.vector_norm(E[:, 0], dim=1, keepdim=True)
    r2 = E[:, 1] - (r1.conj() * E[:, 1]).sum(1, keepdim=True) * r1
    r2 = r2 / torch.linalg.vector_norm(r2, dim=1, keepdim=True)
    r3 = torch.linalg.cross(r1, r2).conj()
    return torch.stack([r1, r2, r3], 1).reshape(4, V, 3, 3).contiguous()


def _in_sites(c):
    V = _volume(c)
    return V if c["what"] in ("solve", "mg") or c["op"] == "D" else V // 2


def _source(c, seed):
    n = _in_sites(c)
    lead = () if c["nrhs"] == 1 and not c["Ls"] else (c["nrhs"] * max(1, c["Ls"]),)
    tail = (3,) if c["kind"] == "staggered" else (4, 3)
    if c.get("source") == "point":  # the spin-colour columns at a site of the caller's choice
        b = torch.zeros(lead + (n,) + tail, dtype=torch.complex128, device=DEV).reshape(-1, n, *tail)
        for k in range(c["nrhs"]):
            b[k, (7919 * seed) % n, k // 3, k % 3] = 1
        return b.reshape(lead + (n,) + tail)
    g = torch.Generator(device=DEV).manual_seed(2 * seed)
    return torch.randn(lead + (n,) + tail, generator=g, device=DEV, dtype=torch.complex128)


def _operator(c):
    if c["kind"] == "staggered":
        return api.make_staggered(c["par"], BC)
    if c["kind"] == "mobius":
        return api.make_mobius(c["Ls"], 1.8, 1.5, 0.5, c["par"], BC)
    return api.make_op(c["kind"], c["par"], 1.0 if c["kind"] == "clover" else 0.0, BC)


class _Fields:
    """Two fields in the GPU layout and the lattice they live on."""

    def __init__(self, lat, prec, subset, nrhs):
        self.lat = lat
        self.f = [api.bridge_field_create(lat.handle, prec, subset, nrhs) for _ in range(2)]

    def __del__(self):
        for f in self.f:
            api.bridge_field_destroy(f)


def prepare(case, seed):
    lat, op = api.Lattice(_dims(case)), _operator(case)
    lat.upload(_gauge(case, seed), op)
    b = _source(case, seed)
    s = dict(case=case, lat=lat, op=op, b=b)
    if case["what"] == "resident":
        s["fields"] = _Fields(lat, case["prec"], _abi.BRIDGE_FULL if case["op"] == "D" else _abi.BRIDGE_EVEN,
                              case["nrhs"])
        s["out"] = torch.empty_like(b)
    elif case["what"] == "solve":
        s["solver"] = api.make_solver(tol=case["tol"], inner_prec=case["prec"])
    elif case["what"] == "mg":
        s["solver"] = api.make_solver(tol=case["tol"], max_iter=1000)
        s["mg"] = api.Multigrid(lat, op, api.make_mg_params(nvec=12, setup_steps=3, coarse_tol=0.1, mr_steps=6))
    return s


def _typed(out, prec):
    if prec == "f64":
        return out
    if prec == "f32":
        return out.to(torch.complex64)
    return torch.view_as_real(out).to(torch.float16 if prec == "f16" else torch.bfloat16)


def run(state):
    c, lat, op, b = state["case"], state["lat"], state["op"], state["b"]
    if c["what"] == "mult":
        if c["op"] == "Deo":
            return _typed(lat.Deo(op, b, 0, c["prec"]), c["prec"])
        return _typed(getattr(lat, c["op"])(op, b, c["prec"]), c["prec"])
    if c["what"] == "resident":
        f = state["fields"].f
        which = _abi.BRIDGE_APPLY_D if c["op"] == "D" else _abi.BRIDGE_APPLY_DHAT
        api.bridge_field_import(f[0], b)
        for k in range(c["applies"]):
            api.bridge_apply(lat.handle, op, which, f[(k + 1) % 2], f[k % 2])
        api.bridge_field_export(f[c["applies"] % 2], state["out"])
        api.bridge_sync(lat.handle)
        return _typed(state["out"], c["prec"])
    if c["what"] == "solve":
        return lat.solve(op, b, state["solver"])[0]
    # the device form of Multigrid.solve
    x = torch.zeros_like(b)
    info = (_abi.bridge_info * 1)()
    torch.cuda.current_stream().synchronize()
    _abi.check(_abi.load().bridge_mg_solve_dev(state["mg"].handle, byref(state["solver"]), c_void_p(b.data_ptr()),
                                               c_void_p(x.data_ptr()), 1, info), "bridge_mg_solve_dev")
    return x


# -------------------------------------------------------------------- work


def work(case):
    """Inputs read once and outputs written once, per launch-wide dependency:
    an operator application reads its canonical input, the links and the site
    terms and writes its output; a solve does so in its inner precision once
    per hopping pass of each iteration, with the vectors of its recurrence.
    Iterations of the Krylov solvers: what these parameters need to 1e-12."""
    V, n, Ls = _volume(case), case["nrhs"], max(1, case["Ls"])
    kind, prec = case["kind"], case["prec"]
    R = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[prec]
    comp = 6 if kind == "staggered" else 24
    link = 4 * V * (18 if prec == "f64" else 12) * R
    site = 72 * R * V if kind == "clover" else 0
    # flops a site: staggered 570, Wilson hop 1320, clover term 504, fifth-dimension factor 192
    hop = 570 if kind == "staggered" else 1344 + (192 if kind == "mobius" else 0)
    fl = (hop + (504 if kind == "clover" else 0)) * V * n * Ls
    if case["what"] in ("mult", "resident"):
        half = 0.5 if case["op"] == "Deo" else 1.0
        k = case.get("applies", 1)
        if case["op"] == "Deo":
            site, fl = 0, hop * V * n * Ls
        canon = 2 * _in_sites(case) * n * Ls * comp * 8
        out = canon // 2 * R // 8 if R < 8 else 0  # the result in the type that holds its precision
        mid = 2 * (V if case["op"] == "D" else V // 2) * n * Ls * comp * R * (k - 1)
        return dict(bytes=canon + out + mid + k * (link + site), flops=half * fl * k)
    if case["what"] == "mg":
        # two cycles and operators per outer iteration: the fine level once per SAP sweep and residual
        its, passes = 14, 10
        return dict(bytes=its * passes * (link + site + 3 * V * comp * R), flops=its * passes * fl)
    its = {"wilson": 45, "clover": 150, "mobius": 430, "staggered": 360}[kind]
    vec = {"wilson": 20, "clover": 20, "mobius": 17, "staggered": 13}[kind] * (V // 2) * n * Ls * comp * R
    per = 2 if kind == "staggered" else 4  # hopping passes of an iteration, each over all links, half the sites
    return dict(bytes=its * (per * (link + site / 2) + vec) + 2 * V * n * Ls * comp * 8, flops=its * per * fl / 2)


# ------------------------------------------------------------------- exact


def _gammas():
    s = [torch.tensor(m, dtype=torch.complex128) for m in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    g = []
    for k in range(4):
        m = torch.zeros((4, 4), dtype=torch.complex128)
        m[:2, 2:] = -1j * s[k] if k < 3 else torch.eye(2)
        m[2:, :2] = 1j * s[k] if k < 3 else torch.eye(2)
        g.append(m.to(DEV))
    return g


class _Exact:
    """The operators from their definitions on complex128, sites [t][z][y][x]."""

    def __init__(self, c, seed):
        self.c, self.d = c, _dims(c)
        self.grid = tuple(reversed(self.d))
        self.U = _gauge(c, seed).reshape(4, *self.grid, 3, 3)
        self.g = _gammas()
        self.one = torch.eye(4, dtype=torch.complex128, device=DEV)
        co = torch.meshgrid(*[torch.arange(k, device=DEV) for k in self.grid], indexing="ij")
        self.coord = list(reversed(co))  # x, y, z, t
        par = (sum(self.coord) % 2).reshape(-1)
        self.sites = [torch.nonzero(par == p)[:, 0] for p in (0, 1)]
        self.blocks = None

    def shift(self, f, mu, step, phase=True):
        """f(x + step mu), with the boundary phase of a wrapping hop."""
        ax = 3 - mu
        r = torch.roll(f, -step, ax)
        if phase and BC[mu] != 1:
            r.select(ax, self.d[mu] - 1 if step > 0 else 0).mul_(BC[mu])
        return r

    def hop(self, psi):
        """H psi of one spinor field (V, 4, 3), or the staggered hop of (V, 3)."""
        stag = self.c["kind"] == "staggered"
        p = psi.reshape(*self.grid, *((3, 1) if stag else (4, 3)))
        out = torch.zeros_like(p)
        for mu in range(4):
            f, bwd = self.shift(p, mu, 1), None
            if stag:
                eta = 1 - 2 * (sum(self.coord[:mu]) % 2) if mu else torch.ones_like(self.coord[0])
                eta = eta[..., None, None]
                bwd = self.shift(self.U[mu].mH @ p, mu, -1)
                out += 0.5 * eta * (self.U[mu] @ f - bwd)
            else:
                out += (self.one - self.g[mu]) @ (f @ self.U[mu].mT)
                bwd = self.shift(p @ self.U[mu].conj(), mu, -1)
                out += (self.one + self.g[mu]) @ bwd
        return out.reshape(psi.shape)

    def term(self):
        """T as two 6x6 blocks a site, (2, V, 6, 6), and its inverse."""
        if self.blocks is None:
            V = math.prod(self.d)
            T = torch.eye(6, dtype=torch.complex128, device=DEV).repeat(2, V, 1, 1)
            for mu in range(4):
                for nu in range(mu + 1, 4):
                    S = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                    F = self.field_strength(mu, nu).reshape(V, 3, 3)
                    for b in (0, 1):
                        s = S[2 * b : 2 * b + 2, 2 * b : 2 * b + 2]
                        T[b] -= self.c["par"] * (s[None, :, None, :, None] * F[:, None, :, None, :]).reshape(V, 6, 6)
            self.blocks = T
        return self.blocks

    def field_strength(self, mu, nu):
        m, n = self.U[mu], self.U[nu]
        sh = lambda f, d, k: self.shift(f, d, k, phase=False)  # noqa: E731
        mm, nn = sh(m, mu, -1), sh(n, nu, -1)
        n_mm, m_nn = sh(n, mu, -1), sh(m, nu, -1)
        q = m @ sh(n, mu, 1) @ sh(m, nu, 1).mH @ n.mH
        q = q + n @ sh(mm, nu, 1).mH @ n_mm.mH @ mm
        q = q + mm.mH @ sh(n_mm, nu, -1).mH @ sh(mm, nu, -1) @ nn
        q = q + nn.mH @ m_nn @ sh(nn, mu, 1) @ m.mH
        F = (q - q.mH) / 8j
        tr = F.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
        return F - tr[..., None, None] * torch.eye(3, dtype=F.dtype, device=DEV)

    def site(self, v, parity=None, inverse=False):
        if self.c["kind"] != "clover":
            return v
        T = self.term() if parity is None else self.term()[:, self.sites[parity]]
        w = v.reshape(-1, 2, 6).transpose(0, 1)[..., None]
        w = torch.linalg.solve(T, w) if inverse else T @ w
        return w[..., 0].transpose(0, 1).reshape(v.shape)

    def half(self, v, q):
        """H v from parity 1 - q to parity q on half-lattice vectors."""
        f = torch.zeros((math.prod(self.d),) + v.shape[1:], dtype=v.dtype, device=DEV)
        f[self.sites[1 - q]] = v
        return self.hop(f)[self.sites[q]]

    def smat(self, which):
        """Fifth-dimension matrices (chirality, Ls, Ls) of A or B."""
        Ls, mf, al = self.c["Ls"], self.c["par"], 4 - 1.8
        S = torch.zeros((2, Ls, Ls), dtype=torch.float64)
        for s in range(Ls):
            S[0, s, s - 1 if s else Ls - 1] = 1 if s else -mf
            S[1, s, s + 1 if s + 1 < Ls else 0] = 1 if s + 1 < Ls else -mf
        d, e = (1.5 * al + 1, 0.5 * al - 1) if which == "A" else (1.5, 0.5)
        return (d * torch.eye(Ls, dtype=torch.float64) + e * S).to(DEV)

    def mix(self, M, v):
        M = M.to(torch.complex128)
        return torch.stack([torch.tensordot(M[b], v[:, :, 2 * b : 2 * b + 2], 1) for b in (0, 1)], 2).reshape(v.shape)

    def hops(self, v, q):
        return torch.stack([self.hop(s) if q is None else self.half(s, q) for s in v])

    def apply(self, op, v):
        """One right-hand side: (V, 4, 3), (V, 3) or (Ls, V, 4, 3)."""
        c = self.c
        if c["kind"] == "mobius":
            A, B = self.smat("A"), self.smat("B")
            if op == "D":
                return self.mix(A, v) - 0.5 * self.hops(self.mix(B, v), None)
            if op == "Deo":
                return -0.5 * self.hops(self.mix(B, v), 0)
            Ai = torch.linalg.inv(A)
            if op == "Dhat":
                w = -0.5 * self.mix(Ai, self.hops(self.mix(B, v), 1))
                return v + 0.5 * self.mix(Ai, self.hops(self.mix(B, w), 0))
            g5 = torch.tensor([1, 1, -1, -1], device=DEV)[:, None]
            w = g5 * self.hops(g5 * self.mix(Ai.mT, v), 1) * -0.5
            w = self.mix(Ai.mT, self.mix(B.mT, w))
            return v + 0.5 * self.mix(B.mT, g5 * self.hops(g5 * w, 0))
        if c["kind"] == "staggered":
            if op == "D":
                return c["par"] * v + self.hop(v)
            return self.half(v, 0) if op == "Deo" else v - self.half(self.half(v, 1), 0) / c["par"] ** 2
        k = c["par"]
        if op == "D":
            return self.site(v) - k * self.hop(v)
        if op == "Deo":
            return -k * self.half(v, 0)
        return v - k * k * self.site(self.half(self.site(self.half(v, 1), 1, True), 0), 0, True)


def _bicgstab(A, b, tol):
    """BiCGStab (van der Vorst) to a relative residual of tol, restarted from the true residual."""
    x = torch.zeros_like(b)
    dot = lambda u, v: torch.vdot(u.reshape(-1), v.reshape(-1))  # noqa: E731
    nb = float(torch.linalg.vector_norm(b))
    for _ in range(6):
        r = b - A(x)
        if float(torch.linalg.vector_norm(r)) <= tol * nb:
            break
        h, p, rho = r.clone(), r.clone(), dot(r, r)
        for _ in range(400):
            v = A(p)
            al = rho / dot(h, v)
            s = r - al * v
            t = A(s)
            om = dot(t, s) / dot(t, t)
            x = x + al * p + om * s
            r = s - om * t
            if float(torch.linalg.vector_norm(r)) <= tol * nb:
                break
            new = dot(h, r)
            p = r + (new / rho) * (al / om) * (p - om * v)
            rho = new
    return x


def exact(case, seed):
    b = _source(case, seed)
    if case["what"] in ("solve", "mg"):
        # the smaller Wilson and clover systems; the others would take minutes in plain torch
        if case["kind"] not in ("wilson", "clover") or case["nrhs"] > 1 or _volume(case) > 8 ** 3 * 16:
            return None
        E = _Exact(case, seed)
        return _bicgstab(lambda v: E.apply("D", v), b.reshape(-1, 4, 3), 1e-14).reshape(b.shape)
    E = _Exact(case, seed)
    Ls = max(1, case["Ls"])
    tail = 2 if case["kind"] == "staggered" else 3
    v = b.reshape((case["nrhs"],) + ((Ls,) if case["Ls"] else ()) + b.shape[-tail:])
    out = []
    for one in v:
        for _ in range(case.get("applies", 1)):
            one = E.apply(case["op"], one)
        out.append(one)
    out = torch.stack(out).reshape(b.shape)
    return out if case["prec"] in ("f64", "f32") else torch.view_as_real(out)
