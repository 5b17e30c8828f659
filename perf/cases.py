"""Performance workloads of the library, through its public calls (``paper_1712_01505_gb300.qcd``).

Three kinds of pass, each on links and fields drawn on the GPU from a seed:

* ``solve``: one ``qcd.solve`` on device fields -- Wilson BiCGStab or domain-wall CG, one or several
  right-hand sides, plain FP64 or mixed precision with IEEE-FP64 outer steps; the output is the solution.
  The target is |b - A x| <= 1e-12 |b| (the molecular dynamics' and the differentiable action's
  default), so that the solution is determined to far better than its last figures of interest.
* ``apply``: one ``qcd.dslash`` -- FP32 / FP16 on the library's internal single-parity buffers (what an
  iteration of a user's own solver calls), FP64 on canonical full-lattice fields (a user's residual check).
* ``md``: one molecular-dynamics step of the even-odd pseudofermion action -- two solves, the force,
  its su(3) projection, the momentum and link updates and the kinetic energy.

``exact`` computes the same in plain torch complex128: the hop by neighbour tables, solves by
iterative refinement (single-precision Krylov corrections of the 64-bit residual, until the residual
is at the rounding of the operator).
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1712_01505_gb300 import qcd

DEV = "cuda"
BC = (1, 1, 1, -1)
TOL = 1e-12
M5, MF = 1.8, 0.02
MD_EPS = 0.02

# Krylov iterations to TOL that work() counts (what the systems below need; more or fewer are the code's own)
ITERS = {"wilson": 64, "dw": 330}
OPS = ("D_EO", "D_OE", "MHAT", "MHAT_DAG", "FULL", "FULL_DAG")


def listed():
    return [
        # the benchmark's mixed solve: a quark propagator's source on the largest lattice
        dict(name="solve 32x32x32x64 f32", kind="solve", L="32x32x32x64", recon=12, fermion="wilson", kappa=0.125,
             eps=0.2, inner="f32", delta=1e-5, nrhs=1, source="z2", dagger=False),
        # the same solver with FP16 inner vectors on the propagator lattice
        dict(name="solve 24x24x24x48 f16", kind="solve", L="24x24x24x48", recon=12, fermion="wilson", kappa=0.124,
             eps=0.2, inner="f16", delta=2e-3, nrhs=1, source="z2", dagger=True),
        # a solve so small that launches and synchronisations are its time
        dict(name="solve 8x8x8x16 f32", kind="solve", L="8x8x8x16", recon=18, fermion="wilson", kappa=0.12,
             eps=0.3, inner="f32", delta=0.0, nrhs=1, source="gauss", dagger=False),
        # plain double precision, extents that no tile divides
        dict(name="solve 12x10x14x18 f64", kind="solve", L="12x10x14x18", recon=18, fermion="wilson", kappa=0.122,
             eps=0.3, inner="f64", delta=0.0, nrhs=1, source="gauss", dagger=False),
        # the 12 spin-colour point sources of a propagator in one batched solve
        dict(name="solve 24x24x24x48 12rhs", kind="solve", L="24x24x24x48", recon=12, fermion="wilson", kappa=0.124,
             eps=0.2, inner="f32", delta=1e-5, nrhs=12, source="point", dagger=False),
        # domain-wall CG on the normal equations, FP16 inner vectors
        dict(name="dw solve 16x16x16x32 Ls16", kind="solve", L="16x16x16x32", recon=12, fermion="shamir", Ls=16,
             eps=0.2, inner="f16", delta=0.0, nrhs=1, source="z2", dagger=False),
        # one force evaluation and update of the links in ensemble generation
        dict(name="md step 16x16x16x16", kind="md", L="16x16x16x16", recon=18, kappa=0.12, eps=0.3, inner="f32"),
        # the FP32 half-dslash the paper's figures are quoted on
        dict(name="D_EO 32x32x32x64 f32", kind="apply", L="32x32x32x64", recon=12, fermion="wilson", kappa=0.125,
             eps=0.2, op="D_EO", prec="f32", nrhs=1),
        # the FP16 Schur operator of a user's own inner solver
        dict(name="MHAT 32x32x32x64 f16", kind="apply", L="32x32x32x64", recon=12, fermion="wilson", kappa=0.125,
             eps=0.2, op="MHAT", prec="f16", nrhs=1),
        # the Mobius Schur operator's adjoint, FP32: the fused hop + fifth-dimension inverse
        dict(name="mobius MHAT_DAG Ls16 f32", kind="apply", L="16x16x16x32", recon=12, fermion="mobius", Ls=16,
             eps=0.2, op="MHAT_DAG", prec="f32", nrhs=1),
        # the unpreconditioned matrix on canonical FP64 fields: a user's residual check
        dict(name="FULL 24x24x24x48 f64", kind="apply", L="24x24x24x48", recon=12, fermion="wilson", kappa=0.124,
             eps=0.2, op="FULL", prec="f64", nrhs=1),
        # the smallest call: a half-dslash whose time is the launch
        dict(name="D_OE 6x4x6x10 f32", kind="apply", L="6x4x6x10", recon=18, fermion="wilson", kappa=0.12,
             eps=0.3, op="D_OE", prec="f32", nrhs=1),
    ]


def _extents(rng, lo, hi, tmax, vlo, vhi):
    """Even extents with a volume spread over its logarithm."""
    target = float(np.exp(rng.uniform(np.log(vlo), np.log(vhi))))
    for _ in range(4000):
        L = [2 * rng.randint(lo // 2, hi // 2) for _ in range(3)] + [2 * rng.randint(lo // 2, tmax // 2)]
        v = float(np.prod(L))
        if vlo <= v <= vhi and 0.7 < v / target < 1.4:
            return L
    raise RuntimeError("no lattice drawn")


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "dw", "batch", "md", "apply", "apply", "apply64", "applydw"])
    eps = round(rng.uniform(0.2, 0.3), 3)
    kappa = round(rng.uniform(0.115, 0.1245), 4)
    recon = rng.choice([12, 18])

    def text(L):
        return "x".join(str(v) for v in L)

    if kind == "solve":
        inner = rng.choice(["f32", "f32", "f16", "f64"])
        L = _extents(rng, 4, 32, 64, 1024, 131072 if inner == "f64" else 2097152)
        delta = {"f32": rng.choice([0.0, 1e-5, 1e-3]), "f16": rng.choice([0.0, 2e-3]), "f64": 0.0}[inner]
        return dict(kind="solve", L=text(L), recon=recon, fermion="wilson", kappa=kappa, eps=eps, inner=inner,
                    delta=delta, nrhs=1, source=rng.choice(["z2", "gauss", "point"]), dagger=rng.random() < 0.5)
    if kind == "dw":
        L = _extents(rng, 4, 16, 32, 1024, 65536)
        return dict(kind="solve", L=text(L), recon=recon, fermion=rng.choice(["shamir", "mobius"]),
                    Ls=rng.choice([6, 8, 10, 12, 16]), eps=eps, inner=rng.choice(["f32", "f16"]), delta=0.0, nrhs=1,
                    source=rng.choice(["z2", "gauss"]), dagger=False)
    if kind == "batch":
        L = _extents(rng, 4, 24, 48, 2048, 331776)
        return dict(kind="solve", L=text(L), recon=recon, fermion="wilson", kappa=kappa, eps=eps, inner="f32",
                    delta=rng.choice([0.0, 1e-5]), nrhs=rng.choice([2, 3, 4, 6, 8, 12]), source=rng.choice(["z2", "gauss"]),
                    dagger=False)
    if kind == "md":
        L = _extents(rng, 4, 16, 24, 1024, 65536)
        return dict(kind="md", L=text(L), recon=18, kappa=min(kappa, 0.122), eps=0.3, inner="f32")
    if kind == "apply":
        nrhs = rng.choice([1, 1, 2, 5, 8, 12])
        L = _extents(rng, 4, 32, 64, 512, 2097152 // nrhs)
        return dict(kind="apply", L=text(L), recon=recon, fermion="wilson", kappa=kappa, eps=eps,
                    op=rng.choice(["D_EO", "D_OE", "MHAT", "MHAT_DAG"]), prec=rng.choice(["f32", "f16"]), nrhs=nrhs)
    if kind == "apply64":
        L = _extents(rng, 4, 24, 48, 1024, 663552)
        return dict(kind="apply", L=text(L), recon=recon, fermion="wilson", kappa=kappa, eps=eps,
                    op=rng.choice(["FULL", "FULL_DAG", "MHAT", "D_EO"]), prec="f64", nrhs=1)
    L = _extents(rng, 4, 16, 32, 512, 131072)
    return dict(kind="apply", L=text(L), recon=recon, fermion=rng.choice(["shamir", "mobius"]),
                Ls=rng.choice([4, 6, 8, 12, 16]), eps=eps, op=rng.choice(["D_EO", "MHAT", "MHAT_DAG"]),
                prec=rng.choice(["f32", "f16"]), nrhs=1)


# ----------------------------------------------------------------------------- inputs
def _lattice(case):
    return tuple(int(v) for v in case["L"].split("x"))


def _is_dw(case):
    return case.get("fermion") in ("shamir", "mobius")


def _ls(case):
    return case["Ls"] if _is_dw(case) else 1


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _su3(n, eps, gen):
    """n smoothed random SU(3) matrices: exp(i eps H) by its series, H Hermitian traceless with Gaussian
    entries, then Gram-Schmidt on the rows (the third is conj(row0 x row1))."""
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device=DEV)
    step = 1 << 20
    for i in range(0, n, step):
        m = min(step, n - i)
        a = torch.view_as_complex(torch.randn((m, 3, 3, 2), dtype=torch.float64, device=DEV, generator=gen))
        h = 0.5 * (a + a.conj().transpose(1, 2))
        tr = (h[:, 0, 0] + h[:, 1, 1] + h[:, 2, 2]) / 3.0
        x = 1j * eps * (h - tr[:, None, None] * torch.eye(3, dtype=h.dtype, device=DEV))
        u = torch.eye(3, dtype=h.dtype, device=DEV) + x
        term = x
        for k in range(2, 9):
            term = _mm(term, x) / k
            u = u + term
        r0, r1 = u[:, 0], u[:, 1]
        r0 = r0 / r0.abs().square().sum(-1, keepdim=True).sqrt()
        r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
        r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
        r2 = torch.linalg.cross(r0, r1).conj()
        out[i:i + m] = torch.stack([r0, r1, r2], dim=1)
    return out


def _mm(a, b):
    """Products of (n, 3, 3) matrices, elementwise over n."""
    return a[:, :, 0:1] * b[:, 0:1, :] + a[:, :, 1:2] * b[:, 1:2, :] + a[:, :, 2:3] * b[:, 2:3, :]


def _links(case, gen):
    V = int(np.prod(_lattice(case)))
    return _su3(4 * V, case["eps"], gen).reshape(4, V, 3, 3)


def _gauss(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device=DEV, generator=gen))


def _source(case, gen):
    V = int(np.prod(_lattice(case)))
    n = case.get("nrhs", 1)
    shape = (n, _ls(case), V, 4, 3) if _is_dw(case) else (n, V, 4, 3)
    what = case.get("source", "gauss")
    if what == "gauss":
        return _gauss(shape, gen)
    if what == "z2":
        s = torch.randint(0, 2, shape + (2,), device=DEV, generator=gen).to(torch.float64) * 2 - 1
        return torch.view_as_complex(s / np.sqrt(2.0))
    b = torch.zeros(shape, dtype=torch.complex128, device=DEV)
    x0 = int(torch.randint(0, V, (1,), device=DEV, generator=gen).item())
    for k in range(n):
        b[k, x0, (k % 12) // 3, k % 3] = 1.0
    return b


def _momenta(V, gen):
    a = _gauss((4, V, 3, 3), gen)
    h = 0.5 * (a + a.conj().transpose(-1, -2))
    tr = (h[..., 0, 0] + h[..., 1, 1] + h[..., 2, 2]) / 3.0
    return 1j * (h - tr[..., None, None] * torch.eye(3, dtype=h.dtype, device=DEV))


def _parity(L):
    V = int(np.prod(L))
    i = torch.arange(V, device=DEV)
    p, r = torch.zeros_like(i), i
    for m in range(4):
        p, r = p + r % L[m], r // L[m]
    return p % 2


def _fermion(case):
    if case.get("fermion") == "shamir":
        return qcd.dwf(case["Ls"], M5, MF)
    if case.get("fermion") == "mobius":
        return qcd.mobius(case["Ls"], M5, MF, 1.5, 0.5)
    return qcd.wilson(case["kappa"])


def _b5c5(case):
    return (1.5, 0.5) if case["fermion"] == "mobius" else (1.0, 0.0)


def _in_parity(op):
    return 1 if op == "D_EO" else 0


def prepare(case, seed):
    gen = _gen(seed)
    L = _lattice(case)
    V = int(np.prod(L))
    U = _links(case, gen)
    g = qcd.Gauge.load(U, L, BC, recon=case["recon"])
    f = _fermion(case)
    s = dict(case=case, g=g, f=f)
    if case["kind"] == "md":
        phi = _gauss((V, 4, 3), gen)
        even = (_parity(L) == 0).to(torch.float64)[:, None, None]
        s.update(U=U, P=_momenta(V, gen), phi=phi * even, even=even, dS=torch.empty((4, V, 3, 3, 2), dtype=torch.float64,
                 device=DEV), F=torch.empty((4, V, 3, 3), dtype=torch.complex128, device=DEV), w=torch.empty_like(phi),
                 X=torch.empty_like(phi), P1=torch.empty_like(U), U1=torch.empty_like(U))
        return s
    b = _source(case, gen)
    if case["kind"] == "solve":
        s.update(b=b, x=torch.zeros_like(b))
        return s
    if case["prec"] == "f64":
        s.update(inp=b, out=torch.empty_like(b))
        return s
    n = qcd.field_bytes(g, f, case["prec"], case["nrhs"])
    s["inp"] = torch.empty(n, dtype=torch.uint8, device=DEV)
    s["out"] = torch.empty(n, dtype=torch.uint8, device=DEV)
    qcd.field_pack(g, f, case["prec"], _in_parity(case["op"]), b, s["inp"], nrhs=case["nrhs"])
    return s


# ----------------------------------------------------------------------------- one pass
def _solve_args(case):
    dw = _is_dw(case)
    return dict(method=qcd.CG_NORMAL if dw else qcd.BICGSTAB, tol=TOL, inner=case["inner"], outer="f64",
                delta=case.get("delta", 0.0), use_graph=True, graph_chunk=32)


def run(state):
    case, g, f = state["case"], state["g"], state["f"]
    if case["kind"] == "solve":
        qcd.solve(g, f, state["b"], state["x"], nrhs=case["nrhs"], dagger=case["dagger"], **_solve_args(case))
        return {"x": state["x"]}
    if case["kind"] == "apply":
        if case["prec"] == "f64":
            qcd.dslash(g, f, case["op"], state["inp"], state["out"], prec="f64", nrhs=case["nrhs"])
            return {"out": state["out"]}
        qcd.dslash(g, f, case["op"], state["inp"], state["out"], prec=case["prec"], nrhs=case["nrhs"],
                   layout=qcd.INTERNAL)
        if case["prec"] == "f32":
            return {"out": state["out"].view(torch.float32)}
        nh = state["out"].numel() // 52 * 48  # 24 binary16 per site, then one FP32 scale per site
        return {"halves": state["out"][:nh].view(torch.float16), "scale": state["out"][nh:].view(torch.float32)}
    kw = _solve_args(case)
    z, X, P, U = state["w"], state["X"], state["P1"], state["U1"]
    qcd.solve(g, f, state["phi"], z, dagger=True, **kw)
    z.mul_(state["even"])
    qcd.solve(g, f, z, X, **kw)
    qcd.force_eo(g, f, X, z, state["dS"])
    qcd.force_project(g, state["dS"], state["F"])
    P.copy_(state["P"])
    qcd.mom_update(P, state["F"], MD_EPS)
    U.copy_(state["U"])
    qcd.link_update(U, P, MD_EPS)
    return {"dS": state["dS"], "P": P, "U": U, "energy": qcd.mom_energy(P)}


# ----------------------------------------------------------------------------- work
def _site_bytes(prec):
    return {"f64": 192, "f32": 96, "f16": 52}[prec]


def _link_bytes(case, prec):
    return {"f64": 144, "f32": 4 * case["recon"], "f16": 2 * case["recon"]}[prec]


def _hop_work(case, prec, n, vh):
    """A half-dslash of n vectors: links once, each spinor in and out once."""
    return vh * 8 * _link_bytes(case, prec) + 2 * n * vh * _site_bytes(prec), 1320 * n * vh


def work(case):
    L = _lattice(case)
    V = int(np.prod(L))
    vh, ls, n = V // 2, _ls(case), case.get("nrhs", 1) * _ls(case)
    if case["kind"] == "apply":
        prec, op = case["prec"], case["op"]
        hops = 2 if op not in ("D_EO", "D_OE") else 1
        links = vh * 8 * _link_bytes(case, prec)
        _, fl = _hop_work(case, prec, n, vh)
        fl5 = 6 * ls * 24 * n * vh if _is_dw(case) and hops == 2 else 0
        field = 192 * 2 if prec == "f64" else _site_bytes(prec)  # FP64: both parities of a canonical field
        return {"bytes": links + 2 * n * vh * field, "flops": hops * fl + fl5}
    if case["kind"] == "md":
        by, fl = _hop_work(case, "f32", 1, vh)
        it = 2 * ITERS["wilson"]
        return {"bytes": it * (4 * by + 14 * vh * 96) + 4 * V * 144 * 6 + 4 * V * 192,
                "flops": it * (4 * fl + 300 * vh) + 4 * V * 600}
    by, fl = _hop_work(case, case["inner"], n, vh)
    site = _site_bytes(case["inner"])
    if _is_dw(case):  # per iteration of CG: Mhat and Mhat^dag, and p, x, r updated once
        it, vec, w5 = ITERS["dw"], 7, 4 * 6 * 24
    else:             # per iteration of BiCGStab: Mhat twice, and p, s, x, r updated once
        it, vec, w5 = ITERS["wilson"], 14, 0
    return {"bytes": it * (4 * by + vec * n * vh * site) + 4 * n * V * 192,
            "flops": it * (4 * fl + (300 + w5) * n * vh)}


# ----------------------------------------------------------------------------- 64-bit values, plain torch
class _Wilson4D:
    """The even-odd hop on (S, 4, 3, Vh) fields of complex dtype, by neighbour tables."""

    B = {0: ((1, -1j), (0, -1j)), 1: ((1, -1), (0, 1)), 2: ((0, -1j), (1, 1j)), 3: ((0, 1), (1, 1))}

    def __init__(self, L, U):
        self.L, V = L, int(np.prod(L))
        i = torch.arange(V, device=DEV)
        x, r = [], i
        for m in range(4):
            x.append(r % L[m])
            r = r // L[m]
        par = (x[0] + x[1] + x[2] + x[3]) % 2
        self.sites = [torch.nonzero(par == p).flatten() for p in (0, 1)]
        self.nb, self.sign, self.U = {}, {}, {}
        stride = 1
        for mu in range(4):
            for d in (1, -1):
                edge = x[mu] == (L[mu] - 1 if d > 0 else 0)
                j = torch.where(edge, i - d * (L[mu] - 1) * stride, i + d * stride)
                for p in (0, 1):
                    s = self.sites[p]
                    self.nb[p, mu, d] = j[s] // 2
                    self.sign[p, mu, d] = torch.where(edge[s], float(BC[mu]), 1.0).to(torch.float64)
            stride *= L[mu]
            for p in (0, 1):
                self.U[p, mu] = U[mu][self.sites[p]].permute(1, 2, 0).contiguous()
        self.U64, self.sign64 = self.U, self.sign
        self.U32 = {k: v.to(torch.complex64) for k, v in self.U.items()}
        self.sign32 = {k: v.to(torch.float32) for k, v in self.sign.items()}

    def split(self, psi):
        """canonical (S, V, 4, 3) -> its even and odd halves (S, 4, 3, Vh)"""
        return [psi[:, s].permute(0, 2, 3, 1).contiguous() for s in self.sites]

    def join(self, e, o):
        out = torch.empty((e.shape[0], 2 * e.shape[3], 4, 3), dtype=e.dtype, device=DEV)
        for h, s in ((e, self.sites[0]), (o, self.sites[1])):
            out[:, s] = h.permute(0, 3, 1, 2)
        return out

    def hop(self, p, psi, dag=False):
        """H_{p,1-p} psi: sum over mu of (1 -+ gamma) U psi(x + mu) + (1 +- gamma) U^dag psi(x - mu)."""
        wide = psi.dtype == torch.complex128
        U, sign = (self.U64, self.sign64) if wide else (self.U32, self.sign32)
        out = torch.zeros_like(psi)
        for mu in range(4):
            (j0, c0), (j1, c1) = self.B[mu]
            for d in (1, -1):
                sg = (-1 if d > 0 else 1) * (-1 if dag else 1)
                nb = self.nb[p, mu, d]
                g = psi[..., nb]
                h = torch.stack([g[:, 0] + (sg * c0) * g[:, 2 + j0], g[:, 1] + (sg * c1) * g[:, 2 + j1]], 1)
                h = h * sign[p, mu, d]
                u = U[p, mu] if d > 0 else U[1 - p, mu][..., nb].conj().transpose(0, 1)
                w = u[:, 0] * h[:, :, 0:1] + u[:, 1] * h[:, :, 1:2] + u[:, 2] * h[:, :, 2:3]
                out[:, :2] += w
                # lower spins: sg B^dag w; row k of B has its element at column j_k
                out[:, 2 + j0] += (sg * np.conj(c0)) * w[:, 0]
                out[:, 2 + j1] += (sg * np.conj(c1)) * w[:, 1]
        return out


def _fifth(Ls, d, e, mf):
    """d + e S on the P+ (lower shift) and P- (upper shift) spins, as two (Ls, Ls) matrices."""
    lo = torch.diag(torch.ones(Ls - 1, dtype=torch.float64, device=DEV), -1)
    lo[0, Ls - 1] = -mf
    one = torch.eye(Ls, dtype=torch.float64, device=DEV)
    up = torch.diag(torch.ones(Ls - 1, dtype=torch.float64, device=DEV), 1)
    up[Ls - 1, 0] = -mf
    return d * one + e * lo, d * one + e * up


def _apply5(pair, psi):
    """The (Ls, Ls) matrices on the upper and lower spins of (n * Ls, 4, 3, Vh)."""
    Ls = pair[0].shape[0]
    v = psi.reshape(-1, Ls, 2, 6 * psi.shape[3])
    out = torch.empty_like(v)
    for h in (0, 1):
        m = pair[h].to(v.dtype)
        for r in range(v.shape[0]):
            out[r, :, h] = m @ v[r, :, h]
    return out.reshape(psi.shape)


class _System:
    """The even-odd system of a case: Mhat, its adjoint, the hop and the fifth-dimension blocks."""

    def __init__(self, case, U):
        self.case, self.D = case, _Wilson4D(_lattice(case), U)
        self.dw = _is_dw(case)
        if self.dw:
            b5, c5 = _b5c5(case)
            Ls = case["Ls"]
            self.B = _fifth(Ls, b5, c5, MF)
            self.A = _fifth(Ls, (4 - M5) * b5 + 1, (4 - M5) * c5 - 1, MF)
            self.W = tuple(b @ torch.linalg.inv(a) for a, b in zip(self.A, self.B))
            self.Wt = tuple(w.T.contiguous() for w in self.W)
            self.Binv = tuple(torch.linalg.inv(b) for b in self.B)

    def mhat(self, v, dag=False):
        if not self.dw:
            k = self.case["kappa"]
            return v - k * k * self.D.hop(0, self.D.hop(1, v, dag), dag)
        if not dag:
            t = _apply5(self.W, self.D.hop(1, v))
            return v - 0.25 * _apply5(self.W, self.D.hop(0, t))
        t = self.D.hop(1, _apply5(self.Wt, v), True)
        return v - 0.25 * self.D.hop(0, _apply5(self.Wt, t), True)

    def _dot(self, a, b):
        """Inner products of each right-hand side, shaped to scale fields."""
        n = a.shape[0] // _ls(self.case)
        s = (a.conj() * b).reshape(n, -1).sum(1)
        return s.repeat_interleave(_ls(self.case)).reshape(-1, 1, 1, 1)

    def _krylov(self, b, dag, drop, most):
        """A correction of the single-precision system Mhat x = b: BiCGStab, or CG on the normal equations."""
        one = torch.ones((), dtype=b.dtype, device=DEV)

        def safe(z):
            return torch.where(z == 0, one, z)

        x = torch.zeros_like(b)
        if self.dw:
            r = self.mhat(b, not dag)
            p, rr = r.clone(), self._dot(r, r)
            stop = drop * drop * rr.real
            for it in range(most):
                q = self.mhat(self.mhat(p, dag), not dag)
                al = rr / safe(self._dot(p, q))
                x, r = x + al * p, r - al * q
                new = self._dot(r, r)
                if it % 4 == 3 and bool((new.real <= stop).all()):
                    break
                p, rr = r + (new / safe(rr)) * p, new
            return x
        r, rt = b.clone(), b.clone()
        p = r.clone()
        rho = self._dot(rt, r)
        stop = drop * drop * rho.real
        for it in range(most):
            v = self.mhat(p, dag)
            al = rho / safe(self._dot(rt, v))
            s = r - al * v
            t = self.mhat(s, dag)
            om = self._dot(t, s) / safe(self._dot(t, t))
            x = x + al * p + om * s
            r = s - om * t
            if it % 4 == 3 and bool((self._dot(r, r).real <= stop).all()):
                break
            new = self._dot(rt, r)
            p = r + (new / safe(rho)) * (al / safe(om)) * (p - om * v)
            rho = new
        return x

    def solve_even(self, b, dag=False):
        """Mhat x = b (Mhat^dag for dag) to the rounding of its residual."""
        x, last = torch.zeros_like(b), float("inf")
        r = b
        for _ in range(12):
            scale = r.abs().max()
            x = x + scale * self._krylov((r / scale).to(torch.complex64), dag, 2e-5, 400).to(torch.complex128)
            r = b - self.mhat(x, dag)
            rel = float((r.abs().square().sum() / b.abs().square().sum()).sqrt())
            if rel < 4e-16 or rel > 0.5 * last:
                break
            last = rel
        return x

    def solve(self, b, dag=False):
        """The full system on canonical (S, V, 4, 3)."""
        be, bo = self.D.split(b)
        if not self.dw:
            k = self.case["kappa"]
            xe = self.solve_even(be + k * self.D.hop(0, bo, dag), dag)
            return self.D.join(xe, bo + k * self.D.hop(1, xe, dag))
        xe = self.solve_even(_apply5(self.W, be + 0.5 * self.D.hop(0, _apply5(self.W, bo))))
        xo = _apply5(self.W, bo + 0.5 * self.D.hop(1, xe))
        return self.D.join(_apply5(self.Binv, xe), _apply5(self.Binv, xo))


def _internal(half, case):
    """(S, 4, 3, Vh) in the order of the FP32 / FP16 internal buffers: (nrhs, 6 spin pairs, Ls * Vh, 4 reals)."""
    S, vh, ls = half.shape[0], half.shape[3], _ls(case)
    v = half.reshape(S // ls, ls, 2, 2, 3, vh).permute(0, 2, 4, 1, 5, 3)  # rhs, half, colour, s, cb, spin of the pair
    v = v.reshape(S // ls, 6, ls * vh, 2)
    return torch.cat([v.real, v.imag], -1)


def _exact_apply(case, U, b):
    sy = _System(case, U)
    op, dag = case["op"], case["op"].endswith("DAG")
    S = b.shape[0] * _ls(case)
    e, o = sy.D.split(b.reshape(S, -1, 4, 3))
    if case["prec"] != "f64":
        # the operator acts on the field as it is stored in the input buffer
        e, o = _stored(e, case), _stored(o, case)
    if op == "D_EO":
        half = sy.D.hop(0, o)
    elif op == "D_OE":
        half = sy.D.hop(1, e)
    elif op.startswith("MHAT"):
        half = sy.mhat(e, dag)
    else:  # FULL, Wilson
        k = case["kappa"]
        return {"out": sy.D.join(e - k * sy.D.hop(0, o, dag), o - k * sy.D.hop(1, e, dag)).reshape(b.shape)}
    if case["prec"] == "f64":
        z = torch.zeros_like(half)
        return {"out": (sy.D.join(z, half) if op == "D_OE" else sy.D.join(half, z)).reshape(b.shape)}
    v = _internal(half, case)
    if case["prec"] == "f32":
        return {"out": v.reshape(-1)}
    scale = v.abs().amax(dim=(1, 3))  # (nrhs, Ls * Vh)
    n, _, sites, _ = v.shape
    h = (v / torch.where(scale == 0, 1.0, scale)[:, None, :, None]).reshape(n, 3, 2, sites, 4)
    return {"halves": h.permute(0, 1, 3, 2, 4).reshape(-1), "scale": scale.reshape(-1)}


def _stored(half, case):
    """A field's values after rounding to the case's storage."""
    if case["prec"] == "f32":
        return half.to(torch.complex64).to(torch.complex128)
    re, im = half.real.to(torch.float32), half.imag.to(torch.float32)
    s = torch.maximum(re.abs(), im.abs()).amax(dim=(1, 2), keepdim=True)
    inv = torch.where(s > 0, 1.0 / s, torch.zeros_like(s))

    def rnd(v):
        return (v * inv).to(torch.float16).to(torch.float64) * s.to(torch.float64)

    return torch.complex(rnd(re), rnd(im))


def _exact_md(case, U, P, phi, L):
    sy = _System(case, U)
    k = case["kappa"]
    pe, _ = sy.D.split(phi[None])
    Y = sy.solve_even(pe, True)
    X = sy.solve_even(Y)
    xi = sy.D.join(X, sy.D.hop(1, X))[0]
    eta = sy.D.join(Y, sy.D.hop(1, Y, True))[0]
    V = xi.shape[0]
    dS = torch.empty((4, V, 3, 3), dtype=torch.complex128, device=DEV)
    i = torch.arange(V, device=DEV)
    r, stride = i, 1
    for mu in range(4):
        xm, r = r % L[mu], r // L[mu]
        edge = xm == L[mu] - 1
        j = torch.where(edge, i - (L[mu] - 1) * stride, i + stride)
        stride *= L[mu]
        s = torch.where(edge, float(BC[mu]), 1.0).to(torch.float64) * (2 * k * k)
        (j0, c0), (j1, c1) = _Wilson4D.B[mu]
        b = torch.zeros((4, 4), dtype=torch.complex128, device=DEV)
        b[0, 2 + j0], b[1, 2 + j1] = c0, c1
        gamma = b + b.conj().T
        one = torch.eye(4, dtype=torch.complex128, device=DEV)
        # dS = s Re(eta(x)^dag (1 - gamma) dU xi(x + mu) + eta(x + mu)^dag (1 + gamma) dU^dag xi(x))
        em = torch.einsum("st,vta->vsa", one - gamma, eta)
        ep = torch.einsum("st,vta->vsa", one + gamma, eta[j])
        Fm = torch.einsum("vsa,vsb->vab", em.conj(), xi[j])
        G = torch.einsum("vsa,vsb->vab", xi, ep.conj())
        dS[mu] = s[:, None, None] * torch.complex(Fm.real + G.real, G.imag - Fm.imag)
    m = _mm(U.reshape(-1, 3, 3), dS.reshape(-1, 3, 3).conj().transpose(1, 2))
    a = 0.5 * (m - m.conj().transpose(1, 2))
    tr = (a[:, 0, 0] + a[:, 1, 1] + a[:, 2, 2]) / 3.0
    F = (a - tr[:, None, None] * torch.eye(3, dtype=a.dtype, device=DEV)).reshape(4, V, 3, 3)
    P1 = P + MD_EPS * F
    x = (MD_EPS * P1).reshape(-1, 3, 3)
    term = e = torch.eye(3, dtype=x.dtype, device=DEV).expand(x.shape)
    for n in range(1, 31):
        term = _mm(term, x) / n
        e = e + term
    U1 = _mm(e, U.reshape(-1, 3, 3)).reshape(U.shape)
    return {"dS": torch.view_as_real(dS), "P": P1, "U": U1, "energy": float(P1.abs().square().sum())}


def exact(case, seed):
    gen = _gen(seed)
    L = _lattice(case)
    V = int(np.prod(L))
    U = _links(case, gen)
    if case["kind"] == "md":
        phi = _gauss((V, 4, 3), gen)
        P = _momenta(V, gen)
        return _exact_md(case, U, P, phi * (_parity(L) == 0).to(torch.float64)[:, None, None], L)
    b = _source(case, gen)
    if case["kind"] == "apply":
        return _exact_apply(case, U, b)
    S = b.shape[0] * _ls(case)
    return {"x": _System(case, U).solve(b.reshape(S, V, 4, 3), case["dagger"]).reshape(b.shape)}
