"""Each component of the FP64 operators against extended precision, measured by its own products and not by the
largest output: links that mix the colours (interacting fields) and links that hardly do or not at all (weak, free, Abelian,
block-diagonal fields), inputs whose components or sites differ by many orders of magnitude."""
import numpy as np
import pytest

from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)
KAPPA = 0.124
L = (6, 4, 4, 6)
V = int(np.prod(L))
# Of S = sum |U| |h| over the products of a component.  Where the fixed-point sum is taken its error is 5.4 2^-53 S rms at
# most (csrc/fixed.cuh), 27 at five standard deviations; where FP64 is, at most 16 2^-53 S (a chain of 14
# additions, one product and the projection): 2^-48 = 32 2^-53 holds for both.
TOL = 2.0 ** -48

# B of (1 - gamma_mu) = (1, B; B^dag, 1): row -> (column, factor)
B = {0: ((1, -1j), (0, -1j)), 1: ((1, -1), (0, 1)), 2: ((0, -1j), (1, 1j)), 3: ((0, 1), (1, 1))}


def _neighbours():
    i = np.arange(V)
    x, r = [], i
    for m in range(4):
        x.append(r % L[m])
        r = r // L[m]
    out, stride = {}, 1
    for mu in range(4):
        for d in (1, -1):
            edge = x[mu] == (L[mu] - 1 if d > 0 else 0)
            out[mu, d] = (np.where(edge, i - d * (L[mu] - 1) * stride, i + d * stride), np.where(edge, BC[mu], 1))
        stride *= L[mu]
    return out, (x[0] + x[1] + x[2] + x[3]) % 2


NB, PAR = _neighbours()


def _hop(U, psi, dag=False):
    """H psi and S (as complex: of the real and of the imaginary parts), extended precision."""
    U, psi = U.astype(np.clongdouble), psi.astype(np.clongdouble)
    out, S = np.zeros_like(psi), np.zeros_like(psi)

    def mag(u, h):  # |re| |re| + |im| |im| and |re| |im| + |im| |re|
        ar, ai, hr, hi = np.abs(u.real), np.abs(u.imag), np.abs(h.real), np.abs(h.imag)
        return (np.einsum("xab,xsb->xsa", ar, hr) + np.einsum("xab,xsb->xsa", ai, hi)
                + 1j * (np.einsum("xab,xsb->xsa", ar, hi) + np.einsum("xab,xsb->xsa", ai, hr)))

    for mu in range(4):
        (j0, c0), (j1, c1) = B[mu]
        for d in (1, -1):
            sg = (-1 if d > 0 else 1) * (-1 if dag else 1)
            n, sign = NB[mu, d]
            g = psi[n] * sign[:, None, None]
            h = np.stack([g[:, 0] + sg * c0 * g[:, 2 + j0], g[:, 1] + sg * c1 * g[:, 2 + j1]], 1)
            u = U[mu] if d > 0 else U[mu][n].conj().transpose(0, 2, 1)
            w, m = np.einsum("xab,xsb->xsa", u, h), mag(u, h)
            out[:, :2] += w
            S[:, :2] += m
            for k, (j, c) in enumerate(((j0, c0), (j1, c1))):
                out[:, 2 + j] += sg * np.conj(c) * w[:, k]
                S[:, 2 + j] += m[:, k] if np.imag(c) == 0 else m[:, k].imag + 1j * m[:, k].real
    return out, S


def _half(v, p):
    return np.where((PAR == p)[:, None, None], v, 0)


def _reach(U, S):
    """sum |U| (|u| + |l|) of a magnitude field: what an error of its components may become"""
    tot = np.zeros_like(S)
    for mu in range(4):
        for d in (1, -1):
            n, _ = NB[mu, d]
            g = S[n]
            u = U[mu] if d > 0 else U[mu][n].conj().transpose(0, 2, 1)
            a, both = np.abs(u.real) + np.abs(u.imag), g.real + g.imag
            for s in (0, 1):
                j = B[mu][s][0]
                m = np.einsum("xab,xb->xa", a, both[:, s] + both[:, 2 + j])
                tot[:, s] += m * (1 + 1j)
                tot[:, 2 + j] += m * (1 + 1j)
    return tot


def _links(kind):
    rng = np.random.default_rng(21)
    if kind == "interacting":
        return inputs.gauge_field(L, 0.3, 22)
    if kind == "weak":
        return inputs.gauge_field(L, 1e-4, 23)
    U = np.zeros((4, V, 3, 3), complex)
    if kind == "free":
        U[:] = np.eye(3)
    elif kind == "abelian":
        a = rng.uniform(-np.pi, np.pi, (4, V, 2))
        for k, p in enumerate((a[..., 0], a[..., 1], -a[..., 0] - a[..., 1])):
            U[..., k, k] = np.exp(1j * p)
    else:  # an SU(2) block
        q = rng.standard_normal((4, V, 4))
        q /= np.linalg.norm(q, axis=-1, keepdims=True)
        a, b = q[..., 0] + 1j * q[..., 1], q[..., 2] + 1j * q[..., 3]
        U[..., 0, 0], U[..., 0, 1], U[..., 1, 0], U[..., 1, 1] = a, b, -b.conj(), a.conj()
        U[..., 2, 2] = 1
    return U


def _field(kind):
    rng = np.random.default_rng(24)
    psi = inputs.gaussian_source((V, 4, 3), 25)
    if kind == "colours":
        psi *= np.array([1.0, 1e-9, 1e-17])
    elif kind == "spins":
        psi *= np.array([1e-8, 1.0, 1e-30, 1e-4])[:, None]
    elif kind == "imaginary":
        psi = psi.real + 1e-12j * psi.imag
    elif kind == "components":
        psi *= 10.0 ** rng.uniform(-20, 0, psi.shape)
    elif kind == "sites":
        psi *= 2.0 ** rng.integers(-140, 0, (V, 1, 1))
    elif kind == "decay":
        psi *= 0.2 ** (np.abs(np.arange(V) - 200) / 4)[:, None, None]
    elif kind == "point":
        psi[:] = 0
        psi[37, 2, 1] = 1.0
    elif kind == "wall":
        psi[:] = 0
        psi[:, 1, 0] = 1.0
    return psi


def _close(got, want, bound, what):
    for part in ("real", "imag"):
        err = np.abs(getattr(got, part) - getattr(want, part))
        b = getattr(bound, part)
        assert (err <= b).all(), (what, part, (err <= b).mean(), err[err > b].max(), b[err > b].min())


@pytest.mark.parametrize("links", ["interacting", "weak", "free", "abelian", "block"])
@pytest.mark.parametrize("field", ["gauss", "colours", "spins", "imaginary", "components", "sites", "decay", "point", "wall"])
def test_components(links, field):
    device()
    U, psi = _links(links), _field(field)
    g = qcd.Gauge.load(to_dev(U), L, BC)
    f = qcd.wilson(KAPPA)
    d = to_dev(psi)

    def apply(op):
        out = torch.empty_like(d)
        qcd.dslash(g, f, op, d, out, prec="f64")
        torch.cuda.synchronize()
        return out.cpu().numpy()

    for po, op in ((0, "D_EO"), (1, "D_OE")):
        ref, S = _hop(U, _half(psi, 1 - po))
        _close(apply(op), _half(ref, po), TOL * _half(S, po), op)
        # the same through an internal buffer, as the second of two right-hand sides
        n = qcd.field_bytes(g, f, "f64", 2)
        bi, bo = (torch.empty(n, dtype=torch.uint8, device=d.device) for _ in range(2))
        two, res = torch.stack([torch.flip(d, [0]), d]), torch.zeros((2,) + d.shape, dtype=d.dtype, device=d.device)
        qcd.field_pack(g, f, "f64", 1 - po, two, bi, nrhs=2)
        qcd.dslash(g, f, op, bi, bo, prec="f64", nrhs=2, layout=qcd.INTERNAL)
        qcd.field_unpack(g, f, "f64", po, bo, res, nrhs=2)
        torch.cuda.synchronize()
        _close(res[1].cpu().numpy(), _half(ref, po), TOL * _half(S, po), op + " internal")
    for dag, op in ((False, "FULL"), (True, "FULL_DAG")):
        ref, S = _hop(U, psi, dag)
        ref = psi - KAPPA * ref
        size = np.abs(psi.real) + np.abs(ref.real) + 1j * (np.abs(psi.imag) + np.abs(ref.imag))
        _close(apply(op), ref, TOL * KAPPA * S + 2.0 ** -52 * size, op)  # the last addition
    for dag, op in ((False, "MHAT"), (True, "MHAT_DAG")):
        e = _half(psi, 0)
        t, S1 = _hop(U, e, dag)
        h, S2 = _hop(U, _half(t, 1), dag)
        ref = e - KAPPA ** 2 * _half(h, 0)
        # an error of TOL S1 in the intermediate spreads with |U|; the second hop has its own
        bound = TOL * KAPPA ** 2 * (_half(S2, 0) + _half(_reach(U, _half(S1, 1)), 0))
        size = np.abs(e.real) + np.abs(ref.real) + 1j * (np.abs(e.imag) + np.abs(ref.imag))
        _close(apply(op), ref, bound + 2.0 ** -52 * size, op)
    g.free()


@pytest.mark.parametrize("links", ["interacting", "free", "abelian"])
@pytest.mark.parametrize("field", ["colours", "spins", "components"])
@pytest.mark.parametrize("dagger", [False, True])
def test_reconstructed_half_of_a_solve(links, field, dagger):
    """A solve that takes its initial guess as it is returns the odd half b_o + kappa H_oe x_e of its outer step."""
    device()
    U, x0 = _links(links), _field(field)
    b = _half(inputs.gaussian_source((V, 4, 3), 27), 0)  # b_o = 0: nothing hides the components of H_oe x_e
    g = qcd.Gauge.load(to_dev(U), L, BC)
    x = to_dev(x0)
    qcd.solve(g, qcd.wilson(KAPPA), to_dev(b), x, tol=1e30, inner="f32", x0_given=True, dagger=dagger)
    h, S = _hop(U, _half(x0, 0), dagger)
    got = x.cpu().numpy()
    assert np.array_equal(_half(got, 0), _half(x0, 0))
    _close(_half(got, 1), KAPPA * _half(h, 1), KAPPA * (TOL * _half(S, 1) + 2.0 ** -52 * np.abs(_half(h, 1))), "odd half")
    g.free()


@pytest.mark.parametrize("inner", ["f64", "f32", "f16"])
@pytest.mark.parametrize("scale", [3.0, 0.3])
def test_solves_on_links_of_other_size(inner, scale):
    """Links outside the fixed-point range: plain and mixed solves on the FP64 kernels, judged in extended precision."""
    device()
    U = scale * _links("interacting")
    kappa = 0.1 / scale
    b = inputs.gaussian_source((V, 4, 3), 28)
    g = qcd.Gauge.load(to_dev(U), L, BC)
    x = torch.zeros((V, 4, 3), dtype=torch.complex128, device=device())
    info, _ = qcd.solve(g, qcd.wilson(kappa), to_dev(b), x, tol=1e-12, inner=inner, use_graph=True)
    x = x.cpu().numpy()
    res = np.linalg.norm(b - (x - kappa * _hop(U, x)[0])) / np.linalg.norm(b)
    assert res <= 1.01e-12 and abs(res - info[0]["true_resid"]) <= 1e-2 * res + 2e-15
    g.free()
