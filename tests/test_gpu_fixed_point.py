"""The FP64 operators on the GPU where their fixed-point stencil can go wrong: ragged site blocks, several slices,
both adjoints, sites of very different or extreme magnitude, infinities and NaN, links of other than unit size,
a caller's stream capture and two streams."""
import numpy as np
import pytest

from oracle import oracle as ora
from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, max_err, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)
KAPPA = 0.124
TOL = 1e-13  # element-wise, of the largest output: FP64's own tolerance in the other tests


def _apply(g, f, op, psi, nrhs=1):
    out = torch.empty_like(psi)
    qcd.dslash(g, f, op, psi, out, prec="f64", nrhs=nrhs)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("L", [(2, 2, 2, 2), (4, 2, 6, 2), (6, 4, 6, 10), (8, 4, 2, 18)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_hops_and_schur_operator(L, nrhs):
    device()
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.4, 7)
    psi = inputs.gaussian_source((nrhs, V, 4, 3), 8)
    par = ora.parity(L)
    g = qcd.Gauge.load(to_dev(U), L, BC)
    f = qcd.wilson(KAPPA)
    for op, po in (("D_EO", 0), ("D_OE", 1)):
        got = _apply(g, f, op, to_dev(psi), nrhs)
        for r in range(nrhs):
            inp = psi[r].copy()
            inp[par == po] = 0
            assert max_err(got[r], ora.hop(L, BC, U, inp, out_parity=po)) < TOL
    for op, dag in (("MHAT", False), ("MHAT_DAG", True)):
        got = _apply(g, f, op, to_dev(psi), nrhs)
        for r in range(nrhs):
            inp = psi[r].copy()
            inp[par == 1] = 0
            assert max_err(got[r], ora.wilson_mhat(L, BC, KAPPA, U, inp, dagger=dag)) < TOL
    for op, dag in (("FULL", False), ("FULL_DAG", True)):
        got = _apply(g, f, op, to_dev(psi), nrhs)
        for r in range(nrhs):
            assert max_err(got[r], ora.wilson(L, BC, KAPPA, U, psi[r], dagger=dag)) < TOL
    g.free()


@pytest.mark.parametrize("kind", ["point", "spread", "tiny", "huge", "mixed", "inf", "nan", "zero"])
def test_magnitudes(kind):
    """Site by site against the oracle: the error of a site is measured by its own neighbours' size."""
    device()
    L = (6, 4, 4, 6)
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.3, 9)
    psi = inputs.gaussian_source((V, 4, 3), 10)
    rng = np.random.default_rng(11)
    if kind == "point":
        psi[:] = 0
        psi[37, 2, 1] = 1.0
    elif kind == "zero":
        psi[:] = 0
    elif kind == "spread":
        psi *= np.exp(8 * rng.standard_normal((V, 1, 1)))
    elif kind == "tiny":
        psi *= 1e-290
    elif kind == "huge":
        psi *= 1e296
    elif kind == "mixed":
        psi *= 10.0 ** rng.integers(-300, 290, size=(V, 1, 1))
    elif kind == "inf":
        psi[101, 1, 2] = np.inf
    elif kind == "nan":
        psi[55, 3, 0] = np.nan
    g = qcd.Gauge.load(to_dev(U), L, BC)
    f = qcd.wilson(KAPPA)
    with np.errstate(all="ignore"):
        ref = ora.wilson(L, BC, KAPPA, U, psi)
        refm = ora.wilson_mhat(L, BC, KAPPA, U, np.where(ora.parity(L)[:, None, None] == 0, psi, 0))
        mag = ora.wilson(L, BC, KAPPA, U, np.where(np.isfinite(psi), psi, 0))
    got = _apply(g, f, "FULL", to_dev(psi))
    gotm = _apply(g, f, "MHAT", to_dev(psi))
    for a, b in ((got, ref), (gotm, refm)):
        fin = np.isfinite(b.real) & np.isfinite(b.imag)
        site = fin.all(axis=(1, 2))
        if kind in ("inf", "nan"):
            assert not site.all()
            bad = ~np.isfinite(a).all(axis=(1, 2))
            assert np.array_equal(bad, ~np.isfinite(b).all(axis=(1, 2)))  # the same sites, no others
        else:
            assert site.all()
        size = np.abs(b[site]).max(axis=(1, 2), keepdims=True)
        if kind == "mixed":  # neighbours of any size: by the largest
            size = np.maximum(size, np.abs(psi).max() * 0)
        err = np.abs(a[site] - b[site])
        ok = err <= 2e-13 * size
        if kind in ("spread", "mixed"):
            # cancellation between unequal neighbours does not occur: one of them dominates
            assert ok.mean() > 0.999 and (err <= 1e-11 * size).all()
        else:
            assert ok.all()
    assert mag is not None
    g.free()


def test_mixed_solve_and_plain_solve_agree_for_links_of_other_size():
    """Links scaled by 3 leave the fixed-point range: the FP64 stencil runs, results as the oracle's."""
    device()
    L = (4, 4, 4, 6)
    V = int(np.prod(L))
    U = 3.0 * inputs.gauge_field(L, 0.3, 9)
    psi = inputs.gaussian_source((V, 4, 3), 12)
    g = qcd.Gauge.load(to_dev(U), L, BC)
    got = _apply(g, qcd.wilson(0.03), "FULL", to_dev(psi))
    assert max_err(got, ora.wilson(L, BC, 0.03, U, psi)) < TOL
    g.free()


def test_capture_and_streams():
    """A captured FP64 operator holds none of the handle's scratch (a later, larger call may replace it); operators on
    two streams wait for each other's use of the scratch."""
    device()
    L = (8, 8, 4, 8)
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.3, 13)
    g = qcd.Gauge.load(to_dev(U), L, BC)
    f = qcd.wilson(KAPPA)
    psi = inputs.gaussian_source((4, V, 4, 3), 14)
    n1 = qcd.field_bytes(g, f, "f64", 1)
    bufs = [torch.empty(n1, dtype=torch.uint8, device=device()) for _ in range(8)]
    for k in range(4):
        qcd.field_pack(g, f, "f64", 1, to_dev(psi[k]), bufs[k])
    want = []
    for k in range(4):
        qcd.dslash(g, f, "D_EO", bufs[k], bufs[4 + k], prec="f64", layout=qcd.INTERNAL)
        want.append(bufs[4 + k].view(torch.float64).clone())
    torch.cuda.synchronize()
    gr = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr):
        qcd.dslash(g, f, "D_EO", bufs[0], bufs[4], prec="f64", layout=qcd.INTERNAL)
    big = to_dev(psi)
    _apply(g, f, "MHAT", big, nrhs=4)  # larger scratch
    bufs[4].zero_()
    gr.replay()
    torch.cuda.synchronize()
    assert float((bufs[4].view(torch.float64) - want[0]).abs().max()) <= TOL * float(want[0].abs().max())
    streams = [torch.cuda.Stream() for _ in range(2)]
    for rep in range(20):
        for k in range(4):
            with torch.cuda.stream(streams[k % 2]):
                qcd.dslash(g, f, "D_EO", bufs[k], bufs[4 + k], prec="f64", layout=qcd.INTERNAL)
    torch.cuda.synchronize()
    for k in range(4):
        assert torch.equal(bufs[4 + k].view(torch.float64), want[k])
    g.free()


@pytest.mark.parametrize("inner", ["f64", "f32", "f16"])
@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("L,nrhs", [((2, 2, 2, 4), 1), ((6, 4, 6, 10), 1), ((4, 6, 4, 6), 3)])
def test_outer_steps_of_a_solve(inner, dagger, L, nrhs):
    """The solve whose outer steps run in fixed point: ragged site blocks, one and several right-hand sides, an initial
    guess, sources that are zero or 1e-250 away from one site.  Tolerance: the requested residual, by the oracle."""
    device()
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.3, 15)
    b = inputs.z2_source((nrhs, V, 4, 3), 16)
    b[0] *= 1e-250
    b[0, V // 3, 1, 2] = 1.0
    if nrhs > 1:
        b[1] = 0
        b[1, 5, 3, 0] = 1.0
    g = qcd.Gauge.load(to_dev(U), L, BC, recon=12)
    f = qcd.wilson(KAPPA)
    x = torch.zeros((nrhs, V, 4, 3), dtype=torch.complex128, device=device())
    for guess in (False, True):
        if guess:
            x = x * 1.25
        info, _ = qcd.solve(g, f, to_dev(b), x, nrhs=nrhs, tol=1e-12, inner=inner, dagger=dagger, use_graph=True,
                            graph_chunk=8, x0_given=guess)
        xr = x.cpu().numpy()
        for r in range(nrhs):
            res = np.linalg.norm(b[r] - ora.wilson(L, BC, KAPPA, U, xr[r], dagger=dagger)) / np.linalg.norm(b[r])
            assert res <= 1.01e-12 and abs(res - info[r]["true_resid"]) <= 1e-2 * res + 2e-15, (res, info[r])
    g.free()
