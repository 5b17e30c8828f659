"""The iteration's inner products where their partial sums change shape: one or several groups of a slice's
per-warp sums, partials summed by one warp or by the block."""
import numpy as np
import pytest

from oracle import oracle as ora
from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)


@pytest.mark.parametrize("L", [(4, 4, 4, 6), (8, 8, 8, 16), (16, 16, 16, 16), (16, 16, 16, 64)])
@pytest.mark.parametrize("inner", ["f32", "f16", "f64"])
def test_bicgstab_alone_and_side_by_side(L, inner):
    """One right-hand side (group sums of the stencil) and the same twice beside another (per-warp sums in groups, or
    separate reductions): the residual asked for, by the oracle, and as many iterations.  A sum that misses a part leaves
    x and r consistent but loses the convergence; rounding alone moves the count by one or two in thirty."""
    device()
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.25, 21)
    b = inputs.z2_source((3, V, 4, 3), 22)
    b[2] = b[0]
    g = qcd.Gauge.load(to_dev(U), L, BC, recon=12)
    f = qcd.wilson(0.12)
    count = {}
    for nrhs in (1, 3):
        bs = to_dev(b[:nrhs])
        x = torch.zeros_like(bs)
        info, _ = qcd.solve(g, f, bs, x, nrhs=nrhs, tol=1e-10, inner=inner, use_graph=True)
        xr = x.cpu().numpy()
        for r in range(nrhs):
            res = np.linalg.norm(b[r] - ora.wilson(L, BC, 0.12, U, xr[r])) / np.linalg.norm(b[r])
            assert res <= 1.01e-10, (nrhs, r, res)
        count[nrhs] = info[0]["iters"]
        if nrhs == 3:
            assert abs(info[2]["iters"] - info[0]["iters"]) == 0
    assert abs(count[1] - count[3]) <= max(2, count[1] // 10), count
    g.free()


@pytest.mark.parametrize("L,Ls", [((4, 4, 4, 4), 8), ((8, 8, 8, 8), 4), ((16, 16, 16, 16), 4), ((8, 8, 8, 16), 20)])
@pytest.mark.parametrize("inner", ["f32", "f16"])
def test_cg_slices(L, Ls, inner):
    """Domain-wall CG: the slices' sums in one or several groups, against the same solve in FP64 (separate reductions)."""
    device()
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.2, 23)
    b = to_dev(inputs.z2_source((Ls, V, 4, 3), 24))
    g = qcd.Gauge.load(to_dev(U), L, BC, recon=12)
    f = qcd.dwf(Ls, 1.8, 0.1)
    out = {}
    for prec in (inner, "f64"):
        x = torch.zeros_like(b)
        info, _ = qcd.solve(g, f, b, x, method=qcd.CG_NORMAL, tol=1e-9, inner=prec, use_graph=True)
        out[prec] = (x, info[0]["iters"])
    d = float((out[inner][0] - out["f64"][0]).norm() / out["f64"][0].norm())
    assert d <= 1e-6, d  # two solutions of residual 1e-9, condition number of a few hundred
    assert out[inner][1] <= 1.5 * out["f64"][1] + 4, (out[inner][1], out["f64"][1])  # restarts cost some
    g.free()
