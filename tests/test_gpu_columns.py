"""The fifth-dimension inverse held in registers, at the slice counts where it changes: fewest slices, odd counts, 16 (its
largest) and 17 and 33 (the shared-memory forms), ragged site blocks, Shamir and Mobius, both adjoints, all precisions.
Mhat's W enters as a kernel of its own (FP64; the adjoint in FP32 / FP16) and in the fused stencil (FP32 / FP16)."""
import numpy as np
import pytest

from oracle import oracle as ora
from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, max_err, rel_err, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)
TOL = {"f64": 1e-13, "f32": 1e-6, "f16": 2e-3}  # as the other operator tests


@pytest.mark.parametrize("Ls", [2, 3, 7, 16, 17, 33])
@pytest.mark.parametrize("b5,c5", [(1.0, 0.0), (1.5, 0.5)])
def test_mhat_over_slice_counts(Ls, b5, c5):
    device()
    L = (4, 2, 6, 2)
    V = int(np.prod(L))
    U = inputs.gauge_field(L, 0.3, 31)
    psi = inputs.gaussian_source((Ls, V, 4, 3), 32)
    pe = psi.copy()
    pe[:, ora.parity(L) == 1] = 0
    f = qcd.mobius(Ls, 1.8, 0.02, b5, c5) if c5 else qcd.dwf(Ls, 1.8, 0.02)
    g = qcd.Gauge.load(to_dev(U), L, BC, recon=12)
    out = torch.empty((Ls, V, 4, 3), dtype=torch.complex128, device=device())
    for dag in (False, True):
        ref = ora.mobius_mhat(L, BC, Ls, 1.8, 0.02, b5, c5, U, pe, dagger=dag)
        for prec, tol in TOL.items():
            qcd.dslash(g, f, "MHAT_DAG" if dag else "MHAT", to_dev(psi), out, prec=prec)
            torch.cuda.synchronize()
            assert (max_err if prec == "f64" else rel_err)(out, ref) < tol, (prec, dag)
    g.free()
