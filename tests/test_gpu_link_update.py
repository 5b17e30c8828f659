"""exp(eps P) U on the GPU at the sizes where its series changes: zero, tiny, either side of the norms 0.1 and 0.5 that
choose the number of terms and the squarings, and general (not anti-Hermitian) matrices."""
import numpy as np
import pytest

from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _exp(a):
    """Taylor series with squarings in extended precision."""
    a = a.astype(np.clongdouble) / 2 ** 6
    e = t = np.broadcast_to(np.eye(3, dtype=np.clongdouble), a.shape)
    for n in range(1, 25):
        t = np.einsum("nij,njk->nik", t, a) / n
        e = e + t
    for _ in range(6):
        e = np.einsum("nij,njk->nik", e, e)
    return e


@pytest.mark.parametrize("norm", [0.0, 1e-9, 0.099, 0.101, 0.499, 0.501, 1.7])
@pytest.mark.parametrize("general", [False, True])
def test_link_update(norm, general):
    """1e-14 of the largest element: about 40 roundings of 1.1e-16, more with squarings (x 2 each)."""
    device()
    n = 700
    if general:
        rng = np.random.default_rng(5)
        P = rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))
    else:
        P = inputs.su3_momenta((n,), 6)
    P = P / np.sqrt((np.abs(P) ** 2).sum((1, 2), keepdims=True)) * norm
    U = inputs.gauge_field((2, 2, 4, 12), 0.5, 7).reshape(-1, 3, 3)[:n]
    Ud = to_dev(U)
    qcd.link_update(Ud, to_dev(P), 1.0)
    torch.cuda.synchronize()
    ref = np.einsum("nij,njk->nik", _exp(P), U.astype(np.clongdouble))
    assert np.abs(Ud.cpu().numpy() - ref).max() <= 1e-14 * np.abs(ref).max()
