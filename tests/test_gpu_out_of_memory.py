"""Allocations that CUDA refuses (a request larger than the device, QCD_FAULT=oom): the fixed-point form of the links and
its scratch are for speed only, so every call answers without them what it answers with them."""
import numpy as np
import pytest

from oracle import oracle as ora
from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, max_err, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)
KAPPA = 0.12
L = (6, 4, 4, 8)
V = int(np.prod(L))
TOL = 1e-13  # of the largest output, as in the other FP64 tests


def _load(seed):
    U = inputs.gauge_field(L, 0.3, seed)
    return U, qcd.Gauge.load(to_dev(U), L, BC)


def _internal(g, f, psi, nrhs):
    """D_EO on an internal buffer: needs no workspace in FP64."""
    n = qcd.field_bytes(g, f, "f64", nrhs)
    bi, bo = (torch.zeros(n, dtype=torch.uint8, device=device()) for _ in range(2))
    qcd.field_pack(g, f, "f64", 1, psi, bi, nrhs=nrhs)
    qcd.dslash(g, f, "D_EO", bi, bo, prec="f64", nrhs=nrhs, layout=qcd.INTERNAL)
    out = torch.zeros_like(psi)
    qcd.field_unpack(g, f, "f64", 0, bo, out, nrhs=nrhs)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _check_hop(U, got, psi, nrhs):
    odd = ora.parity(L)[:, None, None] == 1
    for r in range(nrhs):
        assert max_err(got[r], ora.hop(L, BC, U, np.where(odd, psi[r], 0), out_parity=0)) < TOL


def test_operator_without_its_scratch(monkeypatch):
    device()
    U, g = _load(31)
    f = qcd.wilson(KAPPA)
    psi = inputs.gaussian_source((3, V, 4, 3), 32)
    d = to_dev(psi)
    monkeypatch.setenv("QCD_FAULT", "oom")
    for nrhs in (1, 3):  # no scratch at all; none that is large enough
        _check_hop(U, _internal(g, f, d[:nrhs].contiguous(), nrhs), psi, nrhs)
        out = torch.empty_like(d[:nrhs])
        for op, dag in (("FULL", False), ("FULL_DAG", True)):
            qcd.dslash(g, f, op, d[:nrhs].contiguous(), out, prec="f64", nrhs=nrhs)
            torch.cuda.synchronize()
            for r in range(nrhs):
                assert max_err(out[r], ora.wilson(L, BC, KAPPA, U, psi[r], dagger=dag)) < TOL
        monkeypatch.delenv("QCD_FAULT")
        _check_hop(U, _internal(g, f, d[:nrhs].contiguous(), nrhs), psi, nrhs)
        monkeypatch.setenv("QCD_FAULT", "oom")
    g.free()


def test_links_loaded_without_their_fixed_point_form(monkeypatch):
    device()
    monkeypatch.setenv("QCD_FAULT", "oom")
    U, g = _load(33)
    monkeypatch.delenv("QCD_FAULT")
    psi = inputs.gaussian_source((1, V, 4, 3), 34)
    _check_hop(U, _internal(g, qcd.wilson(KAPPA), to_dev(psi), 1), psi, 1)
    g.free()


@pytest.mark.parametrize("inner,method", [("f64", qcd.BICGSTAB), ("f32", qcd.BICGSTAB), ("f16", qcd.BICGSTAB),
                                          ("f64", qcd.CG_NORMAL), ("f32", qcd.CG_NORMAL)])
@pytest.mark.parametrize("nrhs", [1, 2])
def test_solve_whose_allocations_take_the_links_back(monkeypatch, inner, method, nrhs):
    device()
    U, g = _load(35)
    f = qcd.wilson(KAPPA)
    b = inputs.gaussian_source((nrhs, V, 4, 3), 36)

    def check(x):
        for r in range(nrhs):
            res = np.linalg.norm(b[r] - ora.wilson(L, BC, KAPPA, U, x[r])) / np.linalg.norm(b[r])
            assert res <= 1.01e-11

    x = torch.zeros(b.shape, dtype=torch.complex128, device=device())
    for fault in (None, "oom", None):  # before, while and after the vectors for more right-hand sides are allocated
        if fault:
            monkeypatch.setenv("QCD_FAULT", fault)
            b2 = np.concatenate([b, b])
            y = torch.zeros(b2.shape, dtype=torch.complex128, device=device())
            qcd.solve(g, f, to_dev(b2), y, nrhs=2 * nrhs, tol=1e-11, inner=inner, method=method, use_graph=True)
            y = y.cpu().numpy()
            monkeypatch.delenv("QCD_FAULT")
            check(y[:nrhs])
            check(y[nrhs:])
        else:
            qcd.solve(g, f, to_dev(b), x.zero_(), nrhs=nrhs, tol=1e-11, inner=inner, method=method, use_graph=True)
            check(x.cpu().numpy())
    g.free()


def test_another_handle_gives_its_links_back(monkeypatch):
    """An allocation that only fits without the fixed-point links of an idle handle gets their memory; that handle
    answers as before."""
    device()
    big = (16, 16, 16, 16)
    Vb = int(np.prod(big))
    Ub = inputs.gauge_field(big, 0.3, 37)
    U, g = _load(38)
    gb = qcd.Gauge.load(to_dev(Ub), big, BC)
    f = qcd.wilson(KAPPA)
    psi = inputs.gaussian_source((Vb, 4, 3), 39)
    d = to_dev(psi)
    ref = ora.wilson(big, BC, KAPPA, Ub, psi)

    def full():
        out = torch.empty_like(d)
        qcd.dslash(gb, f, "FULL", d, out, prec="f64")
        torch.cuda.synchronize()
        return max_err(out, ref)

    assert full() < TOL
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    monkeypatch.setenv("QCD_FAULT", "oom")
    b = to_dev(inputs.gaussian_source((V, 4, 3), 40))
    x = torch.zeros_like(b)
    qcd.solve(g, f, b, x, tol=1e-10, inner="f32")  # a lattice of 768 sites
    monkeypatch.delenv("QCD_FAULT")
    assert torch.cuda.mem_get_info()[0] - free >= 1152 * Vb // 2  # 1152 bytes per site came back, a little was used
    assert full() < TOL
    x = torch.zeros_like(d)
    qcd.solve(gb, f, d, x, tol=1e-11, inner="f64", use_graph=True)
    res = np.linalg.norm(psi - ora.wilson(big, BC, KAPPA, Ub, x.cpu().numpy())) / np.linalg.norm(psi)
    assert res <= 1.01e-11
    g.free()
    gb.free()


def test_handles_of_two_threads(monkeypatch):
    """While a call uses a handle, no other thread's allocation takes its links."""
    import threading

    dev = device()
    f = qcd.wilson(KAPPA)
    sets, errors = [_load(41 + k) for k in range(2)], []
    monkeypatch.setenv("QCD_FAULT", "oom")

    def work(k):
        try:
            U, g = sets[k]
            stream = torch.cuda.Stream(dev)
            with torch.cuda.stream(stream):
                for rep in range(6):
                    n = 1 + (rep + k) % 3
                    b = inputs.gaussian_source((n, V, 4, 3), 50 + rep)
                    x = torch.zeros(b.shape, dtype=torch.complex128, device=dev)
                    src = to_dev(b)
                    qcd.solve(g, f, src, x, nrhs=n, tol=1e-11, inner="f64")
                    out = torch.empty_like(x)
                    qcd.dslash(g, f, "FULL", x, out, prec="f64", nrhs=n)
                    stream.synchronize()
                    for r in range(n):
                        assert max_err(out[r], b[r]) < 1e-9
                    if rep == 3:  # loaded again, with its fixed-point form
                        g.free()
                        g = qcd.Gauge.load(to_dev(U), L, BC)
            g.free()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
