"""Which streams the FP64 operators on internal buffers wait for: none but the last user of their own scratch, and that
one whatever became of its stream."""
import ctypes

import numpy as np
import pytest

from paper_1712_01505_gb300 import inputs, qcd
from tests.gpu_util import device, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (1, 1, 1, -1)
L = (8, 8, 8, 8)
V = int(np.prod(L))
SLEEP = 400_000_000  # clock cycles, about 0.2 s


def _setup(n):
    device()
    g = qcd.Gauge.load(to_dev(inputs.gauge_field(L, 0.3, 61)), L, BC)
    f = qcd.wilson(0.12)
    size = qcd.field_bytes(g, f, "f64", 1)
    ins, outs = [], []
    for k in range(n):
        b = torch.empty(size, dtype=torch.uint8, device=device())
        qcd.field_pack(g, f, "f64", 1, to_dev(inputs.gaussian_source((V, 4, 3), 62 + k)), b)
        ins.append(b)
        outs.append(torch.zeros(size, dtype=torch.uint8, device=device()))

    def hop(k, stream=None):
        qcd.dslash(g, f, "D_EO", ins[k], outs[k], prec="f64", layout=qcd.INTERNAL, stream=stream)

    want = []
    for k in range(n):  # tuned, and what each stream has to find
        hop(k)
        torch.cuda.synchronize()
        want.append(outs[k].clone())
        outs[k].zero_()
    return g, hop, outs, want


def test_streams_do_not_wait_for_each_other():
    g, hop, outs, want = _setup(2)
    s = [torch.cuda.Stream() for _ in range(2)]
    for k in range(2):  # both sets of scratch are there
        hop(k, s[k].cuda_stream)
    torch.cuda.synchronize()
    ev = torch.cuda.Event()
    with torch.cuda.stream(s[0]):
        torch.cuda._sleep(SLEEP)
        hop(0, s[0].cuda_stream)
        ev.record()
    hop(1, s[1].cuda_stream)
    s[1].synchronize()
    assert not ev.query()  # the first one is still asleep
    torch.cuda.synchronize()
    for k in range(2):
        assert torch.equal(outs[k], want[k])
    g.free()


def test_a_stream_destroyed_with_its_work_pending():
    """Twelve streams one after the other, each destroyed before its operator has run: the next one is created at the
    same address as often as not."""
    n = 12
    g, hop, outs, want = _setup(n)
    rt = ctypes.CDLL("libcudart.so.13")
    seen = []
    for k in range(n):
        p = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(p), 1) == 0
        seen.append(p.value)
        with torch.cuda.stream(torch.cuda.ExternalStream(p.value)):
            torch.cuda._sleep(SLEEP // 20)
        hop(k, p.value)
        assert rt.cudaStreamDestroy(p) == 0
    torch.cuda.synchronize()
    for k in range(n):
        assert torch.equal(outs[k], want[k]), (k, seen)
    g.free()


def test_more_streams_than_sets_of_scratch():
    n = 9
    g, hop, outs, want = _setup(n)
    s = [torch.cuda.Stream() for _ in range(n)]
    for rep in range(3):
        for k in range(n):
            with torch.cuda.stream(s[k]):
                torch.cuda._sleep(SLEEP // 200)
            hop(k, s[k].cuda_stream)
        torch.cuda.synchronize()
        for k in range(n):
            assert torch.equal(outs[k], want[k])
            outs[k].zero_()
    g.free()
