"""exa_stat("eval_kernel_ms") waits for the call it reports and for nothing else."""
import threading
import time

import pytest
import torch

import synth
from paper_2608_16265_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture
def stepped():
    w = synth.rosenbrock(1000)
    m = B.exa_create(w.flat)
    x, y, s = synth.rosenbrock_point(w, 0)
    X, Y = torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda")
    out = m.eval_all(X, Y, s)
    for _ in range(3):
        m.exa_eval_all(X, Y, s, **out)
    return m


def test_other_streams_are_not_waited_for(stepped):
    assert 0 < stepped.stat("eval_kernel_ms") < 10
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2_000_000_000)  # about a second
    t = time.perf_counter()
    ms = stepped.stat("eval_kernel_ms")
    t = time.perf_counter() - t
    assert not side.query() and t < 0.3 and 0 < ms < 10
    side.synchronize()


def test_a_capture_elsewhere_survives(stepped):
    got = []
    a = torch.ones(1000, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, capture_error_mode="global"):
        b = a + 1
        th = threading.Thread(target=lambda: got.append(stepped.stat("eval_kernel_ms")))
        th.start()
        th.join()
        c = b * 2
    g.replay()
    torch.cuda.synchronize()
    assert 0 < got[0] < 10 and float(c[0]) == 4.0
