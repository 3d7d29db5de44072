"""Emulator kernels away from the usual training step: many parameters.

Cost is compared within one tree: Adam moves 26 bytes a parameter where the
conversion moves 6, so 4.3 times its time; twice that is the bound (one cluster
for every size took 20 times)."""
import math

import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1807_04215_gb300 import _lib  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402

pytestmark = pytest.mark.gpu


def graph_time(f, calls=20, rounds=7):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f()
    torch.cuda.synchronize()
    gr = torch.cuda.CUDAGraph()
    with torch.cuda.graph(gr, stream=s):
        for _ in range(calls):
            f()
    best = math.inf
    for _ in range(rounds):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        gr.replay()
        a.record()
        gr.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / calls)
    return best


def test_update_of_many_parameters_takes_the_whole_gpu():
    n = 1 << 20
    lib = _lib.load()
    master, grad, m, v = (torch.zeros(n, device="cuda") for _ in range(4))
    low, step = torch.zeros(n, dtype=torch.bfloat16, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")

    def stream():
        return torch.cuda.current_stream().cuda_stream

    def adam():
        assert lib.gridspt_mlp_adam(master.data_ptr(), low.data_ptr(), 1, grad.data_ptr(), m.data_ptr(), v.data_ptr(),
                                    step.data_ptr(), n, 1e-3, 0.9, 0.999, 1e-8, stream()) == 0

    def convert():
        assert lib.gridspt_mlp_convert(master.data_ptr(), low.data_ptr(), 1, n, stream()) == 0

    times = graph_time(adam), graph_time(convert)
    assert times[0] <= 9 * times[1], times
