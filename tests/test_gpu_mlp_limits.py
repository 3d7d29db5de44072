"""Emulator kernels away from the usual training step: devices without room for a
large cluster, many parameters, narrow networks and odd rows in large batches.

Values: as in test_gpu_mlp_tiles. Cost is compared within one tree. Adam moves 26
bytes a parameter where the conversion moves 6, so 4.3 times its time; twice that is
the bound (one cluster for every size took 16 times). A narrow network's pass reads
and writes little more than its output: bounds in copies of it (they took 20, 19 and 11, and 6, 8 and 5 now)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import mlp as om  # noqa: E402
from paper_1807_04215_gb300 import _lib  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402
from tests import inputs  # noqa: E402

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


@pytest.mark.parametrize("n", [1, 1000, 1024, 1025, 20000, 50001])
def test_loss_and_update_without_room_for_a_cluster(n, monkeypatch):
    """The injected device refuses every cluster of more than one block: the
    loss, its gradient and the update are those of the device that has room."""
    net = g.MLP(3, 128, 160, bf16=True, seed=1)
    gen = torch.Generator(device="cuda").manual_seed(n)
    y, t = (torch.randn(n, generator=gen, device="cuda") for _ in range(2))
    mask = (torch.rand(n, generator=gen, device="cuda") < 0.8).float()
    net.grad.copy_(torch.randn(net.n, generator=gen, device="cuda"))
    start = [b.clone() for b in (net.master, net.lowp, net.m, net.v, net.step)]

    def run():
        for b, s in zip((net.master, net.lowp, net.m, net.v, net.step), start):
            b.copy_(s)
        dy, loss = torch.empty_like(y), torch.zeros(1, device="cuda")
        net.mse(y, t, mask, dy, loss)
        net.adam(1e-3)
        return [b.clone() for b in (dy, loss, net.master, net.lowp, net.m, net.v, net.step)]

    ref = run()
    monkeypatch.setenv("GRIDSPT_FAULT_INJECT", "cluster")
    for a, b in zip(run(), ref, strict=True):
        assert torch.equal(a, b)


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


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("B,I,H,O", [(1, 3, 2, 1), (33, 1, 1, 256), (700, 3, 4, 4), (8200, 3, 16, 160), (8192, 8, 7, 35),
                                     (16385, 2, 33, 33), (32769, 3, 97, 21)])
def test_forward_of_narrow_and_odd_networks(bf16, B, I, H, O):
    net = g.MLP(I, H, O, bf16=bf16, seed=B)
    x = inputs.rng(B + H).standard_normal((B, I)).astype(np.float32)
    y_ref, _ = om.forward(x.astype(np.float64), net.master.double().cpu().numpy(), H, O,
                          om.bf16_round if bf16 else om.ident)
    act = torch.full((B, 4 * H), float("nan"), device="cuda")
    y = net.forward(torch.from_numpy(x).cuda(), act=act)
    assert torch.equal(y, net.forward(torch.from_numpy(x).cuda()))
    assert np.abs(y.double().cpu().numpy() - y_ref).max() <= (1e-2 if bf16 else 1e-5) * np.abs(y_ref).max()
    z, a = act.view(B, 2, 2, H).unbind(2)
    s = torch.nn.functional.silu(z)
    assert torch.allclose(a, s.bfloat16().float() if bf16 else s, rtol=2.0 ** -7 if bf16 else 1e-6, atol=1e-30)


@pytest.mark.parametrize("H,O,copies", [(1, 1, 12), (16, 16, 12), (16, 160, 8)])
def test_narrow_forward_in_copies_of_its_output(H, O, copies):
    B = 65536
    net = g.MLP(3, H, O, bf16=True, seed=1)
    x, y, z = torch.rand(B, 3, device="cuda"), torch.empty(B, O, device="cuda"), torch.empty(B, O, device="cuda")
    times = graph_time(lambda: net.forward(x, y=y)), graph_time(lambda: z.copy_(y))
    assert times[0] <= copies * times[1], times


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("B,I,H,O", [(16, 3, 1, 1), (65, 3, 16, 16), (64, 3, 16, 16), (1023, 2, 16, 9), (1024, 3, 16, 16),
                                     (4099, 3, 8, 100), (129, 3, 17, 1), (9000, 8, 64, 33), (2049, 3, 4, 4)])
def test_backward_in_row_parts_and_of_narrow_networks(bf16, B, I, H, O):
    """Sums over B rows in parts: against FP64, (B / 16 + 16) 2^-24 of the sum of
    magnitudes at worst, below 1e-5 of the largest gradient for these inputs with the
    factor that random signs leave (sqrt)."""
    net = g.MLP(I, H, O, bf16=bf16, seed=B)
    r = inputs.rng(B + H)
    x, dy = (r.standard_normal((B, k)).astype(np.float32) for k in (I, O))
    rnd = om.bf16_round if bf16 else om.ident
    theta = net.master.double().cpu().numpy()
    _, acts = om.forward(x.astype(np.float64), theta, H, O, rnd)
    act = torch.empty(B, 4 * H, device="cuda")
    xd, dyd = torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda()
    net.forward(xd, act=act)
    ws = torch.full((net.ws_bytes(B) + 4096,), 255, dtype=torch.uint8, device="cuda")
    net.grad.fill_(float("nan"))
    grad = net.backward(xd, act, dyd, ws[:net.ws_bytes(B)]).clone()
    assert bool((ws[net.ws_bytes(B):] == 255).all())
    assert torch.equal(grad, net.backward(xd, act, dyd, ws[:net.ws_bytes(B)]))
    ref = om.backward(x.astype(np.float64), theta, H, O, acts, dy.astype(np.float64), rnd)
    assert np.abs(grad.double().cpu().numpy() - ref).max() <= (1e-2 if bf16 else 1e-5) * np.abs(ref).max()


@pytest.mark.parametrize("H,O", [(16, 16), (16, 160)])
def test_narrow_backward_is_spread_over_the_rows(H, O):
    """A batch four times the size of one that leaves most of the GPU idle takes less than
    three times as long (one block a tile whatever the batch: 3.2 to 3.4)."""
    times = []
    for B in (1024, 4096):
        net = g.MLP(3, H, O, bf16=True, seed=1)
        x, dy = torch.rand(B, 3, device="cuda"), torch.randn(B, O, device="cuda")
        act = torch.empty(B, 4 * H, device="cuda")
        net.forward(x, act=act)
        ws = torch.empty(net.ws_bytes(B), dtype=torch.uint8, device="cuda")
        times.append(graph_time(lambda: net.backward(x, act, dy, ws)))
    assert times[1] <= 3 * times[0], times
