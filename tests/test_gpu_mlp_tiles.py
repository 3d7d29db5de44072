"""Emulator kernels at the edges of their tiles: row tiles of 2, 8 and 32 with
remainders, odd widths (unaligned weight rows), weights larger than one shared
buffer, and networks whose backward scratch holds only part of the batch.

Bounds: FP32 chains of K <= 256 terms against FP64, (K + 3) 2^-24 of the sum of
magnitudes, stays below 1e-5 of the largest value for these inputs; bfloat16
weights are compared with the FP64 network on the same rounded weights, where a
hidden value next to a rounding boundary may differ by one bfloat16 step (2^-8
of it): 1e-2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import mlp as om  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402
from tests import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("B,I,H,O", [(1, 3, 128, 160), (3, 1, 1, 1), (50, 2, 4, 3), (609, 3, 97, 31), (2433, 5, 64, 20),
                                     (700, 3, 256, 256), (257, 8, 255, 1)])
def test_forward_backward_tiles(bf16, B, I, H, O):
    net = g.MLP(I, H, O, bf16=bf16, seed=B)
    r = inputs.rng(B + H)
    x = r.standard_normal((B, I)).astype(np.float32)
    dy = r.standard_normal((B, O)).astype(np.float32)
    rnd = om.bf16_round if bf16 else om.ident
    theta = net.master.double().cpu().numpy()
    y_ref, acts = om.forward(x.astype(np.float64), theta, H, O, rnd)
    act = torch.empty(B, 4 * H, device="cuda")
    y = net.forward(torch.from_numpy(x).cuda(), act=act)
    tol = 1e-2 if bf16 else 1e-5
    assert np.abs(y.double().cpu().numpy() - y_ref).max() <= tol * np.abs(y_ref).max()
    ws = torch.empty(net.ws_bytes(B), dtype=torch.uint8, device="cuda")
    net.grad.fill_(float("nan"))
    grad = net.backward(torch.from_numpy(x).cuda(), act, torch.from_numpy(dy).cuda(), ws).double().cpu().numpy()
    ref = om.backward(x.astype(np.float64), theta, H, O, acts, dy.astype(np.float64), rnd)
    assert np.abs(grad - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 31, 1024, 8193, 50001])
def test_mse_sums_every_element(n):
    r = inputs.rng(n)
    y, t = (r.standard_normal(n).astype(np.float32) for _ in range(2))
    m = (r.random(n) < 0.8).astype(np.float32)
    net = g.MLP(1, 1, 1, bf16=False)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    dy, loss = torch.empty(n, device="cuda"), torch.zeros(1, device="cuda")
    net.mse(dev(y), dev(t), dev(m), dy, loss)
    L, d = om.masked_mse(y.astype(np.float64), t.astype(np.float64), m.astype(np.float64)) if m.sum() else (0.0, 0 * m)
    assert abs(loss.item() - L) <= 1e-5 * L
    assert np.abs(dy.cpu().numpy() - d).max() <= 1e-5 * max(np.abs(d).max(), 1e-30)


def test_networks_of_different_widths_run_from_two_threads():
    """The kernels' shared memory differs with the width: a thread's launch must
    not depend on the width of the network that another thread launches."""
    from concurrent.futures import ThreadPoolExecutor

    def run(H):
        with torch.cuda.stream(torch.cuda.Stream()):
            net = g.MLP(3, H, 20, bf16=False, seed=H)
            x = torch.from_numpy(inputs.rng(H).standard_normal((40, 3)).astype(np.float32)).cuda()
            ref = net.forward(x)
            return all(bool(torch.equal(net.forward(x), ref)) for _ in range(200))

    with ThreadPoolExecutor(2) as pool:
        assert all(pool.map(run, (8, 256)))
