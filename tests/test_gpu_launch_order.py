"""Programmatically dependent launches: order and cost.

Order: every kernel waits for the whole previous kernel of its stream. Calls
queued back to back, each overwriting what the one before it reads, writes or
leaves in shared buffers, give what the same calls give with a synchronisation
after each.
Cost: a plan's default pass variants are not slower than its tile variants where
launches are short. Blocks let in too early lie unevenly on the SMs: the fifth-order
recursion at 96^3 took 1.15 times the tile variants' time then, 0.91 without; bound 1.08."""
import math

import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1807_04215_gb300 import gridspt as g  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 64, 96, 128])
def test_back_to_back_calls_equal_synchronised_ones(N):
    L, kF = 4.0 * N, 2.0 * math.pi / (4.0 * N)
    plan = g.Plan(N, 3, L)
    net = g.MLP(3, 64, 40, bf16=True, seed=1)
    edges = [kF * (0.5 + i) for i in range(9)]
    x = torch.empty(N, N, N, device="cuda")
    d1, k = (torch.empty(plan.half_shape(1), dtype=torch.complex64, device="cuda") for _ in range(2))
    spectra = torch.empty(plan.half_shape(1, 2, 2), dtype=torch.complex64, device="cuda")
    ws = torch.empty(plan.workspace_size(), dtype=torch.uint8, device="cuda")
    pw = torch.empty(g.power_workspace_size(plan, 8), dtype=torch.uint8, device="cuda")
    bw = torch.empty(g.bispectrum_workspace_size(plan, 8), dtype=torch.uint8, device="cuda")
    p, nk = torch.empty(8, dtype=torch.float64, device="cuda"), torch.empty(8, dtype=torch.int64, device="cuda")
    rows = torch.empty(300, 3, device="cuda")
    y = torch.empty(300, 40, device="cuda")

    def sequence(sync):
        out = []

        def step(f, *results):
            f()
            if sync:
                torch.cuda.synchronize()
            out.extend(r.clone() for r in results)
            if sync:
                torch.cuda.synchronize()

        for seed in range(6):
            step(lambda: g.make_linear_field(plan, [seed], out=d1), d1)
            step(lambda: g.run_orders(plan, d1, spectra=spectra, ws=ws), spectra)
            step(lambda: g.power(plan, d1[0], spectra[0, 0, 0], edges, ws=pw, out=p, nk=nk), p, nk)
            step(lambda: g.c2r(plan, d1, out=x[None]), x)
            step(lambda: g.r2c(plan, x[None], out=k), k)
            out.extend(t.clone() for t in g.bispectrum(plan, k[0], spectra[0, 0, 0], edges, ws=bw))
            step(lambda: d1.mul_(0.5))
            step(lambda: g.run_orders(plan, d1, spectra=spectra, ws=ws), spectra)
            step(lambda: g.power(plan, d1[0], k[0], edges, ws=pw, out=p, nk=nk), p)
            step(lambda: rows.fill_(0.01 * seed).add_(torch.arange(300, device="cuda")[:, None] / 300.0))
            step(lambda: net.forward(rows, y=y), y)
            step(lambda: rows.zero_())
        torch.cuda.synchronize()
        return out

    for a, b in zip(sequence(True), sequence(False), strict=True):
        assert torch.equal(a, b)


def graph_time(f, calls=10, rounds=7):
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


@pytest.mark.parametrize("N", [64, 96, 128, 192])
def test_default_variants_not_slower_than_tiles(N):
    plan = g.Plan(N, 5, 4.0 * N)
    d1 = g.make_linear_field(plan, [5])
    spectra = torch.empty(plan.half_shape(1, 4, 2), dtype=torch.complex64, device="cuda")
    ws = torch.empty(plan.workspace_size(), dtype=torch.uint8, device="cuda")
    default = g.get_tuning(plan)
    times = []
    for choice in (default, [0] * 5):
        g.set_tuning(plan, choice)
        times.append(graph_time(lambda: g.run_orders(plan, d1, spectra=spectra, ws=ws)))
    assert times[0] <= 1.08 * times[1], times


@pytest.mark.parametrize("N", [48, 64, 96, 128, 192])
def test_autotuned_variants_not_slower_than_default(N):
    """The tuner times what a run launches. With the finished rows' forward z pass left
    out it took tiles at 96^3, 1.11 times the default's time; bound 1.05."""
    plan = g.Plan(N, 5, 4.0 * N)
    d1 = g.make_linear_field(plan, [5])
    spectra = torch.empty(plan.half_shape(1, 4, 2), dtype=torch.complex64, device="cuda")
    ws = torch.empty(plan.workspace_size(), dtype=torch.uint8, device="cuda")
    default = g.get_tuning(plan)
    tuned = g.autotune(plan)
    times = []
    for choice in (tuned, default):
        g.set_tuning(plan, choice)
        times.append(graph_time(lambda: g.run_orders(plan, d1, spectra=spectra, ws=ws)))
    assert times[0] <= 1.05 * times[1], (times, tuned, default)
