"""Warp-row z passes (z expansion and z forward variant 2) on every row length:
two warps per row at N = 1024, twelve elements a thread at N = 3 * 2^a, down to
one thread per row. They regroup the work of the tile kernels, so the recursion
and the transforms agree with them bit for bit."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1807_04215_gb300 import gridspt as g  # noqa: E402

pytestmark = pytest.mark.gpu


# n_max = 5: one and two targets, band-limited and full inputs; 768 and 1024: one target
@pytest.mark.parametrize("N,n_max", [(8, 5), (12, 5), (16, 5), (24, 5), (48, 5), (96, 5), (384, 5), (768, 3),
                                     (1024, 2)])
def test_warp_rows_equal_the_tile_kernels(N, n_max):
    plan = g.Plan(N, n_max, 4.0 * N)
    d1 = g.make_linear_field(plan, [7])
    out = []
    for choice in ([0] * 5, [0, 0, 0, 2, 2]):
        g.set_tuning(plan, choice)
        x = g.c2r(plan, d1)
        out.append((g.run_orders(plan, d1), x, g.r2c(plan, x)))
        torch.cuda.empty_cache()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    del out, x, a, b
    torch.cuda.empty_cache()


@pytest.mark.parametrize("N", [24, 48, 192])
def test_warp_row_shell_sums_equal_the_tile_kernel(N):
    L = 4.0 * N
    kc = 2 * 3.141592653589793 / L * N * 0.3
    edges = [kc * i / 6 for i in range(7)]
    out = []
    for choice in ([0] * 5, [0, 0, 0, 2, 0]):
        plan = g.Plan(N, 4, L)
        g.set_tuning(plan, choice)
        d1 = g.make_linear_field(plan, [8])
        sp = g.run_orders(plan, d1)
        out.append([t.clone() for t in g.bispectrum(plan, d1[0], sp[0, 0, 0], edges)] +
                   [t.clone() for t in g.bispectrum_one_loop(plan, d1[0], sp[0, 0, 0], sp[0, 1, 0], sp[0, 2, 0], edges)])
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_recursions_of_different_orders_run_from_two_threads():
    """The z pass stages as many partner rows as its order has, so its shared
    memory differs between launches: no launch may depend on another thread's."""
    from concurrent.futures import ThreadPoolExecutor

    def run(n_max):
        with torch.cuda.stream(torch.cuda.Stream()):
            plan = g.Plan(64, n_max, 256.0)
            d1 = g.make_linear_field(plan, [n_max])
            ref = g.run_orders(plan, d1).clone()
            return all(bool(torch.equal(g.run_orders(plan, d1), ref)) for _ in range(100))

    with ThreadPoolExecutor(2) as pool:
        assert all(pool.map(run, (2, 6)))
