"""Kernels against another form of the same computation.

Columns: the one-exchange transform of the x, y and forward column passes equals the
transform with one exchange per stage bit for bit (its stages, butterflies and twiddle
values are the same), in both directions and the widths that the passes (16) and the
work queue (32) use; and both are the Fourier transform: log2(N) FP32 stages of error
2^-23 each, in the root mean square of the output.
Normals: the deviates' pairs against FP64 at the ends of the words' range, next to
table midpoints and quarter turns, within 1e-12 of the modulus (the header's bound)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1807_04215_gb300 import _lib  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402
from tests import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [1, -1])
@pytest.mark.parametrize("N,width", [(128, 16), (128, 32), (256, 16), (256, 32), (512, 16), (1024, 16)])
def test_one_exchange_columns(N, width, direction):
    lib, plan = _lib.load(), g.Plan(N, 2, 4.0 * N)
    r = inputs.rng(N + width)
    x = (r.standard_normal((2, N, width)) + 1j * r.standard_normal((2, N, width))).astype(np.complex64)
    x[0, :, 1] = 0
    x[0, :, 2] = 1
    x[0, :, 3] = 0
    x[0, N - 1, 3] = 1j
    x[1, :, :4] *= np.float32(1e30), np.float32(1e-30), np.float32(1e-41), np.float32(1)
    xd = torch.from_numpy(x).cuda()
    out = [torch.full_like(xd, float("nan")) for _ in range(2)]
    for one in (0, 1):
        _lib.check("columns", lib.gridspt_selftest_columns(plan.handle, width, direction, one, xd.data_ptr(),
                                                           out[one].data_ptr(), None))
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))
    x64 = x.astype(np.complex128)
    ref = np.fft.ifft(x64, axis=1) * N if direction > 0 else np.fft.fft(x64, axis=1)
    got = out[1].cpu().numpy().astype(np.complex128)
    for s in range(2):
        for c in range(width):
            if s == 1 and c == 2:
                continue                                     # subnormal inputs: bits above only
            rms = np.sqrt(np.mean(np.abs(ref[s, :, c]) ** 2))
            assert np.abs(got[s, :, c] - ref[s, :, c]).max() <= 8 * np.log2(N) * 2.0 ** -23 * rms


def test_column_selftest_refuses_other_sizes():
    lib, buf = _lib.load(), torch.zeros(1 << 16, device="cuda")
    for N, width, direction in ((96, 16, 1), (64, 16, 1), (512, 32, 1), (128, 8, 1), (128, 16, 0)):
        assert lib.gridspt_selftest_columns(g.Plan(N, 2, 4.0 * N).handle, width, direction, 1, buf.data_ptr(),
                                            buf.data_ptr(), None) == 1


def test_normal_deviates_at_chosen_words():
    ends = [0, 1, 2, 3, (1 << 31) - 1, 1 << 31, (1 << 31) + 1, (1 << 32) - 2, (1 << 32) - 1]
    u1 = ends + [1 << k for k in range(2, 32)] + [(1 << k) - 1 for k in range(2, 32)]
    # words whose h = u1 2^-k lies beside the table's midpoints (2 i + 1) / 512
    u1 += [(((2 * i + 1) << 23) + d) % (1 << 32) for i in range(128, 256) for d in (-2, -1, 0, 1)]
    # turns beside the angle table's points, midpoints and the quarters
    u2 = ends + [((j << 22) + d) % (1 << 32) for j in range(0, 1024, 13) for d in (-1, 0)]
    u2 += [((q << 30) + d) % (1 << 32) for q in range(4) for d in (-3, -2, -1, 0, 1, 2)]
    r = inputs.rng(5)
    words = np.array([(a, u2[i % len(u2)]) for i, a in enumerate(u1)] + [(u1[i % len(u1)], b) for i, b in enumerate(u2)],
                     dtype=np.uint32)
    words = np.concatenate([words, r.integers(0, 1 << 32, size=(100000, 2), dtype=np.uint32)])
    out = torch.empty(len(words), 2, dtype=torch.float64, device="cuda")
    wd = torch.from_numpy(words.view(np.int32)).cuda()
    lib, plan = _lib.load(), g.Plan(8, 1, 32.0)
    _lib.check("normals", lib.gridspt_selftest_normals(plan.handle, wd.data_ptr(), len(words), out.data_ptr(), None))
    got = out.cpu().numpy()
    w = words.astype(np.int64)
    v1 = 2 * w[:, 0] + 1                                             # u1 2^33
    near = v1 > 1 << 32                                              # u1 > 1/2: through 1 - u1, exact
    lnu = np.where(near, np.log1p(-((1 << 33) - v1) * 2.0 ** -33), np.log(v1 * 2.0 ** -33))
    rad = np.sqrt(-2.0 * lnu)
    v2 = 2 * w[:, 1] + 1                                             # turns 2^33, reduced to the nearest eighth exactly
    j = (v2 + (1 << 29)) >> 30
    d = 2.0 * np.pi * ((v2 - (j << 30)) * 2.0 ** -33)
    s2 = np.sqrt(0.5)
    cj = np.array([1, s2, 0, -s2, -1, -s2, 0, s2])[j % 8]
    sj = np.array([0, s2, 1, s2, 0, -s2, -1, -s2])[j % 8]
    cs, sn = cj * np.cos(d) - sj * np.sin(d), sj * np.cos(d) + cj * np.sin(d)
    err = np.maximum(np.abs(got[:, 0] - rad * cs), np.abs(got[:, 1] - rad * sn)) / rad
    assert err.max() <= 1e-12, (err.max(), words[err.argmax()])
