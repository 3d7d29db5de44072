"""The initial field at the ends of the amplitude's range: beyond FP32 every mode is
an infinity of the deviate's sign (as the FP64 product rounded to FP32 gives), far
below 1 it keeps half an FP32 step while the pair's error is a normal number."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import cosmology, spt  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma8", [1e45, 1e30, 1e-12, 1e-24])
def test_amplitude_range(sigma8):
    N, L, n_max, seed = 16, 64.0, 1, 7
    cosmo = dict(cosmology.DEFAULT_COSMO, sigma8=sigma8)
    got = g.make_linear_field(g.Plan(N, n_max, L), [seed], cosmo)[0].cpu().numpy()
    ref = spt.linear_field(N, L, n_max, cosmo, seed)[:, :, : N // 2]
    with np.errstate(over="ignore"):
        for part in (np.real, np.imag):
            a, r = part(got), part(ref)
            if sigma8 == 1e45:
                assert np.all(np.abs(r[r != 0]) > 1e39)
                assert np.array_equal(a, r.astype(np.float32))
            else:
                assert np.all(np.abs(a.astype(np.float64) - r) <= 2.0 ** -24 * np.abs(r) * (1 + 1e-6) + 1e-12 * np.abs(ref))
