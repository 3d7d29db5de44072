"""The initial field's row kernel against the FP64 oracle at row lengths below,
at and above a warp's 32 modes, with the default cut and with every mode kept.

Bound: the value is formed in FP64 with a relative error far below FP32's and
rounded once, so each component is off by at most half an FP32 step, 2^-24 of
it (plus 1e-12 of the mode's modulus); zeros are exact and in the same places."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import cosmology, spt  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cut", [0.0, 100.0])
@pytest.mark.parametrize("N,n_max,seed", [(8, 1, 0), (12, 2, 3), (24, 1, (1 << 64) - 1), (48, 5, 17), (64, 1, 1 << 40),
                                          (96, 3, 123456789)])
def test_initial_field_rows(N, n_max, seed, cut):
    L = 4.0 * N
    cosmo = dict(cosmology.DEFAULT_COSMO, n_s=0.93, gamma=0.19)
    plan = g.Plan(N, n_max, L, batch=2, kcut_lin=cut)
    got = g.make_linear_field(plan, [seed, 5], cosmo).cpu().numpy()
    for b, s in enumerate((seed, 5)):
        ref = spt.linear_field(N, L, n_max, cosmo, s, kcut_lin=cut)[:, :, : N // 2]
        assert np.array_equal(got[b] == 0, ref == 0)
        for part in (np.real, np.imag):
            assert np.all(np.abs(part(got[b]).astype(np.float64) - part(ref)) <=
                          2.0 ** -24 * np.abs(part(ref)) * (1 + 1e-6) + 1e-12 * np.abs(ref))
