"""Shell power by symmetric row sets: every grid mode below the top edge is
counted once with its weight, up to a top edge at the Nyquist wavenumber.

Bound per bin: a term x.re y.re + x.im y.im formed in FP32 is off by at most
2^-23 |x||y|, so the bin's sum by at most 2^-23 sqrt(P_aa P_bb) (Cauchy-Schwarz);
the sums themselves are compensated (1e-12)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import estimators  # noqa: E402
from paper_1807_04215_gb300 import gridspt as g  # noqa: E402
from tests import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _half(N, seed):
    """A Hermitian full-grid spectrum (FP32 values) without Nyquist modes."""
    f = np.fft.fftn(inputs.rng(seed).standard_normal((N, N, N)))
    f[N // 2] = f[:, N // 2] = f[:, :, N // 2] = 0
    half = f[:, :, : N // 2].astype(np.complex64)
    full = np.fft.fftn(np.fft.ifftn(f).real)
    full[:, :, : N // 2] = half
    idx = (-np.arange(N)) % N
    for kz in range(1, N // 2):     # the conjugate half, from the rounded values
        full[:, :, N - kz] = np.conj(half[:, :, kz].astype(np.complex128))[idx][:, idx]
    return half, full


@pytest.mark.parametrize("accum", ["compensated", "fp64"])
@pytest.mark.parametrize("N,nbins,top", [(8, 1, 1.0), (12, 3, 1.0), (24, 64, 1.0), (64, 7, 1.0), (96, 20, 0.37)])
def test_power_row_sets(N, nbins, top, accum):
    L = 3.0 * N
    kF, kny = 2 * math.pi / L, math.pi * N / L
    edges = [kF * 0.5 + (kny * top - kF * 0.5) * i / nbins for i in range(nbins + 1)]
    (ha, fa), (hb, fb) = _half(N, 1), _half(N, 2)
    plan = g.Plan(N, 2, L, accum=accum)
    a, b = torch.from_numpy(ha).cuda(), torch.from_numpy(hb).cuda()
    paa, _ = estimators.power(fa, fa, L, edges)
    pbb, _ = estimators.power(fb, fb, L, edges)
    for x, y, fx, fy in ((a, b, fa, fb), (a, a, fa, fa)):
        p, nk = g.power(plan, x, y, edges)
        ref, nref = estimators.power(fx, fy, L, edges)
        assert np.array_equal(nk.cpu().numpy(), nref)
        assert np.all(np.abs(p.cpu().numpy() - ref) <= (2.0 ** -23 + 1e-12) * np.sqrt(paa * pbb if fy is fb else paa * paa))
