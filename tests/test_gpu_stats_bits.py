"""The statistics' x derivative rounds the same whether a mode's row is known
zero at compile time or checked at run time: counts of a field whose modes fill
the whole dealiased set are the same for the field and for its mirror image
in every coordinate (x -> -x conjugates every mode; A_ij is then negated, so
the invariants Q, eps, omega^2 are the same numbers at mirrored points and
their tail histograms agree exactly up to FP32 rounding of the transforms: at
most 1e-4 of the points change bin)."""
import numpy as np
import pytest

import ens_inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [32, 64, 128, 384])
def test_mirrored_field_has_the_same_tails(N):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    m = E.Member(N=N, nu=0.02, lam=0.0, k_lo=1, k_hi=2, dt=0.01, rk_order=2, seed=3)
    h = E.hist_spec(qr_bins=16, tail_bins=64, nu_norm=0.02)
    f = I.random_spectral(N, 3, scale=1e-3)
    k = np.fft.fftfreq(N, 1.0 / N)
    kx, ky, kz = k[:, None, None], k[None, :, None], np.arange(N // 2 + 1)[None, None, :]
    k2 = np.maximum(kx ** 2 + ky ** 2 + kz ** 2, 1.0)
    p = (kx * f[0] + ky * f[1] + kz * f[2]) / k2
    f -= np.stack([kx * p, ky * p, kz * p])
    f[:, :, :, 0] = 0     # no Hermitian constraint left inside the plane
    e = E.Ensemble([m, m], hist=h)
    e.set_field(0, f)
    e.set_field(1, np.conj(f))
    e.gradient_stats(accumulate=False)
    c, mom = e.stats()
    e.close()
    tails = slice(16 * 16, 16 * 16 + 128)
    assert c[0, tails].sum() > 1.9 * N ** 3
    d = np.abs(c[0, tails].astype(np.int64) - c[1, tails].astype(np.int64)).sum()
    assert d <= 2 * 2 * 1e-4 * N ** 3, d
    assert np.all(np.abs(mom[0, 38:44] - mom[1, 38:44]) <= 1e-5 * np.abs(mom[0, 38:44]))
