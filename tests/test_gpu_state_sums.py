"""Energy, dissipation and band energy of an uploaded field (k_state_sums),
one to many chunks per member, against FP64 sums over the same field; FP32
terms in FP32 partial sums of at most 2048 x 3 modes: 1e-5 relative.  And the
mixture weights' neighbour search (ordered integers) with negative, equal,
zero and unsorted lambdas."""
import numpy as np
import pytest

import ens_inputs as I
import oracle.mixture as OM

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2506_23712_gb300.ens as ens
    return ens


@pytest.mark.parametrize("N,change", [(16, {}), (32, {}), (64, {"tile_x": 8}), (64, {"fx_split": 1}), (128, {}),
                                      (256, {}), (256, {"fx_split": 0}), (256, {"fx_split": 2})])
def test_sums_of_uploaded_field(E, N, change):
    kc = (N + 2) // 3 - 1
    m = E.Member(N=N, nu=0.03, lam=0.0, k_lo=2, k_hi=3.5, dt=0.01, rk_order=2, seed=1)
    e = E.Ensemble([m, m])
    t = e.tuning()
    t["groups"][0].update(change)
    e.set_tuning(t)
    f = I.random_spectral(N, 7, scale=1e-2)
    f[:, 0, 0, 0] = 0
    e.set_field(1, f)
    d = e.diagnostics()[1]
    e.close()
    f = f.astype(np.complex64).astype(np.complex128)
    k = np.fft.fftfreq(N, 1.0 / N)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + np.arange(N // 2 + 1)[None, None, :] ** 2
    a2 = (np.abs(f) ** 2).sum(0)
    a2[:, :, 1:] *= 2.0
    assert kc > 0
    assert d["E"] == pytest.approx(0.5 * a2.sum(), rel=1e-5)
    assert d["diss"] == pytest.approx(0.03 * (k2 * a2).sum(), rel=1e-5)
    band = (k2 >= 4) & (k2 <= 12.25)
    assert d["EB"] == pytest.approx(0.5 * a2[band].sum(), rel=1e-5)


@pytest.mark.parametrize("lams", [[0.0], [-0.0, 0.0, 1.0], [2.0, -3.0, -3.0, 0.5, -1e-300, 1e-300], [1e300, -1e300, 0.1],
                                  list(np.linspace(3, -3, 33))])
def test_mixture_bins(E, lams):
    n = len(lams)
    h = E.hist_spec(qr_bins=3, tail_bins=4)
    counts = I.synthetic_member_counts(lams if max(map(abs, lams)) < 10 else [0.0] * n, 3, 4, 1000, seed=1)
    got = E.ens_mixture_host(lams, counts, np.ones((n, 48)), h, kind=E.W_GAUSS, mu=0.2, sigma=1.1, renormalize=False)
    w, cov = OM.member_weights(lams, "gauss", mu=0.2, sigma=1.1, renormalize=False)
    assert np.allclose(got["weights"], w, rtol=1e-12, atol=1e-15)
