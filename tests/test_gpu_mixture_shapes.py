"""The mixture kernels at the edges of their split (32 bins per block, 8
member slices per bin, 5 for the moments) and the quadrature mixture's (8
slices of the points), against the oracle and against plain FP64 sums.
Bounds: every sum is FP64 over at most 1024 terms of one sign (PDFs) or of
mixed sign (moments): 1e-12 relative to the largest value."""
import numpy as np
import pytest

import ens_inputs as I
import oracle as O
import oracle.mixture as OM
from test_gpu_surrogate import E  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,nt", [(1, 1, 1), (2, 5, 7), (7, 6, 32), (8, 8, 33), (9, 16, 40), (33, 10, 50),
                                     (257, 12, 16), (1024, 4, 9)])
def test_mixture_shapes(E, n, nq, nt):  # noqa: F811
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    rng = np.random.Generator(np.random.Philox(key=n))
    lams = np.sort(rng.standard_normal(n)) if n > 1 else np.array([0.2])
    counts = I.synthetic_member_counts(lams, nq, nt, 50000, seed=n)
    moments = rng.standard_normal((n, 48)) * 50000
    moments[:, 0:36:4] = np.abs(moments[:, 0:36:4])
    got = E.ens_mixture_host(lams, counts, moments, h, kind=E.W_GAUSS_PAPER, c=0.023, Z=2.0)
    w, cov = OM.member_weights(lams, "gauss_paper", c=0.023, Z=2.0)
    assert np.allclose(got["weights"], w, rtol=1e-12, atol=1e-15) and got["covered"] == pytest.approx(cov, rel=1e-12)
    qr, pe, pw = OM.mix_counts(counts, w, O.HistSpec(qr_bins=nq, tail_bins=nt))
    for a, b in ((got["pdf_qr"], qr), (got["pdf_eps"], pe), (got["pdf_ens"], pw)):
        assert np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 1e-300)
    mm = OM.mix_moments(moments, counts[:, -2], w)
    assert np.abs(got["moments"] - mm).max() <= 1e-12 * np.abs(mm).max()
    for k, v in OM.gradient_moment_ratios(mm).items():
        assert got["ratios"][k] == pytest.approx(v, rel=1e-9)


@pytest.mark.parametrize("nquad,nq,nt", [(1, 5, 7), (7, 6, 33), (9, 16, 40), (600, 4, 9)])
def test_quadrature_is_the_weighted_density(E, nquad, nq, nt):  # noqa: F811
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    S = E.Surrogate(seed=2)
    lo, hi = -1.5, 2.0
    m = S.mixture(h, lo, hi, nquad=nquad, kind=E.W_GAUSS, mu=0.3, sigma=0.9)
    edges = lo + (hi - lo) / nquad * np.arange(nquad + 1)
    q = S.density(edges[:-1] + 0.5 * (hi - lo) / nquad, h)
    S.close()
    w = np.array([OM.normal_interval_mass(a, b, 0.3, 0.9) for a, b in zip(edges[:-1], edges[1:])])
    pdf = (w / w.sum()) @ q
    ref = pdf[:nq * nq].reshape(nq, nq) / ((2 * h.q_lim / nq) * (2 * h.r_lim / nq))
    assert np.abs(m["pdf_qr"] - ref).max() <= 1e-6 * np.abs(ref).max()   # densities are FP32
    ref = pdf[nq * nq:nq * nq + nt] / ((h.tail_hi - h.tail_lo) / nt)
    assert np.abs(m["pdf_eps"] - ref).max() <= 1e-6 * np.abs(ref).max()
