"""A member without points (no snapshot of it was taken) is left out of the
mixture, whatever its moment sums hold: NaN and infinity there give the result
of zeros, bit for bit (the same sums of the other members)."""
import numpy as np
import pytest

import ens_inputs as I
from test_gpu_surrogate import E  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["ens_mixture_host", "ens_mixture_host_noalloc"])
@pytest.mark.parametrize("n,empty", [(1, 0), (2, 0), (7, 6), (40, 13)])
def test_empty_member_is_left_out(E, n, empty, entry):  # noqa: F811
    nq, nt = 6, 20
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    lams = np.linspace(-1.0, 1.5, n)
    rng = np.random.Generator(np.random.Philox(key=n))
    counts = I.synthetic_member_counts(lams, nq, nt, 4000, seed=n)
    moments = rng.standard_normal((n, 48)) ** 2
    counts[empty] = 0

    def mix(fill):
        m = moments.copy()
        m[empty, ::2] = fill
        m[empty, 1::2] = -fill
        return getattr(E, entry)(lams, counts, m, h, kind=E.W_GAUSS, mu=0.1, sigma=0.8)

    ref = mix(0.0)
    assert np.isfinite(ref["moments"]).all() and (n == 1 or ref["moments"].all())
    for fill in (np.nan, np.inf):
        got = mix(fill)
        for k in ("weights", "pdf_qr", "pdf_eps", "pdf_ens", "moments"):
            assert np.array_equal(got[k], ref[k]), k
