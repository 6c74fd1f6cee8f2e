"""The statistics pass splits a member's rows over more CTAs when there are few
members, and counts the gradient components into as many histogram copies as
fit: neither may change a member's counts, nor its moments beyond the order of
FP64 additions (1e-13; the FP32 sums are over the same points in the same
order in every split)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,many,grad_bins", [
    (16, 700, 0), (16, 40, 33), (32, 700, 128), (32, 30, 2048), (64, 330, 0), (64, 16, 129), (128, 40, 64),
    (256, 20, 0),
])
def test_split_does_not_change_statistics(N, many, grad_bins):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    h = E.hist_spec(qr_bins=31, tail_bins=70, nu_norm=0.02, grad_bins=grad_bins)

    def stats(n, accumulate_twice=False):
        ms = [E.Member(N=N, nu=0.02, lam=0.3, k_lo=1, k_hi=2, dt=0.01, rk_order=2, seed=5 + i % 2) for i in range(n)]
        e = E.Ensemble(ms, hist=h)
        e.gradient_stats(accumulate=False)
        if accumulate_twice:
            e.gradient_stats(accumulate=True)
        out = e.stats()
        e.close()
        return out
    c1, m1 = stats(1)
    c2, m2 = stats(2, True)
    cn, mn = stats(many)
    assert c1[0].sum() > 0 and int(c1[0][31 * 31 + 140 + 6]) == N ** 3
    for i in (0, many // 2, many - 1):
        same = i % 2 == 0
        assert np.array_equal(cn[i], c1[0] if same else c2[1] // 2), i
        ref = m1[0] if same else m2[1] / 2
        assert np.all(np.abs(mn[i] - ref) <= 1e-13 * np.abs(ref) + 1e-300), i
    assert np.array_equal(c2[0], 2 * c1[0])
