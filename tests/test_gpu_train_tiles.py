"""The fused training step with many 128-row tiles per CTA (every barrier of the
backward kernel through several phases, a ragged last tile).

test_gradient_of_many_tiles: against the FP64 oracle MLP, bounds as for the
gradient test of test_gpu_surrogate.py (BF16 operands, FP32 accumulation).

test_gradient_is_the_mean_over_sub_batches: 32 members (1118 tiles, 7 or 8 per
CTA) against 8 batches of 4 members (140 tiles, one per CTA).  The factor 8
between their weights is a power of two, so every BF16 operand of a row is the
same but for its exponent, and only the order of FP32 sums differs: up to about
160 accumulations of 16 rows per split, 160 x 2^-23 = 2e-5 of the sum of
magnitudes, which the cancellation of dlogit (it sums to zero over a histogram)
may make 50 times the gradient: 1e-3.  A tile that used another tile's operands
changes it by its share of the rows.
"""
import numpy as np
import pytest

import ens_inputs as I
import oracle.mlp as OMLP
from test_gpu_surrogate import E, bf16_params  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_gradient_of_many_tiles(E):  # noqa: F811
    n, nq, nt = 25, 63, 250          # 111725 rows, 873 tiles
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    lams = np.linspace(-2.0, 2.5, n)
    counts = I.synthetic_member_counts(lams, nq, nt, 100000, seed=n)
    S = E.Surrogate(seed=4)
    loss, g = S.loss_grad(lams, counts, h)
    rl, rg = OMLP.loss_grad(bf16_params(S.params()), lams, counts, nq, nt)
    S.close()
    assert loss == pytest.approx(rl, rel=2e-3)
    rel = np.linalg.norm(g - rg) / np.linalg.norm(rg)
    assert rel < 3e-2 and g @ rg / (np.linalg.norm(g) * np.linalg.norm(rg)) > 0.999, rel


def test_gradient_is_the_mean_over_sub_batches(E):  # noqa: F811
    n, sub, nq, nt = 32, 4, 63, 250
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    lams = np.linspace(-2.0, 2.5, n)
    counts = I.synthetic_member_counts(lams, nq, nt, 100000, seed=n)
    S = E.Surrogate(seed=5)
    loss, g = S.loss_grad(lams, counts, h)
    parts = [S.loss_grad(lams[k:k + sub], counts[k:k + sub], h) for k in range(0, n, sub)]
    S.close()
    assert loss == pytest.approx(np.mean([p[0] for p in parts]), rel=1e-6)
    ref = np.mean([p[1].astype(np.float64) for p in parts], axis=0)
    assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref)
