"""The fused training step (tcgen05 backward and weight-gradient kernels) at
the edges of its 128-row tiles, 64-row half tiles and row splits, against the
FP64 oracle MLP.

Bounds as for the gradient test of test_gpu_surrogate.py: BF16 operands with
FP32 accumulation, every product of a gradient rounded three times to BF16
(2^-9 relative each, independent over rows and columns): relative L2 <= 3e-2,
cosine >= 0.999, loss 2e-3.
"""
import numpy as np
import pytest

import ens_inputs as I
import oracle.mlp as OMLP
from test_gpu_surrogate import E, bf16_params  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,nt", [
    (1, 1, 1),       # 3 rows of one tile, one half tile empty of real rows
    (1, 7, 7),       # 63 rows: one short of a half tile
    (1, 8, 32),      # exactly one tile
    (1, 9, 24),      # 129 rows: one row in the second tile
    (3, 16, 40),     # groups straddle tiles
    (5, 33, 150),    # more half tiles than splits of a layer, ragged end
    (33, 24, 10),    # every CTA of the backward kernel has a tile
    (40, 24, 10),    # more tiles than CTAs: a second tile on a few
])
def test_gradient_at_tile_edges(E, n, nq, nt):  # noqa: F811
    h = E.hist_spec(qr_bins=nq, tail_bins=nt)
    lams = np.linspace(-2.0, 2.5, n) if n > 1 else np.array([0.4])
    counts = I.synthetic_member_counts(lams, nq, nt, 100000, seed=n)
    S = E.Surrogate(seed=3)
    loss, g = S.loss_grad(lams, counts, h)
    again, g2 = S.loss_grad(lams, counts, h)
    rl, rg = OMLP.loss_grad(bf16_params(S.params()), lams, counts, nq, nt)
    S.close()
    assert loss == again and np.array_equal(g, g2)
    if nq * nq == 1 and nt == 1:     # one bin per kind: the softmax is 1, loss and gradient vanish
        assert abs(loss) < 1e-6 and np.abs(g).max() < 1e-6
        return
    assert loss == pytest.approx(rl, rel=2e-3)
    rel = np.linalg.norm(g - rg) / np.linalg.norm(rg)
    assert rel < 3e-2 and g @ rg / (np.linalg.norm(g) * np.linalg.norm(rg)) > 0.999, rel
