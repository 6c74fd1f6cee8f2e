"""The stage's middle in one launch, and the link of two stages in one launch
(N <= 64), against the separate passes: the
same lines with the same transforms, only the n_z rows that share a complex
line are paired differently, so fields agree to FP32 rounding (1e-6 after a
step of three stages) and the CFL maximum, a maximum over the same points of
the first stage, is equal.  Member counts around the number of CTAs that fill
the chip, RK2 and RK3, a forced bounded-wait path (which runs the separate
passes)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,n,rk", [(16, 1, 2), (16, 21, 3), (32, 1, 2), (32, 11, 3), (64, 1, 3), (64, 3, 2),
                                    (64, 10, 3), (64, 12, 3)])
def test_plane_equals_separate_passes(N, n, rk):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    ms = [E.Member(N=N, nu=0.01, lam=l, k_lo=1, k_hi=2, dt=-1.0, dt_max=0.01, rk_order=rk, seed=i)
          for i, l in enumerate(np.linspace(-1.0, 1.0, n))]
    a, b = E.Ensemble(ms), E.Ensemble(ms)
    t = b.tuning()
    t["groups"][0].update(tile_y=8)
    b.set_tuning(t)
    assert E.ens_kernels_per_step(a.ctx) < E.ens_kernels_per_step(b.ctx)
    a.step(1)
    b.step(1)
    da, db = a.diagnostics(), b.diagnostics()
    for i in range(n):
        fa, fb = a.field(i), b.field(i)
        assert np.linalg.norm(fa - fb) <= 1e-6 * np.linalg.norm(fb), i
        assert da[i]["umax"] == db[i]["umax"] and da[i]["dt"] == db[i]["dt"], i
    # run state after further steps: the stage ends run in other launches
    a.step(2)
    b.step(2)
    for x, y in zip(a.diagnostics(), b.diagnostics()):
        assert x["steps"] == y["steps"] == 3
        for k in ("t", "dt", "E", "diss", "EB", "P", "umax"):
            assert abs(x[k] - y[k]) <= 1e-5 * abs(y[k]), k
    a.close()
    b.close()
