"""The stage's middle in one launch (N <= 64) beside last-pass variants that do
not link the stages (8-column tiles, split last pass): the end of the stage in
its own launch.  Against the separate passes with the same last pass, bounds as
in test_gpu_plane.py: fields to FP32 rounding of a step (1e-6), the CFL maximum
of the first stage equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("change", [{"tile_x": 8}, {"fx_split": 1}])
@pytest.mark.parametrize("N,n,rk", [(16, 5, 3), (32, 3, 2), (64, 2, 3)])
def test_plane_without_chain(N, n, rk, change):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    ms = [E.Member(N=N, nu=0.01, lam=l, k_lo=1, k_hi=2, dt=-1.0, dt_max=0.01, rk_order=rk, seed=i)
          for i, l in enumerate(np.linspace(-1.0, 1.0, n))]
    a, b = E.Ensemble(ms), E.Ensemble(ms)
    for e, extra in ((a, {}), (b, {"tile_y": 8})):
        t = e.tuning()
        t["groups"][0].update(change, **extra)
        e.set_tuning(t)
    last = 2 if change.get("fx_split") else 1
    assert E.ens_kernels_per_step(a.ctx) == rk * (2 + last + 1)   # IX, PLANE, last pass, end
    assert E.ens_kernels_per_step(b.ctx) == rk * (4 + last + 1)
    a.step(1)
    b.step(1)
    for i, (x, y) in enumerate(zip(a.diagnostics(), b.diagnostics())):
        fa, fb = a.field(i), b.field(i)
        assert np.linalg.norm(fa - fb) <= 1e-6 * np.linalg.norm(fb), i
        assert x["umax"] == y["umax"] and x["dt"] == y["dt"], i
        for k in ("E", "diss", "EB", "P"):
            assert abs(x[k] - y[k]) <= 1e-6 * abs(y[k]), k
    a.close()
    b.close()
