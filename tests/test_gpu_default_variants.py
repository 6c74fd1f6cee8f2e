"""The pass variants a new context starts with, on both sides of each size
rule, and that they compute what the plain variants do (FP32 rounding of one
step: 1e-6 relative)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sizes,parallel,want", [
    ((16, 128), 1, {16: (16, 0, 0), 128: (16, 0, 0)}),
    ((64, 256), 0, {64: (16, 0, 0), 256: (16, 2, 1)}),
    ((384,), 0, {384: (8, 0, 1)}),
])
def test_default_variants(sizes, parallel, want):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    ms = [E.Member(N=N, nu=0.02, lam=0.2, k_lo=1, k_hi=2, dt=-1.0, dt_max=0.01, rk_order=3, seed=i)
          for i, N in enumerate(sizes)]
    a, b = E.Ensemble(ms), E.Ensemble(ms)
    t = a.tuning()
    assert t["parallel_groups"] == parallel
    for g in t["groups"]:
        assert (g["tile_x"], g["z_variant"], g["fx_split"]) == want[g["N"]]
        g.update(tile_x=16, z_variant=0, z_ctas_per_sm=1, fx_split=0)
    b.set_tuning(t)
    a.step(1)
    b.step(1)
    da, db = a.diagnostics(), b.diagnostics()
    for i in range(len(ms)):
        fa, fb = a.field(i), b.field(i)
        assert np.linalg.norm(fa - fb) <= 1e-6 * np.linalg.norm(fb), i
        assert abs(da[i]["E"] - db[i]["E"]) <= 1e-6 * db[i]["E"]
    a.close()
    b.close()
