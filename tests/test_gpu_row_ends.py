"""Rows of the compact state end in zeros.

The passes write each kz row up to the end of its last 64 bytes, zeros past
the kept modes, whatever the pass variant; a value left there would end up in
the checkpoint and in the state that ens_get_state hands out.  Odd and even
mode counts, sizes whose rows end inside a sector (all but 384), the fused,
split and two-group last passes, narrow tiles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,change", [
    (16, {}), (32, {}), (64, {}), (64, {"fx_split": 1}), (64, {"tile_x": 8, "tile_y": 8}), (128, {}),
    (128, {"fx_split": 1, "plan_x": 1}), (256, {}), (256, {"fx_split": 1, "z_variant": 2, "z_ctas_per_sm": 1}),
    (256, {"fx_split": 2}), (512, {"fx_split": 1, "z_variant": 1}),
])
def test_padding_stays_zero(N, change):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    members = [E.Member(N=N, nu=0.02, lam=l, k_lo=1, k_hi=2, dt=-1.0, dt_max=0.01, rk_order=3, seed=i)
               for i, l in enumerate((-0.5, 0.5))]
    e = E.Ensemble(members)
    t = e.tuning()
    t["groups"][0].update(change)
    e.set_tuning(t)
    kc = (N + 2) // 3 - 1
    NK, NZ = 2 * kc + 1, kc + 1
    NZp = (NZ + 15) // 16 * 16
    host = torch.empty(e.state_bytes() // 4, dtype=torch.float32, pin_memory=True)
    e.step(2)
    E.ens_get_state(e.ctx, host.data_ptr(), e.state_bytes())
    e.diagnostics()
    e.close()
    s = host.numpy().reshape(2, 3, NK, NK, NZp, 2)
    assert not s[..., NZ:, :].any()
    assert np.isfinite(s).all() and np.abs(s[..., :NZ, :]).max() > 0
