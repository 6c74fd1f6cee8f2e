"""ens_step_host and ens_step_sequential on a context whose tuning says
persistent = 1: both launch pass by pass with the groups' variants, so the run
state and the fields are those of the same calls with persistent = 0, bit for
bit (the same launches, and every stage end adds up all partial sums that the
launch before it wrote)."""
import json

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("change", [{}, {"fx_split": 0, "tile_x": 8}, {"fx_split": 1}])
@pytest.mark.parametrize("sizes", [(128, 256, 256), (384,)])
def test_host_and_sequential_steps(sizes, change):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_23712_gb300 import ens as E
    ms = [E.Member(N=N, nu=0.01, lam=0.3 * i, k_lo=2, k_hi=4, dt=-1.0, dt_max=0.002, rk_order=3, seed=i)
          for i, N in enumerate(sizes)]
    ctx = [E.Ensemble(ms) for _ in range(2)]
    for persistent, e in enumerate(ctx):
        t = json.loads(json.dumps(e.tuning()))
        t["persistent"] = persistent
        for g in t["groups"]:
            g.update(change)
        e.set_tuning(t)

    def same():
        d0, d1 = (e.diagnostics() for e in ctx)
        for i in range(len(ms)):
            for k in ("steps", "t", "dt", "E", "diss", "EB", "P", "umax"):
                assert d1[i][k] == d0[i][k], (i, k)
            assert np.array_equal(ctx[1].field(i), ctx[0].field(i)), i

    for e in ctx:
        E.ens_step_sequential(e.ctx, 2)
    same()
    for e in ctx:
        nbytes = E.ens_state_bytes(e.ctx)
        host = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
        E.ens_get_state(e.ctx, host.data_ptr(), nbytes)
        E.ens_step_host(e.ctx, host.data_ptr(), host.data_ptr(), nbytes, 0)
    same()
    for e in ctx:
        e.close()
