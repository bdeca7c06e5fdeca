"""One-launch steps of small meshes whose grid-barrier wait gives up: the host learns of it
from the status word, and the next call starts from clean barrier words."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
dg = pytest.importorskip("paper_2404_08952_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_timeout_is_reported_and_the_next_call_is_clean(precision):
    m = synth.tri_mesh(40, 36, jitter=0.2, seed=8)
    M = dg.Mesh(m)
    sch = dg.Scheme(k=3, r=1, n_diff=2, flux="upwind", nv=1, precision=precision, adv=(1.0, 0.5))
    ws = dg.workspace(M, sch)
    u0 = 1.0 + 0.1 * np.random.default_rng(3).random((1, M.n_cells))
    dg.dolinc_mesh_set_spin_limit(M, 0)               # every wait gives up at its first poll
    u = torch.from_numpy(u0).cuda()
    for _ in range(3):
        dg.dolinc_rk_steps(M, sch, 1e-3, 2, u, ws)
        with pytest.raises(dg.DolincError) as e:
            dg.dolinc_sync_status(M, ws)
        assert e.value.status == 5
    dg.dolinc_mesh_set_spin_limit(M)
    got = []
    for _ in range(2):
        u = torch.from_numpy(u0).cuda()
        dg.dolinc_rk_steps(M, sch, 1e-3, 2, u, ws)
        dg.dolinc_sync_status(M, ws)
        got.append(u.cpu().numpy())
    # the separate launches that a set shape takes
    dg.dolinc_set_tuning(M, sch, *((1, 64, -2, 64) if precision == "fp64" else (4, 256, 4, 128)))
    u = torch.from_numpy(u0).cuda()
    dg.dolinc_rk_steps(M, sch, 1e-3, 2, u, ws)
    dg.dolinc_sync_status(M, ws)
    for g in got:
        np.testing.assert_array_equal(g, u.cpu().numpy())
