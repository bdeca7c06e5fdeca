"""Grid-barrier waits that give up: the host learns of it from the status word, and the
next call starts from clean barrier words."""
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


@pytest.mark.parametrize("precision,k,r,n_diff", [("fp64", 3, 1, 2), ("fp64", 3, 1, 4), ("fp32", 3, 1, 3),
                                                  ("fp32", 5, 2, 3), ("fp64", 5, 2, 4)])
def test_every_block_of_a_batch_leaves_on_a_timeout(precision, k, r, n_diff):
    """Blocks start while others give up already: all leave, the state stays, and a launch
    that finds the abort word set does nothing."""
    ms = [synth.tri_mesh(60, 50, 0.2, s) for s in (1, 2, 3)]
    bt = dg.Batch([dg.Mesh(m) for m in ms])
    meshes = bt.meshes
    sch = dg.Scheme(k=k, r=r, n_diff=n_diff, flux="burgers", nv=1, precision=precision)
    ws = bt.workspace(sch)
    u0 = 1.0 + 0.1 * np.random.default_rng(4).random((1, sum(M.n_cells for M in meshes)))
    u = torch.from_numpy(u0).cuda()
    dt = torch.full((3,), 1e-4, dtype=torch.float64, device="cuda")
    bt.set_spin_limit(0)
    for _ in range(10):
        bt.rk_step(sch, dt, u, ws, use_graph=False)
        with pytest.raises(dg.DolincError) as e:
            dg.dolinc_sync_status(meshes[0], ws)
        assert e.value.status == 5
        np.testing.assert_array_equal(u.cpu().numpy(), u0)
    bt.set_spin_limit(1 << 23)
    bt.rk_step(sch, dt, u, ws, use_graph=False)
    dg.dolinc_sync_status(meshes[0], ws)
    assert np.abs(u.cpu().numpy() - u0).max() > 0


def test_every_block_of_a_solve_leaves_on_a_timeout():
    m = synth.hexprism_mesh(30, 0.2, 5)
    M = dg.Mesh(m)
    sch = dg.Scheme(k=3, r=1, n_diff=2, flux="upwind", nv=1, adv=(1.0, 0.6, 0.4))
    S = dg.Implicit(M, sch, 0.02, 1.0)
    ws = dg.workspace(M, sch)
    u0 = 1.0 + 0.1 * np.random.default_rng(5).random((1, M.n_cells))
    ref = torch.from_numpy(u0).cuda()
    S.step(ref, ws)
    assert S.info()["converged"]
    for _ in range(10):
        S.set_solver(spin_limit=0)
        u = torch.from_numpy(u0).cuda()
        S.step(u, ws, n_outer=2)                      # the second solve finds the abort word set
        with pytest.raises(dg.DolincError) as e:
            S.info()
        assert e.value.status == 5
        S.set_solver()
        u = torch.from_numpy(u0).cuda()
        S.step(u, ws)
        assert S.info()["converged"]
        np.testing.assert_array_equal(u.cpu().numpy(), ref.cpu().numpy())


@pytest.mark.parametrize("precision,k,r,n_diff", [("fp64", 3, 1, 2), ("fp64", 3, 1, 4), ("fp32", 3, 1, 3),
                                                  ("fp32", 3, 1, 4), ("fp32", 5, 2, 4)])
def test_a_batch_step_is_whole_or_leaves_the_state(precision, k, r, n_diff):
    """Whatever poll limit a launch runs into, a reported timeout leaves the state as it was,
    and a step that reports none is the step of the normal limit."""
    bt = dg.Batch([dg.Mesh(synth.tri_mesh(120, 110, 0.2, s)) for s in (1, 2, 3)])
    sch = dg.Scheme(k=k, r=r, n_diff=n_diff, flux="burgers", nv=1, precision=precision)
    ws = bt.workspace(sch)
    u0 = torch.from_numpy(1.0 + 0.1 * np.random.default_rng(6).random((1, sum(M.n_cells for M in bt.meshes)))).cuda()
    dt = torch.full((3,), 1e-4, dtype=torch.float64, device="cuda")
    want = u0.clone()
    bt.rk_step(sch, dt, want, ws, use_graph=False)
    dg.dolinc_sync_status(bt.meshes[0], ws)
    gave_up = 0
    for limit in [0] + list(range(1, 120, 2)):
        bt.set_spin_limit(limit)
        u = u0.clone()
        bt.rk_step(sch, dt, u, ws, use_graph=False)
        try:
            dg.dolinc_sync_status(bt.meshes[0], ws)
            assert torch.equal(u, want), limit
        except dg.DolincError as e:
            assert e.status == 5
            gave_up += 1
            assert torch.equal(u, u0), limit
    assert gave_up > 0
