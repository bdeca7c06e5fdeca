"""The untuned launch shape by size, precision and scheme: every path of a step takes the
same sums (device, host state, parts of a mesh), and the residual's shape below and above
its limit gives the residual of the shapes that can be set."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
dg = pytest.importorskip("paper_2404_08952_gb300")
pytestmark = pytest.mark.gpu

STENCIL = {3: (3, 1), 5: (5, 2)}
MESHES = {
    "tri_small": lambda: synth.tri_mesh(40, 49, 0.2, 1),            # 3,920 cells
    "tri_over": lambda: synth.tri_mesh(40, 51, 0.2, 1),             # 4,080
    "hexprism_small": lambda: synth.hexprism_mesh(12, 0.2, 2),      # 2,592
    "hexprism_over": lambda: synth.hexprism_mesh(15, 0.2, 2),       # 4,950 or so
}


def _setup(name, order, n_diff, values=False):
    m = MESHES[name]()
    if values:
        m = synth.tri_mesh(40, 49, 0.2, 1, boundary="transmissive")
        kind = np.where(np.asarray(m["face_neighbour"]) < 0, 2, 0).astype(np.int32)
        m = dict(m, boundary_kind=kind)
    k, r = STENCIL[order]
    dim = m["dim"]
    sch = dg.Scheme(k=k, r=r, n_diff=n_diff, flux="upwind", nv=1, precision="fp64", adv=(1.0, 0.7, 0.4)[:dim])
    M = dg.Mesh(m)
    if values:
        dg.dolinc_set_boundary_values(M, np.ones((1, M.n_faces)))
    u0 = 1.0 + 0.1 * np.random.default_rng(9).random((1, M.n_cells))
    return m, M, sch, u0


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("order,n_diff", [(3, 1), (3, 2), (3, 4), (5, 3)])
def test_residual_shape(name, order, n_diff):
    m, M, sch, u0 = _setup(name, order, n_diff)
    lanes = 4 if name.startswith("tri") else 8
    u = torch.from_numpy(u0).cuda()
    R = [torch.empty_like(u) for _ in range(3)]
    dg.dolinc_residual(M, sch, u, R[0], dg.workspace(M, sch))
    for i, shape in enumerate(((lanes, 256, lanes, 128), (1, 64, -2, 64))):
        dg.dolinc_set_tuning(M, sch, *shape)
        dg.dolinc_residual(M, sch, u, R[1 + i], dg.workspace(M, sch))
    assert torch.equal(R[0], R[1 if M.n_cells <= 4000 else 2])
    scale = R[1].abs().max().item()
    assert (R[1] - R[2]).abs().max().item() <= 1e-11 * scale


@pytest.mark.parametrize("name,order,n_diff,values", [
    ("tri_small", 3, 2, False), ("tri_small", 3, 4, False), ("tri_small", 5, 3, False), ("tri_small", 3, 2, True),
    ("tri_over", 5, 3, False), ("hexprism_small", 3, 2, False), ("hexprism_small", 5, 4, False),
    ("hexprism_over", 3, 3, False)])
def test_every_path_of_a_step_sums_alike(name, order, n_diff, values):
    m, M, sch, u0 = _setup(name, order, n_diff, values)
    dt = 1e-3
    ws = dg.workspace(M, sch)
    want = torch.from_numpy(u0).cuda()
    dg.dolinc_rk_step(M, sch, dt, want, ws)
    dg.dolinc_sync_status(M, ws)
    want = want.cpu().numpy()
    assert np.abs(want - u0).max() > 0
    host = torch.from_numpy(u0.copy()).pin_memory()
    dg.dolinc_rk_step_host(M, sch, dt, host, torch.empty((1, M.n_cells), dtype=torch.float64, device="cuda"), ws)
    dg.dolinc_sync_status(M, ws)
    np.testing.assert_array_equal(host.numpy(), want)
    u = torch.from_numpy(u0).cuda()
    dg.dolinc_profile_enable(M, True)                    # timed calls take the separate launches
    dg.dolinc_rk_step(M, sch, dt, u, ws)
    dg.dolinc_profile_enable(M, False)
    np.testing.assert_array_equal(u.cpu().numpy(), want)
    # two parts of the mesh
    from test_gpu_partition import exchange_in_process
    pc = dg.dolinc_partition(m, 2)
    parts = [dg.Mesh(m, part=(pc, 2, p)) for p in range(2)]
    orig, whole = M.from_lib(u0), M.from_lib(want)
    wss, us = [], []
    for P in parts:
        if values:
            dg.dolinc_set_boundary_values(P, np.ones((1, P.n_faces)))
        wss.append(dg.workspace(P, sch))
        us.append(torch.from_numpy(orig[:, P.plan["local_cells"]].copy()).cuda())
    hs = [dg.dolinc_part_step_begin(P, sch, dt, x, w) for P, x, w in zip(parts, us, wss)]
    while hs[0].pending:
        exchange_in_process(parts, wss, hs)
        hs = [dg.dolinc_part_step_continue(P, sch, w) for P, w in zip(parts, wss)]
    for P, x, w in zip(parts, us, wss):
        dg.dolinc_sync_status(P, w)
        own = P.plan["owned"].astype(bool)
        np.testing.assert_array_equal(x.cpu().numpy()[:, own], whole[:, P.plan["local_cells"][own]])


@pytest.mark.parametrize("flux,precision,n_diff", [("upwind", "fp32", 2), ("rusanov", "fp32", 2), ("rusanov", "fp32", 1),
                                                   ("burgers", "fp32_bf16", 2)])
@pytest.mark.parametrize("nx", [149, 162])                # 47,680 and 51,840 cells: both sides of the limit
def test_few_passes_give_the_lane_bits_on_both_sides(flux, precision, n_diff, nx):
    m = synth.tri_mesh(nx, 160, 0.2, 3)
    M = dg.Mesh(m)
    nv = 4 if flux == "rusanov" else 1
    sch = dg.Scheme(k=3, r=1, n_diff=n_diff, flux=flux, nv=nv, precision=precision, adv=(1.0, 0.7))
    s = 0.1 * np.random.default_rng(2).random(M.n_cells)
    u0 = torch.from_numpy((1.0 + s)[None] if nv == 1 else np.stack([1.0 + s, 0.4 + s, 0.2 - s, 3.0 + s])).cuda()
    out = []
    for tuned in (False, True):
        if tuned:
            dg.dolinc_set_tuning(M, sch, 4, 256, 4, 128)
        ws = dg.workspace(M, sch)
        u, R = u0.clone(), torch.empty_like(u0)
        dg.dolinc_residual(M, sch, u, R, ws)
        dg.dolinc_rk_steps(M, sch, 1e-4, 2, u, ws)
        dg.dolinc_sync_status(M, ws)
        out.append((u, R))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
