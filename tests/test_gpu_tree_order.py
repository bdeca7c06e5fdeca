"""The untuned launch shape of larger meshes (one thread per cell, face-centric stage)
sums in the order of one lane per face slot, so below FP64 it gives the bits of that
shape, which smaller meshes use and dolinc_set_tuning selects."""
import numpy as np
import pytest

import synth
import paper_2404_08952_gb300 as dg

pytestmark = pytest.mark.gpu

STENCIL = {2: (2, 1), 3: (3, 1), 4: (4, 1), 5: (5, 2)}


def _mesh(name):
    if name == "tri":
        return synth.tri_mesh(150, 137, jitter=0.2, seed=1)
    if name == "tri_open":
        return synth.tri_mesh(143, 145, jitter=0.2, seed=2, boundary="transmissive")
    if name == "tet":
        return synth.tet_mesh((20, 22, 20), jitter=0.15, seed=3)
    if name == "hexprism":
        return synth.hexprism_mesh((31, 32, 33), jitter=0.2, seed=4)
    return synth.hex_mesh(np.linspace(0, 1, 36), np.linspace(0, 1, 37), np.linspace(0, 1, 35) ** 1.3,
                          periodic=(True, True, False))


@pytest.mark.parametrize("name,flux,order,n_diff,precision,limiter", [
    ("tri", "upwind", 3, 2, "fp32", "none"),
    ("tri", "burgers", 4, 3, "fp32_bf16", "none"),
    ("tri_open", "rusanov", 3, 2, "fp32", "weno5_all"),
    ("tri_open", "rusanov", 2, 1, "fp32_bf16", "none"),
    ("tri_open", "rusanov", 3, 2, "fp32", "eno3_all"),
    ("tri_open", "rusanov", 3, 2, "fp32", "weno5_flagged"),
    ("tri", "rusanov", 4, 2, "fp32_bf16", "eno3_flagged"),
    ("tet", "rusanov", 3, 2, "fp32", "weno5_flagged"),
    ("hexprism", "rusanov", 5, 3, "fp32", "weno5_flagged"),
    ("hexprism", "upwind", 3, 2, "fp32", "eno3_flagged"),
    ("tet", "rusanov", 3, 2, "fp32", "none"),
    ("tet", "rusanov", 4, 3, "fp32_bf16", "eno3_all"),
    ("tet", "rusanov", 5, 4, "fp32", "none"),
    ("hexprism", "upwind", 5, 4, "fp32", "none"),
    ("hexprism", "upwind", 3, 2, "fp32_bf16", "none"),
    ("hexprism", "rusanov", 3, 2, "fp32", "none"),
    ("hexprism", "rusanov", 5, 4, "fp32", "none"),
    ("hex", "rusanov", 4, 3, "fp32", "none"),
    ("hex", "upwind", 5, 4, "fp32_bf16", "none"),
])
def test_untuned_shape_gives_the_lane_shape_bits(name, flux, order, n_diff, precision, limiter):
    import torch
    m = _mesh(name)
    M = dg.Mesh(m)
    assert M.n_cells >= 40000
    dim = M.dim
    nv = dim + 2 if flux == "rusanov" else 1
    k, r = STENCIL[order]
    sch = dg.Scheme(k=k, r=r, n_diff=n_diff, flux=flux, nv=nv, precision=precision, limiter=limiter,
                    adv=(1.0, 0.7, -0.4)[:dim])
    rng = np.random.default_rng(5)
    xc = M.geometry()["xc"]
    s = 0.3 * np.sin(2 * np.pi * xc[:, 0] + 1.0) * np.cos(2 * np.pi * xc[:, 1]) + 0.02 * rng.random(M.n_cells)
    if nv == 1:
        u0 = (1.0 + s)[None]
    else:
        u0 = np.stack([1.0 + s] + [0.4 + 0.2 * np.roll(s, 7 * d) for d in range(dim)] + [3.0 + 0.5 * s])
    lanes = 4 if name in ("tri", "tri_open", "tet") else 8
    flags = torch.from_numpy((np.sin(9 * xc[:, 0]) * np.sin(7 * xc[:, 1]) > 0.9).astype(np.uint8)).cuda()
    dg.dolinc_set_flags(M, flags)

    def run():
        ws = dg.workspace(M, sch)
        u = torch.from_numpy(u0).cuda()
        R = torch.empty_like(u)
        dg.dolinc_residual(M, sch, u, R, ws)
        dg.dolinc_rk_steps(M, sch, 1e-3, 2, u, ws)
        d = torch.zeros(dg.dolinc_diff_layout(M, sch, n_diff)[3] + 256, dtype=torch.uint8, device="cuda")
        d = d[(-d.data_ptr()) % 256:]
        dg.dolinc_differentials(M, sch, torch.from_numpy(u0).cuda(), n_diff, d, ws)
        return [R.cpu().numpy(), u.cpu().numpy()] + dg.diff_to_numpy(M, sch, d, n_diff)

    got = run()
    dg.dolinc_set_tuning(M, sch, lanes, 256, lanes, 128)
    want = run()
    for a, b in zip(got, want):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("name,args,flux,order,n_diff,precision,limiter", [
    ("tri_mesh", (3, 4), "upwind", 3, 2, "fp64", "none"),
    ("tri_mesh", (64, 64), "upwind", 3, 2, "fp64", "none"),
    ("tri_mesh", (45, 37), "rusanov", 3, 2, "fp32", "first_order_flagged"),
    ("tri_mesh", (37, 29), "burgers", 4, 2, "fp32_bf16", "none"),
    ("tri_mesh", (150, 133), "rusanov", 2, 1, "fp32", "none"),
    ("tet_mesh", ((4, 6, 4),), "rusanov", 3, 2, "fp32", "none"),
    ("tet_mesh", ((12, 10, 12),), "rusanov", 3, 1, "fp64", "none"),
    ("hexprism_mesh", ((20, 21, 22),), "upwind", 4, 2, "fp64", "none"),
    ("hexprism_mesh", ((5, 6, 7),), "upwind", 3, 2, "fp32", "none"),
    ("hexprism_mesh", ((20, 21, 22),), "rusanov", 4, 2, "fp32_bf16", "none"),
])
def test_steps_of_a_small_mesh_in_one_launch(name, args, flux, order, n_diff, precision, limiter):
    """Untuned steps of small meshes run in one cooperative launch: the bits of the separate
    launches, also under stream capture, and a second call starts from clean barriers."""
    import torch
    m = getattr(synth, name)(*args, jitter=0.15, seed=7)
    M = dg.Mesh(m)
    assert M.n_cells <= 40000
    dim = M.dim
    nv = dim + 2 if flux == "rusanov" else 1
    k, r = STENCIL[order]
    sch = dg.Scheme(k=k, r=r, n_diff=n_diff, flux=flux, nv=nv, precision=precision, limiter=limiter,
                    adv=(1.0, 0.7, -0.4)[:dim])
    rng = np.random.default_rng(6)
    s = 0.1 * rng.random(M.n_cells)
    u0 = (1.0 + s)[None] if nv == 1 else np.stack([1.0 + s] + [0.4 + s] * dim + [3.0 + s])
    flags = torch.from_numpy((rng.random(M.n_cells) < 0.3).astype(np.uint8)).cuda()
    if limiter != "none":
        dg.dolinc_set_flags(M, flags)
    ws = dg.workspace(M, sch)
    dt = 2e-3 / round(M.n_cells ** (1.0 / dim))
    u = torch.from_numpy(u0).cuda()
    dg.dolinc_rk_step(M, sch, dt, u, ws)
    dg.dolinc_rk_steps(M, sch, dt, 3, u, ws)
    got = u.cpu().numpy()
    u.copy_(torch.from_numpy(u0))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dg.dolinc_rk_steps(M, sch, dt, 4, u, ws)
    g.replay()
    captured = u.cpu().numpy()
    dg.dolinc_sync_status(M, ws)
    lanes = 4 if name != "hexprism_mesh" else 8
    dg.dolinc_set_tuning(M, sch, *((1, 64, -2, 64) if precision == "fp64" else (lanes, 256, lanes, 128)))
    u.copy_(torch.from_numpy(u0))
    dg.dolinc_rk_steps(M, sch, dt, 4, u, ws)
    want = u.cpu().numpy()
    assert np.abs(want - u0).max() > 0
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(captured, want)
