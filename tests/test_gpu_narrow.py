"""FP64 <-> FP32 conversions by integer operations: boundary face states return the cell
value through both, so they must equal numpy's round-to-nearest conversion bit for bit."""
import numpy as np
import pytest

import synth
import paper_2404_08952_gb300 as dg

pytestmark = pytest.mark.gpu


def test_boundary_states_are_the_rounded_cell_values():
    import torch
    m = synth.tri_mesh(4, 2000, boundary="transmissive")
    M = dg.Mesh(m)
    sch = dg.Scheme(k=2, r=1, n_diff=1, flux="upwind", nv=1, precision="fp32", adv=(1.0, 0.5))
    rng = np.random.default_rng(0)
    n = M.n_cells
    u = rng.standard_normal(n) * 10.0 ** rng.integers(-50, 45, n)              # subnormal results and overflow too
    f = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32).view(np.float32).astype(np.float64)
    pick = rng.integers(0, 6, n)
    ulp = np.spacing(np.abs(f.astype(np.float32))).astype(np.float64)
    with np.errstate(invalid="ignore", over="ignore"):
        u = np.where(pick == 0, f, u)
        u = np.where(pick == 1, f + 0.5 * ulp, u)                                # ties
        u = np.where(pick == 2, f + 0.5 * ulp * (1 + 2.0 ** -28), u)             # just above a tie
        u = np.where(pick == 3, rng.standard_normal(n), u)
        sp = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028234663852886e38, 3.4028235677973366e38,
                       1.1754943508222875e-38, 1.1754943e-38, 1.401298464324817e-45, 7e-46, 5e-324, 1.7e308])
        u[::17] = sp[np.arange(u[::17].size) % sp.size]
        want = u.astype(np.float32).astype(np.float64)
    ws = dg.workspace(M, sch)
    fL = torch.zeros((1, M.n_faces), dtype=torch.float64, device="cuda")
    fR = torch.zeros_like(fL)
    dg.dolinc_reconstruct_faces(M, sch, torch.from_numpy(M.to_lib(u[None])).cuda(), fL, fR, ws)
    b = m["face_neighbour"] < 0
    got = fL.cpu().numpy()[0][b]
    exp = want[m["face_owner"][b]]
    assert b.sum() > 4000
    np.testing.assert_array_equal(np.isnan(got), np.isnan(exp))
    ok = ~np.isnan(exp)
    np.testing.assert_array_equal(got[ok].view(np.uint64), exp[ok].view(np.uint64))
