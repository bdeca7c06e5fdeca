"""Branches that only larger calls take: the semi-implicit solve with some of its vectors
outside shared memory (from about 584k cells on 152 SMs), and a gradient whose thread
blocks take several tiles of rows (more than 19,456 rows)."""
import numpy as np
import pytest

import oracle
import oracle.mlp as omlp
import synth

torch = pytest.importorskip("torch")
dg = pytest.importorskip("paper_2404_08952_gb300")
pytestmark = pytest.mark.gpu

from test_gpu_implicit import cfl_dt, oracle_matrix, schemes, to_dev  # noqa: E402


@pytest.mark.parametrize("n,held", [(75, 6), (79, 5), (85, 4), (92, 0)])
def test_solve_with_vectors_outside_shared_memory(n, held):
    """The increment satisfies the oracle's equation row by row; held: the vectors that a
    chunk's shared memory holds (0: the kernel of larger meshes)."""
    m = synth.hexprism_mesh(n, 0.2, 31)
    O = oracle.Oracle(m, parallel=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        chunk = ((O.n_cells + sms - 1) // sms + 31) // 32 * 32
        fit = (226 * 1024 - 4 * 512 * 8) // 8 // chunk
        assert (fit if fit >= 4 else 0) == held
    adv = (1.0, 1.0, 1.0)
    M = dg.Mesh(m, renumber="morton")
    sd, so = schemes(3, 1, adv)
    dt = cfl_dt(O, adv, 4.0)
    S = dg.Implicit(M, sd, dt, 1.0)
    S.set_solver(rel_tol=1e-12)
    ws = dg.workspace(M, sd)
    xc = O.xc
    u = (np.sin(2 * np.pi * xc[:, 0]) * np.cos(2 * np.pi * xc[:, 1]) + 0.3 * np.sin(2 * np.pi * xc[:, 2])
         + 1e-3 * np.random.default_rng(2).standard_normal(O.n_cells))[None, :]
    ud = to_dev(M, u)
    S.step(ud, ws)
    info = S.info()
    assert info["converged"], info
    delta = M.from_lib(ud.cpu().numpy())[0] - u[0]
    b = O.V * O.residual(u, so)[0]
    A = oracle_matrix(O, so, dt, 1.0)
    assert np.abs(A @ delta - b).max() <= 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("n", [19456, 19457, 50011])
def test_gradient_over_several_tiles_per_block(n):
    rng = np.random.default_rng(n)
    theta = omlp.init(11)
    X = np.abs(rng.normal(size=(n, 24))).astype(np.float32)
    y = (rng.uniform(size=n) < 0.2).astype(np.uint8)
    net = dg.MLP(seed=2)
    net.set_params(theta)
    g = torch.zeros(dg.MLP_PARAMS, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    net.loss_grad(xd, yd, 3.0, g, loss)
    L, G = omlp.loss_and_grad(theta, X.astype(np.float64), y, pos_weight=3.0, weights_bf16=True)
    assert abs(loss.item() - L) < 1e-4 * abs(L)
    assert np.abs(g.cpu().numpy() - G).max() < 1e-3 * np.abs(G).max()
    again = torch.zeros_like(g)
    net.loss_grad(xd, yd, 3.0, again, loss)
    assert torch.equal(g, again)                          # summed in a fixed order
