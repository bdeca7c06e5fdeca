"""One batch handle stepped with several schemes: each takes the grid that its own kernel
allows, so the order of the schemes does not matter, and a shape autotuned for one scheme
serves the others."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
dg = pytest.importorskip("paper_2404_08952_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,nv", [(2, 1), (2, 4), (3, 1), (3, 5)])
@pytest.mark.parametrize("tuned", [False, True])
def test_schemes_in_any_order(dim, nv, tuned):
    mk = (lambda s: synth.tri_mesh(20 + s, 17, 0.2, s)) if dim == 2 else (lambda s: synth.tet_mesh(4 + 2 * (s % 2), 0.15, s))
    meshes = [dg.Mesh(mk(s)) for s in (1, 2, 3)]
    n = sum(M.n_cells for M in meshes)
    s = 0.1 * np.random.default_rng(7).random(n)
    u0 = torch.from_numpy((1.0 + s)[None] if nv == 1 else np.stack([1.0 + s] + [0.3 + s] * dim + [3.0 + s])).cuda()
    dt = torch.full((3,), 1e-4, dtype=torch.float64, device="cuda")
    schemes = [dg.Scheme(k=k, r=r, n_diff=nd, flux="burgers" if nv == 1 else "rusanov", nv=nv, precision=p)
               for k, r, nd in ((3, 1, 2), (5, 2, 3)) for p in ("fp64", "fp32", "fp32_bf16")]

    def run(bt, sch):
        ws = bt.workspace(sch)
        u = u0.clone()
        bt.rk_step(sch, dt, u, ws)
        dg.dolinc_sync_status(meshes[0], ws)
        return u

    want = [run(dg.Batch(meshes), sch) for sch in schemes]
    for first in (0, 1, 4):
        bt = dg.Batch(meshes)
        if tuned:
            bt.autotune(schemes[first], dt, u0.clone(), bt.workspace(schemes[first]))
        for i in [first] + list(range(6)):
            assert torch.equal(run(bt, schemes[i]), want[i]), (first, i)


@pytest.mark.parametrize("dim,nv", [(2, 1), (2, 4), (3, 1), (3, 5)])
def test_large_and_small_batches_give_the_same_bits(dim, nv):
    """Below FP64 a batch of more cells than its first kernel has threads takes another one:
    ten meshes as one batch (about 160k cells) and as ten batches."""
    m = synth.tri_mesh(90, 89, 0.2, 4) if dim == 2 else synth.tet_mesh((14, 16, 14), 0.15, 4)
    meshes = [dg.Mesh(m)] * 10
    n = meshes[0].n_cells
    s = 0.1 * np.random.default_rng(8).random(10 * n)
    u0 = torch.from_numpy((1.0 + s)[None] if nv == 1 else np.stack([1.0 + s] + [0.3 + s] * dim + [3.0 + s])).cuda()
    dt = torch.linspace(1e-4, 3e-4, 10, dtype=torch.float64, device="cuda")

    def run(part, lo):
        bt, hi = dg.Batch(part), lo + len(part)
        u = u0[:, lo * n:hi * n].clone().contiguous()
        ws = bt.workspace(sch)
        for _ in range(2):
            bt.rk_step(sch, dt[lo:hi].clone(), u, ws, use_graph=False)
        dg.dolinc_sync_status(meshes[0], ws)
        return u

    for k, r, nd in ((3, 1, 1), (3, 1, 2), (4, 1, 4), (5, 2, 2), (5, 2, 3)):
        for p in ("fp32", "fp32_bf16"):
            sch = dg.Scheme(k=k, r=r, n_diff=nd, flux="burgers" if nv == 1 else "rusanov", nv=nv, precision=p)
            one = run(meshes, 0)
            assert torch.isfinite(one).all() and not torch.equal(one, u0)
            assert torch.equal(one, torch.cat([run(meshes[:1], i) for i in range(10)], 1)), (k, r, nd, p)
