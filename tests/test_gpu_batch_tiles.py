"""The batch's tiles (batch_cg.cuh, the FP64 tile list) at their edges: meshes one
node below, at and above the widest row, cut in x, y and z, one-element axes, one
instance -- K.V FP64 per instance against the oracle, and the mixed solve judged
by the oracle's residual (<= 1.5e-8 at rtol 1e-8)."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MESHES = [(63, 4, 3), (64, 5, 4), (62, 3, 2), (130, 2, 3), (1, 1, 1), (2, 127, 2), (3, 5, 90),
          (16, 16, 16), (31, 8, 7), (1, 40, 3)]


@pytest.mark.parametrize("meshes", [MESHES, MESHES[3:4], [(8, 4, 4)] * 40])
def test_batch_tiles(cuda, meshes):
    import torch
    from paper_2604_18020_gb300 import mfto
    problems = [W.cantilever(*s) for s in meshes]
    Es = [fem.simp_modulus(W.rho_random(P.mesh, seed=50 + i, lo=0.2, hi=1.0), 3.0)
          for i, P in enumerate(problems)]
    fs = [P.f for P in problems]
    vs = [W.vec_random(P.mesh.n_dof, seed=70 + i) for i, P in enumerate(problems)]
    with mfto.Batch(meshes, [P.fixed for P in problems]) as b:
        tE = torch.tensor(np.concatenate(Es), device=cuda)
        Y = torch.zeros(b.n_dof, dtype=torch.float64, device=cuda)
        b.kv(tE, torch.tensor(np.concatenate(vs), device=cuda), Y, form=mfto.FORMS["f64"])
        y = Y.cpu().numpy()
        U = torch.zeros(b.n_dof, dtype=torch.float64, device=cuda)
        sts = b.solve(tE, torch.tensor(np.concatenate(fs), device=cuda), U, inner_tol=1e-2)
        u = U.cpu().numpy()
        offs = b.dof_off
    for i, P in enumerate(problems):
        op = (fem.ke_exact(), Es[i], fem.edof_table_fast(*meshes[i]))
        fd = fem.dof_mask(P.fixed)
        ref = fem.kv(*op, vs[i], fd)
        assert np.abs(y[offs[i]:offs[i + 1]] - ref).max() <= 1e-12 * np.abs(ref).max(), meshes[i]
        assert sts[i].status == mfto.OK, meshes[i]
        r = fs[i] - fem.kv(*op, u[offs[i]:offs[i + 1]], fd)
        assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(fs[i]), meshes[i]
