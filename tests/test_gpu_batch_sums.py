"""The batch's dot products are summed in FP64: loads whose squares fit FP32 (a
warp's 128 sum to at most 2e37) while an instance's sum of them does not (over
1e39) are solved like others (oracle's residual <= 1.5e-8 at rtol 1e-8)."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_large_loads(cuda):
    import torch
    from paper_2604_18020_gb300 import mfto
    meshes = [(48, 24, 24), (24, 12, 12), (48, 24, 24)]
    rng = np.random.default_rng(61)
    fixed, Es, fs = [], [], []
    for shape, size in zip(meshes, (4e17, 4e17, 1.0)):
        m = W.Mesh(*shape)
        # two thirds of the nodes held: displacements of the size of f / E, few iterations
        fixed.append(np.where(rng.random(m.n_node) < 0.67, 7, 0).astype(np.uint8))
        Es.append(rng.uniform(0.5, 1.0, m.n_elem))
        fs.append(np.where(fem.dof_mask(fixed[-1]), 0.0, size * rng.uniform(-1, 1, m.n_dof)))
    assert (fs[0] ** 2).sum() > 1e39
    with mfto.Batch(meshes, fixed) as b:
        U = torch.zeros(b.n_dof, dtype=torch.float64, device=cuda)
        sts = b.solve(torch.tensor(np.concatenate(Es), device=cuda),
                      torch.tensor(np.concatenate(fs), device=cuda), U, inner_tol=1e-2)
        u = U.cpu().numpy()
        offs = b.dof_off
    for i, shape in enumerate(meshes):
        assert sts[i].status == mfto.OK, i
        r = fs[i] - fem.kv(fem.ke_exact(), Es[i], fem.edof_table_fast(*shape),
                           u[offs[i]:offs[i + 1]], fem.dof_mask(fixed[i]))
        assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(fs[i]), i
