"""The FP64 column K.v (kv_column64.cuh) at the edges of its tiles: meshes for
which each of its tile shapes is chosen, node counts one below, at and one
above a tile's owned nodes, one-element axes, several z-chunks, and masks that
fix single components anywhere -- K.v against the oracle (relative inf-norm
<= 1e-12: a few roundings of |KE||v|, as test_gpu_core.py), its CG form through
a PCG solve judged by the oracle's residual (<= 1.5e-8 at rtol 1e-8)."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# on 152 SMs these meshes get the tiles 32x4 (EDGES), 16x8, 32x8, 8x16 and 16x16
EDGES = [(30, 2, 3), (31, 3, 1), (29, 6, 4), (63, 5, 2), (1, 9, 30), (2, 1, 70)]
SHAPES = [(48, 24, 24), (142, 9, 14), (6, 90, 60), (40, 22, 24)]


def _random_mask(m, seed):
    rng = np.random.default_rng(seed)
    fixed = np.where(rng.random(m.n_node) < 0.1, rng.integers(1, 8, m.n_node), 0).astype(np.uint8)
    fixed[:3] = 7
    return fixed


@pytest.mark.parametrize("shape", EDGES + SHAPES)
def test_kv_f64_tiles(cuda, shape):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*shape)
    fixed = _random_mask(m, seed=4)
    fd = fem.dof_mask(fixed)
    E = fem.simp_modulus(W.rho_random(m, seed=5), 3.0)
    v = W.vec_random(m.n_dof, seed=6)
    with mfto.Handle(*shape, fixed) as h:
        y = torch.full((m.n_dof,), float("nan"), dtype=torch.float64, device=cuda)
        h.kv(torch.tensor(E, device=cuda), torch.tensor(v, device=cuda), y)
        got = y.cpu().numpy()
        again = torch.empty_like(y)
        h.kv(torch.tensor(E, device=cuda), torch.tensor(v, device=cuda), again)
        assert torch.equal(again, y)
    ref = fem.kv(fem.ke_exact(), E, fem.edof_table_fast(*shape), v, fd)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.array_equal(got[fd], v[fd])


@pytest.mark.parametrize("shape", [(29, 6, 4), (48, 24, 24), (6, 90, 60), (142, 9, 14), (40, 22, 24)])
def test_pcg_f64_tiles(cuda, shape):
    import torch
    from paper_2604_18020_gb300 import mfto
    P = W.cantilever(*shape)
    m = P.mesh
    E = fem.simp_modulus(W.rho_random(m, seed=7, lo=0.2, hi=1.0), 3.0)
    u = torch.zeros(m.n_dof, dtype=torch.float64, device=cuda)
    with mfto.Handle(*shape, P.fixed, mfto.default_params(rtol=1e-8)) as h:
        st = h.pcg(torch.tensor(E, device=cuda), torch.tensor(P.f, device=cuda), u)
    assert st.status == mfto.OK
    r = P.f - fem.kv(fem.ke_exact(), E, fem.edof_table_fast(*shape), u.cpu().numpy(),
                     fem.dof_mask(P.fixed))
    assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(P.f)
