"""The FP64 operator and energies on the FP64 pipe (kv_column64.cuh,
compliance_kernel), which serve Poisson's ratios outside [0, 0.454) and variant 2:
at the edges of the tiles, in CG, for several load cases and in a batch.  Bounds as
for the fixed-point route: K.v 1e-12 of the largest value, energies 1e-12 of the
largest, solves by the oracle's residual (<= 1.5e-8 at rtol 1e-8)."""
import numpy as np
import pytest

from oracle import fem, simp as osimp
from paper_2604_18020_gb300 import workloads as W
from test_gpu_column64 import EDGES, SHAPES, _random_mask

pytestmark = pytest.mark.gpu

ROUTES = [(0.47, 0), (-0.2, 0), (0.3, 2)]     # Poisson's ratio, variant


@pytest.mark.parametrize("nu,variant", ROUTES)
@pytest.mark.parametrize("shape", [(1, 1, 1)] + EDGES + SHAPES)
def test_kv_and_energies(cuda, shape, nu, variant):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*shape)
    fixed = _random_mask(m, seed=81)
    fd, edof, KE = fem.dof_mask(fixed), fem.edof_table_fast(*shape), fem.ke_exact(1.0, nu)
    rho = W.rho_random(m, seed=82)
    E = fem.simp_modulus(rho, 3.0)
    V = np.stack([W.vec_random(m.n_dof, seed=83 + i) for i in range(3)])
    with mfto.Handle(*shape, fixed, mfto.default_params(nu=nu, max_rhs=3)) as h:
        h.set_kv_variant(variant)
        tE, tV = torch.tensor(E, device=cuda), torch.tensor(V.reshape(-1), device=cuda)
        y = torch.full((m.n_dof,), float("nan"), dtype=torch.float64, device=cuda)
        h.kv(tE, tV[:m.n_dof], y)
        Y = torch.full_like(tV, float("nan"))
        h.kv_multi(tE, tV, Y, 3)
        dc = torch.full((m.n_elem,), float("nan"), dtype=torch.float64, device=cuda)
        c = h.compliance_sens(torch.tensor(rho, device=cuda), tV[:m.n_dof], dc)
        got = [y.cpu().numpy()] + list(Y.cpu().numpy().reshape(3, -1))
        dc = dc.cpu().numpy()
    for g, v in zip(got, [V[0], *V]):
        ref = fem.kv(KE, E, edof, v, fd)
        assert np.abs(g - ref).max() <= 1e-12 * np.abs(ref).max()
        assert np.array_equal(g[fd], v[fd])
    c_ref, dc_ref = osimp.compliance_sens(KE, edof, V[0], rho, 3.0)
    assert np.abs(dc - dc_ref).max() <= 1e-12 * np.abs(dc_ref).max()
    assert abs(c - c_ref) <= 1e-12 * c_ref


@pytest.mark.parametrize("nu,variant", ROUTES)
@pytest.mark.parametrize("shape", [(29, 6, 4), (48, 24, 24), (6, 90, 60), (142, 9, 14)])
def test_solves(cuda, shape, nu, variant):
    import torch
    from paper_2604_18020_gb300 import mfto
    P = W.cantilever(*shape)
    m = P.mesh
    E = fem.simp_modulus(W.rho_random(m, seed=86, lo=0.2, hi=1.0), 3.0)
    with mfto.Handle(*shape, P.fixed, mfto.default_params(nu=nu)) as h:
        h.set_kv_variant(variant)
        for solve in (h.pcg, h.ir_solve):
            u = torch.zeros(m.n_dof, dtype=torch.float64, device=cuda)
            st = solve(torch.tensor(E, device=cuda), torch.tensor(P.f, device=cuda), u)
            assert st.status == mfto.OK
            r = P.f - fem.kv(fem.ke_exact(1.0, nu), E, fem.edof_table_fast(*shape),
                             u.cpu().numpy(), fem.dof_mask(P.fixed))
            assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(P.f)


@pytest.mark.parametrize("nu", [0.47, -0.2])
@pytest.mark.parametrize("shape", [0, 3])
def test_batch(cuda, nu, shape):
    import torch
    from paper_2604_18020_gb300 import mfto
    meshes = [(16, 9, 5), (3, 5, 30), (1, 1, 1), (70, 4, 3)]
    problems = [W.cantilever(*s) for s in meshes]
    Es = [fem.simp_modulus(W.rho_random(P.mesh, seed=87 + i, lo=0.2, hi=1.0), 3.0)
          for i, P in enumerate(problems)]
    vs = [W.vec_random(P.mesh.n_dof, seed=91 + i) for i, P in enumerate(problems)]
    with mfto.Batch(meshes, [P.fixed for P in problems], mfto.default_params(nu=nu)) as b:
        b.set_shape(shape)
        tE = torch.tensor(np.concatenate(Es), device=cuda)
        Y = torch.zeros(b.n_dof, dtype=torch.float64, device=cuda)
        b.kv(tE, torch.tensor(np.concatenate(vs), device=cuda), Y)
        U = torch.zeros_like(Y)
        sts = b.solve(tE, torch.tensor(np.concatenate([P.f for P in problems]), device=cuda), U,
                      inner_tol=1e-2)
        y, u, offs = Y.cpu().numpy(), U.cpu().numpy(), b.dof_off
    for i, P in enumerate(problems):
        op = (fem.ke_exact(1.0, nu), Es[i], fem.edof_table_fast(*meshes[i]))
        fd = fem.dof_mask(P.fixed)
        ref = fem.kv(*op, vs[i], fd)
        assert np.abs(y[offs[i]:offs[i + 1]] - ref).max() <= 1e-12 * np.abs(ref).max(), meshes[i]
        assert sts[i].status == mfto.OK, meshes[i]
        r = P.f - fem.kv(*op, u[offs[i]:offs[i + 1]], fd)
        assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(P.f), meshes[i]
