"""A solve after mfto_set_params applies the new operator throughout: with the same
handle and vectors (whose launches the first solve captured), Poisson's ratio
changed within the fixed-point range, to either side of it and back.  Judged by the
oracle's residual (<= 1.5e-8 at rtol 1e-8)."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", ["pcg", "mixed", "mixed_engine_0", "multi", "gmg", "gmg_mixed"])
def test_solves_follow_the_parameters(cuda, solver):
    import torch
    from paper_2604_18020_gb300 import mfto
    shape = (16, 10, 8)
    P = W.cantilever(*shape)
    m = P.mesh
    fd, edof = fem.dof_mask(P.fixed), fem.edof_table_fast(*shape)
    E = fem.simp_modulus(W.rho_random(m, seed=71, lo=0.3, hi=1.0), 3.0)
    tE, tf = torch.tensor(E, device=cuda), torch.tensor(P.f, device=cuda)
    many = 2 if solver == "multi" else 1
    tF = tf.repeat(many)
    u = torch.zeros(many * m.n_dof, dtype=torch.float64, device=cuda)
    with mfto.Handle(*shape, P.fixed, mfto.default_params(max_rhs=2)) as h:
        for nu in (0.3, 0.1, 0.47, -0.2, 0.3):
            h.set_params(mfto.default_params(nu=nu, max_rhs=2))
            u.zero_()
            if solver == "pcg":
                st = h.pcg(tE, tf, u)
            elif solver == "multi":
                st = h.ir_solve_multi(tE, tF, u, 2)[1]
            elif solver.startswith("mixed"):
                h.set_cg_engine(0 if solver.endswith("0") else 2)
                st = h.ir_solve(tE, tf, u)
            else:
                h.gmg_setup(tE, mfto.default_gmg_params(mixed=int(solver == "gmg_mixed")))
                st = h.gmg_solve(tE, tf, u)
            assert st.status == mfto.OK, nu
            got = u.cpu().numpy().reshape(many, -1)[-1]
            r = P.f - fem.kv(fem.ke_exact(1.0, nu), E, edof, got, fd)
            assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(P.f), nu
