"""Wide, flat meshes: more tiles of element columns than one grid reduction has
partial sums (16,384), for the operator in fixed point and on the FP64 pipe."""
import numpy as np
import pytest

from oracle import fem, solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [0.3, 0.47])
@pytest.mark.parametrize("shape", [(2100, 2100, 1), (1500, 1500, 4)])
def test_compliance_on_wide_meshes(cuda, shape, nu):
    """A constant strain with displacements exact in FP64: one energy everywhere,
    to a few roundings; the sum over 4.4 (9) million equal elements likewise."""
    import torch
    from paper_2604_18020_gb300 import mfto
    nx, ny, nz = (s + 1 for s in shape)
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device=cuda)
                               for n in (nz, ny, nx)), indexing="ij")
    u = torch.stack([x / 16 + y / 64, -y / 32, z / 8 - x / 128], dim=-1).reshape(-1)
    c = np.array([[i & 1, i >> 1 & 1, i >> 2] for i in range(8)], dtype=np.float64)
    ue = np.stack([c[:, 0] / 16 + c[:, 1] / 64, -c[:, 1] / 32, c[:, 2] / 8 - c[:, 0] / 128],
                  axis=-1).reshape(-1)
    ce = ue @ fem.ke_exact(1.0, nu) @ ue
    with mfto.Handle(*shape, np.zeros(nx * ny * nz, np.uint8), mfto.default_params(nu=nu)) as h:
        rho = torch.full((h.n_elem,), 0.5, dtype=torch.float64, device=cuda)
        dc = torch.full_like(rho, float("nan"))
        total = h.compliance_sens(rho, u, dc)
        ref = -3.0 * 0.25 * (1.0 - 1e-9) * ce
        assert (dc - ref).abs().max().item() <= 1e-13 * abs(ref)
        E = 1e-9 + (1.0 - 1e-9) * 0.125
        assert abs(total - h.n_elem * E * ce) <= 1e-11 * h.n_elem * E * ce


@pytest.mark.parametrize("nu", [0.3, 0.47, -0.2])
def test_pcg_on_wide_meshes(cuda, nu):
    """Two FP64 CG iterations against the oracle's recurrence: the CG operator takes
    a tile shape that leaves at most 16,384 partial sums."""
    import torch
    from paper_2604_18020_gb300 import mfto
    shape = (1400, 1400, 1)
    nx, ny, nz = (s + 1 for s in shape)
    fixed = np.zeros(nx * ny * nz, np.uint8)
    fixed[::nx] = 7
    fd = fem.dof_mask(fixed)
    rng = np.random.default_rng(31)
    E = rng.uniform(0.5, 1.0, shape[0] * shape[1] * shape[2])
    f = np.where(fd, 0.0, rng.uniform(-1.0, 1.0, 3 * fixed.size))
    KE, edof = fem.ke_exact(1.0, nu), fem.edof_table_fast(*shape)
    d = fem.jacobi_diag(KE, E, edof, fd)
    u, _ = solve.pcg(lambda v: fem.kv(KE, E, edof, v, fd), d, f, np.zeros_like(f), 1e-8, 2)
    with mfto.Handle(*shape, fixed, mfto.default_params(nu=nu, maxit=2, check_every=2)) as h:
        got = torch.zeros(h.n_dof, dtype=torch.float64, device=cuda)
        st = h.pcg(torch.tensor(E, device=cuda), torch.tensor(f, device=cuda), got)
        assert st.status == mfto.NOT_CONVERGED and st.iterations == 2
    assert np.abs(got.cpu().numpy() - u).max() <= 1e-12 * np.abs(u).max()
