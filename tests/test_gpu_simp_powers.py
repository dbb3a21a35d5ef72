"""Compliance, sensitivities and moduli against the oracle over the penalties
a continuation uses (products: multiples of 1/2 up to 8) and others (pow), with
densities that include 0, 1, the smallest normal number and values above 1,
on meshes at the edges of the compliance kernel's tiles (1e-12 relative, as
test_gpu_core.py; moduli within 4 ulp)."""
import numpy as np
import pytest

from oracle import fem, simp as osimp
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _densities(m, seed):
    rho = W.rho_random(m, seed=seed)
    rho[::7] = 0.0
    rho[1::11] = 1.0
    rho[2::13] = 2.2250738585072014e-308
    rho[3::17] = 1.75
    return rho


@pytest.mark.parametrize("penal", [1.0, 1.5, 2.0, 2.5, 3.0, 3.5, 4.5, 8.0, 8.5, 2.7])
def test_modulus(cuda, penal):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(13, 7, 5)
    rho = _densities(m, 1)
    with mfto.Handle(13, 7, 5, np.zeros(m.n_node, np.uint8),
                     mfto.default_params(penal=penal)) as h:
        E = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        h.simp_modulus(torch.tensor(rho, device=cuda), E)
    ref = fem.simp_modulus(rho, penal)
    assert np.all(np.abs(E.cpu().numpy() - ref) <= 4 * np.spacing(ref))


@pytest.mark.parametrize("penal", [1.0, 1.5, 3.0, 2.7])
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 4, 2), (32, 8, 3), (33, 9, 7), (3, 40, 9),
                                   (48, 24, 24), (70, 70, 31)])
def test_compliance(cuda, shape, penal):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*shape)
    rho = _densities(m, 2)
    u = W.vec_random(m.n_dof, seed=3)
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8),
                     mfto.default_params(penal=penal)) as h:
        dc = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        c = h.compliance_sens(torch.tensor(rho, device=cuda), torch.tensor(u, device=cuda), dc)
    c_ref, dc_ref = osimp.compliance_sens(fem.ke_exact(), fem.edof_table_fast(*shape), u, rho,
                                          penal)
    assert abs(c - c_ref) <= 1e-12 * abs(c_ref)
    assert np.abs(dc.cpu().numpy() - dc_ref).max() <= 1e-12 * np.abs(dc_ref).max()
