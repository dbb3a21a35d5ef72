"""The fixed-point FP64 operator and energies where one size does not govern: a
component that is far larger than the others, stiff parts moved rigidly inside
soft ones, values and moduli near the lower end of FP64's range.

References are the oracle's with the part that contributes exactly nothing left
out: a uniform translation (no DOF is fixed here) or the elements of a rigid
part, which the operator maps to zero.  Bounds are those of
test_gpu_fixed_point.py for what remains: per node 2^-48 sum |E| max|v_e|
||KE||_inf, and 64 roundings of an energy."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W
from test_gpu_fixed_point import _bound, _energies, _kv

pytestmark = pytest.mark.gpu

SHAPE = (18, 10, 7)


def _moved(m, axis, size, seed):
    """(v, what remains of it): components of order 1, one of them a translation."""
    v = np.random.default_rng(seed).uniform(-1, 1, m.n_dof)
    rest = v.copy()
    v[axis::3] = size * 0.7309
    rest[axis::3] = 0.0
    return v, rest


@pytest.mark.parametrize("nu", [0.0, 0.3, 0.4, 0.45])
@pytest.mark.parametrize("size", [30.0, 1e4, 1e9, 1e18])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_kv_translated_component(cuda, axis, size, nu):
    m = W.Mesh(*SHAPE)
    E = np.random.default_rng(21).uniform(0.01, 1.0, m.n_elem)
    v, rest = _moved(m, axis, size, 22)
    none = np.zeros(m.n_node, np.uint8)
    got = _kv(cuda, SHAPE, none, nu, E, v)
    ref = fem.kv(fem.ke_exact(1.0, nu), E, fem.edof_table_fast(*SHAPE), rest, fem.dof_mask(none))
    assert np.all(np.abs(got - ref) <= 2.0 ** -48 * _bound(SHAPE, nu, E, rest, fem.dof_mask(none)))


@pytest.mark.parametrize("motion", ["translation", "rotation"])
def test_kv_rigid_stiff_part(cuda, motion):
    m = W.Mesh(*SHAPE)
    nx, ny = SHAPE[0] + 1, SHAPE[1] + 1
    node = np.arange(m.n_node)
    x, y, z = node % nx, (node // nx) % ny, node // (nx * ny)
    inside = (x >= 5) & (x <= 11) & (y >= 3) & (y <= 7) & (z >= 2) & (z <= 5)
    v = np.zeros(m.n_dof)
    if motion == "translation":
        v[0::3] = inside * 1.0
    else:
        v[0::3], v[1::3] = inside * -(y - 5.0), inside * (x - 8.0)
    edof = fem.edof_table_fast(*SHAPE)
    stiff = inside[edof[:, ::3] // 3].all(axis=1)
    soft = np.where(stiff, 0.0, 1.2345e-9)
    none = np.zeros(m.n_node, np.uint8)
    got = _kv(cuda, SHAPE, none, 0.3, np.where(stiff, 1.0, soft), v)
    ref = fem.kv(fem.ke_exact(), soft, edof, v, fem.dof_mask(none))
    assert np.all(np.abs(got - ref) <= 2.0 ** -48 * _bound(SHAPE, 0.3, soft, v, fem.dof_mask(none)))


@pytest.mark.parametrize("nu", [0.0, 0.3, 0.45])
@pytest.mark.parametrize("size", [30.0, 1e4, 1e9, 1e18])
def test_energy_translated_component(cuda, size, nu):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*SHAPE)
    u, rest = _moved(m, 0, size, 23)
    rho = np.random.default_rng(24).uniform(0.2, 1.0, m.n_elem)
    with mfto.Handle(*SHAPE, np.zeros(m.n_node, np.uint8), mfto.default_params(nu=nu)) as h:
        dc = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        h.compliance_sens(torch.tensor(rho, device=cuda), torch.tensor(u, device=cuda), dc)
        got = dc.cpu().numpy()
    ref = (-3.0 * rho ** 2 * (1.0 - 1e-9)) * _energies(SHAPE, nu, rest)
    assert np.all(np.abs(got - ref) <= 64 * 2.0 ** -53 * np.abs(ref))


@pytest.mark.parametrize("nu", [0.0, 0.3])
def test_variant_2_runs_on_the_fp64_pipe(cuda, nu):
    """Beside a shear of another component (exact in FP64) x forces keep their
    own precision, which a block's common exponent does not give them."""
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*SHAPE)
    E = np.random.default_rng(25).uniform(0.01, 1.0, m.n_elem)
    rest = np.random.default_rng(26).uniform(-1, 1, m.n_dof)
    rest[1::3] = rest[2::3] = 0.0
    v = rest.copy()
    v[1::3] = 2.0 ** 30 * (np.arange(m.n_node) // ((SHAPE[0] + 1) * (SHAPE[1] + 1)))
    none = np.zeros(m.n_node, np.uint8)
    ref = fem.kv(fem.ke_exact(1.0, nu), E, fem.edof_table_fast(*SHAPE), rest, fem.dof_mask(none))
    bound = 2.0 ** -48 * _bound(SHAPE, nu, E, rest, fem.dof_mask(none))
    with mfto.Handle(*SHAPE, none, mfto.default_params(nu=nu)) as h:
        y = torch.empty(m.n_dof, dtype=torch.float64, device=cuda)
        tE, tv = torch.tensor(E, device=cuda), torch.tensor(v, device=cuda)
        first = torch.empty_like(y)
        h.kv(tE, tv, first)
        h.set_kv_variant(2)
        h.kv(tE, tv, y)
        assert np.all((np.abs(y.cpu().numpy() - ref) <= bound)[0::3])
        h.set_kv_variant(0)
        h.kv(tE, tv, y)
        assert torch.equal(y, first)


# powers of two: inputs are whole numbers times 2^low, the reference is formed at 2^0
@pytest.mark.parametrize("low", [-1074, -1060, -1040, -1000, -960, -900])
def test_kv_lower_end_values(cuda, low):
    m = W.Mesh(*SHAPE)
    E = np.random.default_rng(27).uniform(0.1, 1.0, m.n_elem)
    whole = np.random.default_rng(28).integers(-2 ** 30, 2 ** 30, m.n_dof).astype(np.float64)
    whole[::7] %= 5.0            # small ones among them
    none = np.zeros(m.n_node, np.uint8)
    fd = fem.dof_mask(none)
    got = _kv(cuda, SHAPE, none, 0.3, E, np.ldexp(whole, low))
    ref = fem.kv(fem.ke_exact(), E, fem.edof_table_fast(*SHAPE), whole, fd)
    err = np.abs(np.ldexp(np.ldexp(got, 500), -low - 500) - ref)
    # half a unit of the last subnormal place where the result is subnormal
    assert np.all(err <= 2.0 ** -48 * _bound(SHAPE, 0.3, E, whole, fd) + np.ldexp(0.51, -1074 - low))


@pytest.mark.parametrize("low", [-1074, -1060, -1030, -1000])
def test_kv_lower_end_moduli(cuda, low):
    m = W.Mesh(*SHAPE)
    whole = np.random.default_rng(29).integers(1, 2 ** 40, m.n_elem).astype(np.float64)
    whole[::5] %= 7.0            # zeros and single bits among them
    v = np.random.default_rng(30).uniform(-1.0, 1.0, m.n_dof)
    none = np.zeros(m.n_node, np.uint8)
    fd = fem.dof_mask(none)
    got = np.ldexp(_kv(cuda, SHAPE, none, 0.3, np.ldexp(whole, low), np.ldexp(v, 900)), -900 - low)
    ref = fem.kv(fem.ke_exact(), whole, fem.edof_table_fast(*SHAPE), v, fd)
    assert np.all(np.abs(got - ref) <= 2.0 ** -48 * _bound(SHAPE, 0.3, whole, v, fd))
