"""The fixed-point FP64 operator (kv_fixed.cuh) where it can go wrong: tiles and
axes of one element, Poisson's ratios on both sides of its range (outside it the
FP64 column kernel runs), values and moduli over many orders of magnitude,
signs, non-finite entries, exponents near the ends of FP64's range, and strains
far below the displacements.

K.v against the oracle: per node, |error| <= 2^-48 sum over its elements of
|E| max|v_e| ||KE||_inf (the oracle's 24-term products and 8-term sums, in FP64,
and the operator's block error of about 2^-53 of the same bound).  Energies
against extended precision: 64 roundings of the energy, plus what the inputs'
rounding to their node's exponent can change."""
import numpy as np
import pytest

from oracle import fem
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (31, 3, 1), (2, 1, 70), (16, 8, 5), (47, 15, 9)]
NUS = [0.0, 0.1, 0.3, 0.33, 0.4, 0.45, 0.47, -0.2]


def _mask(m, seed):
    rng = np.random.default_rng(seed)
    return np.where(rng.random(m.n_node) < 0.1, rng.integers(1, 8, m.n_node), 0).astype(np.uint8)


def _kv(cuda, shape, fixed, nu, E, v):
    import torch
    from paper_2604_18020_gb300 import mfto
    with mfto.Handle(*shape, fixed, mfto.default_params(nu=nu)) as h:
        y = torch.full((v.size,), float("nan"), dtype=torch.float64, device=cuda)
        h.kv(torch.tensor(E, device=cuda), torch.tensor(v, device=cuda), y)
        return y.cpu().numpy()


def _bound(shape, nu, E, v, fd):
    """Per node: the sum over its elements of |E| max|v_e| ||KE||_inf."""
    edof = fem.edof_table_fast(*shape)
    KE = fem.ke_exact(1.0, nu)
    be = np.abs(E) * np.abs(np.where(fd, 0.0, v))[edof].max(axis=1) * np.abs(KE).sum(axis=1).max()
    nodes = edof[:, ::3] // 3
    return np.repeat(np.bincount(nodes.reshape(-1), weights=np.repeat(be, 8),
                                 minlength=v.size // 3), 3)


def _check(cuda, shape, nu, E, v):
    fixed = _mask(W.Mesh(*shape), 3)
    fd = fem.dof_mask(fixed)
    got = _kv(cuda, shape, fixed, nu, E, v)
    ref = fem.kv(fem.ke_exact(1.0, nu), E, fem.edof_table_fast(*shape), v, fd)
    assert np.array_equal(got[fd], v[fd])
    assert np.all((np.abs(got - ref) <= 2.0 ** -48 * _bound(shape, nu, E, v, fd))[~fd])


@pytest.mark.parametrize("nu", NUS)
@pytest.mark.parametrize("shape", SHAPES)
def test_kv(cuda, shape, nu):
    m = W.Mesh(*shape)
    rng = np.random.default_rng(11)
    _check(cuda, shape, nu, rng.uniform(1e-9, 1.0, m.n_elem), rng.uniform(-1, 1, m.n_dof))


@pytest.mark.parametrize("kind", ["range", "extreme", "scaled_down", "scaled_up", "signs", "zeros"])
def test_kv_values(cuda, kind):
    shape = (21, 9, 6)
    m = W.Mesh(*shape)
    rng = np.random.default_rng(12)
    E, v = rng.uniform(0.1, 1.0, m.n_elem), rng.uniform(-1, 1, m.n_dof)
    if kind == "range":
        E = 10.0 ** rng.uniform(-9, 0, m.n_elem)
        v *= 10.0 ** rng.uniform(-6, 6, m.n_dof)
    elif kind == "extreme":
        v *= 2.0 ** rng.integers(-80, 80, m.n_dof)
    elif kind == "scaled_down":
        v *= 1e-280
    elif kind == "scaled_up":
        v *= 1e300
    elif kind == "signs":
        E *= rng.choice([-1.0, 1.0], m.n_elem)
        v = rng.choice([-1.0, 1.0], m.n_dof)     # the largest sums the operator forms
    elif kind == "zeros":
        E[::3] = 0.0
        v[::2] = 0.0
    _check(cuda, shape, 0.3, E, v)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_kv_non_finite(cuda, bad):
    shape = (18, 9, 4)
    m = W.Mesh(*shape)
    rng = np.random.default_rng(13)
    fixed = np.zeros(m.n_node, np.uint8)
    E, v = rng.uniform(0.1, 1.0, m.n_elem), rng.uniform(-1, 1, m.n_dof)
    v[3 * 401 + 1] = bad
    E[17] = bad
    got = _kv(cuda, shape, fixed, 0.3, E, v)
    with np.errstate(all="ignore"):
        ref = fem.kv(fem.ke_exact(), E, fem.edof_table_fast(*shape), v, fem.dof_mask(fixed))
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))


def _energies(shape, nu, u):
    """Element energies in extended precision from the 1-D integrals."""
    L = np.longdouble
    nu = L(nu)
    lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 1 / (2 * (1 + nu))
    M = np.array([[L(1) / 3, L(1) / 6], [L(1) / 6, L(1) / 3]])
    S = np.array([[1, -1], [-1, 1]], dtype=L)
    D = np.array([[-1, -1], [1, 1]], dtype=L) / 2
    K = np.zeros((24, 24), dtype=L)

    def integral(i, j, a, b):
        r = L(1)
        for ax in range(3):
            p, q = (a >> ax) & 1, (b >> ax) & 1
            r *= S[p, q] if i == j == ax else D[p, q] if i == ax else D[q, p] if j == ax else M[p, q]
        return r

    for a in range(8):
        for b in range(8):
            for i in range(3):
                for j in range(3):
                    t = lam * integral(i, j, a, b) + mu * integral(j, i, a, b)
                    if i == j:
                        t += mu * sum(integral(k, k, a, b) for k in range(3))
                    K[3 * a + i, 3 * b + j] = t
    ue = u.astype(L)[fem.edof_table_fast(*shape)]
    return ((ue @ K) * ue).sum(axis=1)


@pytest.mark.parametrize("kind", ["random", "rotated", "translated", "tiny", "zero"])
@pytest.mark.parametrize("nu", [0.0, 0.3, 0.4, 0.45])
def test_energy(cuda, nu, kind):
    import torch
    from paper_2604_18020_gb300 import mfto
    shape = (33, 17, 5)
    m = W.Mesh(*shape)
    rng = np.random.default_rng(14)
    u = rng.uniform(-1, 1, m.n_dof)
    if kind == "rotated":     # a strain of 1e-6 on a rotation of order 1 (displacements of 50)
        n = np.arange(m.n_node)
        x, y = n % (shape[0] + 1), (n // (shape[0] + 1)) % (shape[1] + 1)
        u *= 1e-6
        u[0::3] -= 1.5 * y
        u[1::3] += 1.5 * x
    elif kind == "translated":
        u = 1e-4 * u + 1000.0
    elif kind == "tiny":
        u *= 1e-120
    elif kind == "zero":
        u[:] = 0.0
    rho = rng.uniform(0.2, 1.0, m.n_elem)
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8), mfto.default_params(nu=nu)) as h:
        dc = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        c = h.compliance_sens(torch.tensor(rho, device=cuda), torch.tensor(u, device=cuda), dc)
        got = dc.cpu().numpy()
    ce = _energies(shape, nu, u)
    ref = (-3.0 * rho ** 2 * (1.0 - 1e-9)) * ce
    # an input error of d per value changes an element's energy by at most this
    # (||KE|| <= 2 / (1 - 2 nu)); d: its node's 57 bits
    d = 2.0 ** -56 * np.abs(u).max()
    lam = 2.0 / (1.0 - 2.0 * nu)
    own = (2.0 * np.sqrt(24 * lam * np.abs(ce)) * d + 24 * lam * d * d).astype(np.float64)
    assert np.all(np.abs(got - ref) <= 64 * 2.0 ** -53 * np.abs(ref) + 3.0 * own)
    E = 1e-9 + (1 - 1e-9) * rho ** 3
    assert abs(c - (E * ce).sum()) <= 64 * 2.0 ** -53 * (E * ce).sum() + own.sum()
