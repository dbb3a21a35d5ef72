"""The fixed-point FP64 operator (kv_fixed.cuh) where it can go wrong: tiles and
axes of one element, Poisson's ratios on both sides of its range (outside it the
FP64 column kernel runs), values and moduli over many orders of magnitude,
signs, non-finite entries and exponents near the ends of FP64's range.

K.v against the oracle: per node, |error| <= 2^-48 sum over its elements of
|E| max|v_e| ||KE||_inf (the oracle's 24-term products and 8-term sums, in FP64,
and the operator's block error of about 2^-53 of the same bound)."""
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
