"""The OC update where FP32 copies of its values could mislead it, against the
oracle's bisection (design 1e-9, multiplier 4e-10, as in test_gpu_design_edges.py):
sensitivities whose candidates underflow FP32, designs above their upper bound,
lower bounds that FP32 holds to few bits."""
import numpy as np
import pytest

from oracle import simp as osimp
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMALL, LARGE = (24, 13, 11), (100, 100, 63)


def _check(cuda, shape, rho, dc, volfrac, move, lam_tol=4e-10):
    import torch
    from paper_2604_18020_gb300 import mfto
    ref, info = osimp.oc_update(rho, dc, volfrac, move)
    m = W.Mesh(*shape)
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8),
                     mfto.default_params(volfrac=volfrac, move=move)) as h:
        out = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        st = h.oc_update(torch.tensor(rho, device=cuda), torch.tensor(dc, device=cuda), out)
    got = out.cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-9
    assert abs(st.change - info["change"]) <= 1e-9
    assert abs(st.lambda_ - info["lambda"]) <= lam_tol * info["lambda"]


@pytest.mark.parametrize("size", [1e-60, 1e-80, 1e-95, 1e-200, 1e-290])
def test_small_sensitivities(cuda, size):
    rng = np.random.default_rng(41)
    n = W.Mesh(*SMALL).n_elem
    _check(cuda, SMALL, rng.uniform(0.05, 0.6, n), -size * rng.uniform(1e-4, 1.0, n), 0.35, 0.2)


@pytest.mark.parametrize("over", [0.5, 1e-3])
@pytest.mark.parametrize("shape", [SMALL, LARGE])
def test_designs_above_one(cuda, shape, over):
    """rho - move above 1 (by up to `over`): the lower bound then holds whatever the
    upper one is.  Steep sensitivities there, so that the candidates lie above both."""
    rng = np.random.default_rng(42)
    n = W.Mesh(*shape).n_elem
    above = rng.random(n) < (0.3 if over > 0.1 else 2e-3)
    rho = np.where(above, 1.2 + over * rng.random(n), rng.uniform(0.05, 0.6, n))
    dc = -np.where(above, 100.0, rng.uniform(1e-4, 1.0, n))
    _check(cuda, shape, rho, dc, 0.6 if over > 0.1 else 0.35, 0.2)


@pytest.mark.parametrize("shape", [SMALL, LARGE])
def test_lower_bounds_of_few_fp32_bits(cuda, shape):
    """Densities just above the move limit whose candidates meet their lower bounds
    at the solution: rho - move is known to 1e-8 in FP32, the bounds are 1e-4."""
    rng = np.random.default_rng(43)
    n = W.Mesh(*shape).n_elem
    rho = 0.2 + 10.0 ** rng.uniform(-6.0, -3.0, n)
    cand = (rho - 0.2) * (1.0 + rng.uniform(-2e-4, 2e-4, n))
    free = rng.random(n) < 0.3
    cand[free] = rng.uniform(0.05, 0.35, free.sum())
    dc = -(cand / rho) ** 2 / n          # the candidates at lambda = 1
    volume = np.fmax(rho - 0.2, np.fmin(rho + 0.2, cand)).mean()
    _check(cuda, shape, rho, dc, float(volume), 0.2)


@pytest.mark.parametrize("size", [1e8, 1.0, 1e-20, 2.0 ** -510, 2.0 ** -512, 1e-250])
def test_square_root(cuda, size):
    """Densities of 1/2 and no bound active: the new ones are sqrt(-dc n) times one
    number, each rounded once more.  Their ratios to that root in extended precision
    spread by at most 2 (2^-53 + 1.02 2^-53) if the root is good to 0.51 ulp; on both
    sides of the exponent (2^-511) below which CUDA's sqrt takes over."""
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*LARGE)
    n = m.n_elem
    cand = np.random.default_rng(44).uniform(0.06, 0.94, n)
    dc = -(2.0 * cand) ** 2 * size / n
    with mfto.Handle(*LARGE, np.zeros(m.n_node, np.uint8),
                     mfto.default_params(volfrac=float(cand.mean()), move=0.45)) as h:
        out = torch.empty(n, dtype=torch.float64, device=cuda)
        h.oc_update(torch.full((n,), 0.5, dtype=torch.float64, device=cuda),
                    torch.tensor(dc, device=cuda), out)
    got = out.cpu().numpy()
    assert got.min() > 0.055 and got.max() < 0.945
    root = np.sqrt((dc * -float(n)).astype(np.longdouble))
    ratio = got.astype(np.longdouble) / root
    assert ratio.max() / ratio.min() - 1 <= 2.02 * 2.0 ** -52
