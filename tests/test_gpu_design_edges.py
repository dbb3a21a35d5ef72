"""The OC update and the cone filter where their fast paths can go wrong.

OC against the oracle's bisection (design within 1e-9: both stop at a relative
bracket width of 1e-10 in lambda, so 0.5e-10 in the candidate, and volumes that
differ by summation order can turn one branch): a smooth design, one near 0 and
1, targets out of reach from above and below, breakpoints exactly at the
solution, all elements alike, zero and positive sensitivities, tiny move
limits, sensitivities beyond FP32's range, one element, and a mesh too large
for registers.  Filter and transpose bit for bit against the oracle at the
edges of its tiles, for every stencil of one element and a wider one."""
import numpy as np
import pytest

from oracle import filter as cone, simp as osimp
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMALL, LARGE = (24, 13, 11), (100, 100, 63)   # 630,000 elements: above 152 x 512 x 8


def _oc_case(kind, n):
    """rho, dc, volfrac, move"""
    rng = np.random.default_rng(17)
    rho, dc = rng.uniform(0.05, 0.6, n), -rng.uniform(1e-4, 1.0, n)
    if kind == "near01":
        rho = np.where(rng.random(n) < 0.3, 1.0, 1e-3)
        return rho, -rho ** 2 * rng.lognormal(0, 2, n), 0.3, 0.05
    if kind == "below":          # the lower bounds alone exceed the target
        return rho + 0.4, dc, 0.2, 0.2
    if kind == "above":          # the upper bounds do not reach it
        return rho * 0.5, dc, 0.6, 0.2
    if kind == "breakpoint":     # half of the elements meet their bound at the solution
        rho = np.full(n, 0.3)
        dc = -np.where(np.arange(n) % 2, 1.0, 25.0 / 9.0)
        return rho, dc, 0.4, 0.2
    if kind == "alike":
        return np.full(n, 0.3), np.full(n, -2.5), 0.3, 0.2
    if kind == "mixed_sign":
        return rho, rng.normal(-0.2, 0.5, n), 0.3, 0.2
    if kind == "zeros":
        return np.where(rng.random(n) < 0.4, 0.0, rho), np.where(rng.random(n) < 0.3, 0.0, dc), 0.2, 0.2
    if kind == "tiny_move":
        return rho, dc, float(rho.mean()), 1e-4
    if kind == "huge":
        return rho, dc * 1e90, 0.3, 0.2
    if kind == "small":
        return rho, dc * 1e-12, 0.3, 0.2
    return rho, dc, 0.3, 0.2


def _oc_check(cuda, shape, kind):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*shape)
    rho, dc, volfrac, move = _oc_case(kind, m.n_elem)
    ref, info = osimp.oc_update(rho, dc, volfrac, move)
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8),
                     mfto.default_params(volfrac=volfrac, move=move)) as h:
        out = torch.empty(m.n_elem, dtype=torch.float64, device=cuda)
        st = h.oc_update(torch.tensor(rho, device=cuda), torch.tensor(dc, device=cuda), out)
        again = torch.empty_like(out)
        h.oc_update(torch.tensor(rho, device=cuda), torch.tensor(dc, device=cuda), again)
        assert torch.equal(out, again)
    got = out.cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-9
    assert abs(st.change - info["change"]) <= 1e-9
    assert abs(st.volume - got.mean()) <= 1e-12 * max(1.0, got.mean())
    if kind not in ("breakpoint", "above"):
        assert abs(st.lambda_ - info["lambda"]) <= 4e-10 * info["lambda"]


@pytest.mark.parametrize("kind", ["plain", "near01", "below", "above", "breakpoint", "alike",
                                  "mixed_sign", "zeros", "tiny_move", "huge", "small"])
def test_oc_small(cuda, kind):
    _oc_check(cuda, SMALL, kind)


@pytest.mark.parametrize("kind", ["plain", "near01", "below", "zeros", "breakpoint"])
def test_oc_large(cuda, kind):
    _oc_check(cuda, LARGE, kind)


def test_oc_one_element(cuda):
    _oc_check(cuda, (1, 1, 1), "plain")


@pytest.mark.parametrize("rmin", [1.0, 1.2, 1.5, 1.75, 2.0, 2.3])
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 16, 2), (32, 15, 3), (33, 17, 1), (65, 33, 9),
                                   (3, 2, 40)])
def test_filter_bits(cuda, shape, rmin):
    import torch
    from paper_2604_18020_gb300 import mfto
    m = W.Mesh(*shape)
    x = W.vec_random(m.n_elem, seed=19)
    x[::5] = 0.0
    x[1::7] = -0.0
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8), mfto.default_params(rmin=rmin)) as h:
        tx = torch.tensor(x, device=cuda)
        y = torch.empty_like(tx)
        h.filter(tx, y)
        assert np.array_equal(y.cpu().numpy().view(np.int64),
                              cone.filter_fwd(x, *shape, rmin).view(np.int64))
        h.filter(tx, y, transpose=True)
        assert np.array_equal(y.cpu().numpy().view(np.int64),
                              cone.filter_T(x, *shape, rmin).view(np.int64))
