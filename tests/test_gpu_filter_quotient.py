"""The streamed cone filter's own quotient by the row sum, and the division it
keeps for exponents near the ends of FP64's range: bit for bit the oracle's."""
import numpy as np
import pytest

from oracle import filter as cone
from paper_2604_18020_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rmin", [1.35, 1.5, 2.0])
def test_filter_quotients(cuda, rmin):
    import torch
    from paper_2604_18020_gb300 import mfto
    shape = (40, 19, 7)
    m = W.Mesh(*shape)
    rng = np.random.default_rng(15)
    x = rng.uniform(-1, 1, m.n_elem) * 2.0 ** rng.integers(-1070, 900, m.n_elem)
    x[:m.n_elem // 2] = rng.uniform(0, 1, m.n_elem // 2)
    with mfto.Handle(*shape, np.zeros(m.n_node, np.uint8), mfto.default_params(rmin=rmin)) as h:
        tx = torch.tensor(x, device=cuda)
        y = torch.empty_like(tx)
        h.filter(tx, y)
        assert np.array_equal(y.cpu().numpy(), cone.filter_fwd(x, *shape, rmin))
        h.filter(tx, y, transpose=True)
        assert np.array_equal(y.cpu().numpy(), cone.filter_T(x, *shape, rmin))
