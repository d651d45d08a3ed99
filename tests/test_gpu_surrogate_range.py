"""Surrogate features of extreme squeezing."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_12749_gb300 as g
    g.build()
    return g


def test_fourth_powers_beyond_the_range(gbs):
    """eta^2 sinh^4 r is finite where sinh^4 r is not (r = 180, eta = 0.0025).
    Every part is a product of correctly rounded or few-ulp functions: 1e-13."""
    import torch
    r, t = 180.0, 0.05
    feat = torch.zeros(1, gbs.GBS_SUR_RECORD, dtype=torch.float64, device="cuda")
    gbs.gbs_surrogate_features([1], [1], [t], [4096], [0], [np.array([r])], feat.data_ptr())
    f = feat.cpu().numpy()[0]
    x, eta = np.longdouble(r), np.longdouble(t) ** 2
    sh2 = np.sinh(x) ** 2
    s = np.sqrt(eta * sh2 + eta * eta * sh2 * np.cosh(2 * x))
    assert abs(f[11] - float(s)) <= 1e-13 * float(s)
    assert abs(f[9] - float(np.log(s))) <= 1e-13 * float(np.log(s))
