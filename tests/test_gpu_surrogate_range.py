"""Surrogate features of extreme squeezing, and of parameters at any address."""
import ctypes

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


@pytest.mark.parametrize("shift", [0, 1, 4, 8])
def test_parameters_at_any_address(gbs, shift):
    """The C entry takes squeezing parameters that are not aligned."""
    import torch
    N = 600
    r = np.random.default_rng(2).uniform(0.4, 1.2, size=N)
    raw = np.zeros(8 * N + 16, dtype=np.uint8)
    start = -raw.ctypes.data % 8 + shift
    raw[start:start + 8 * N] = r.view(np.uint8)
    feat = torch.zeros(2, gbs.GBS_SUR_RECORD, dtype=torch.float64, device="cuda")
    gbs.gbs_surrogate_features([N], [N], [0.9], [4096], [0], [r], feat[0].data_ptr())
    i32, i64, f64 = ctypes.c_int * 1, ctypes.c_int64 * 1, ctypes.c_double * 1
    code = gbs.lib().gbs_surrogate_features(
        1, i32(N), i32(N), f64(0.9), i32(4096), i64(0),
        ctypes.cast(raw.ctypes.data + start, ctypes.POINTER(ctypes.c_double)),
        (ctypes.c_int64 * 2)(0, N), None, ctypes.c_void_p(feat[1].data_ptr()))
    assert code == gbs.GBS_OK
    assert torch.equal(feat[0], feat[1])
