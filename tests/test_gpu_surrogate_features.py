"""Surrogate features whose first squeezing parameter lies far from the others
(the sums run about it), at the edges of the 512-parameter blocks, against
numpy in extended precision.

Bound: a two-pass variance in FP64 errs by less than (N / 64 + 64)
2^-53 of itself where its sums are formed in trees of 64 or more (blocks of 512,
then at most 4 blocks here), and sinh, cosh and the root add a few ulp: 1e-13.
"""
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


@pytest.mark.parametrize("N", [1, 2, 255, 257, 511, 512, 513, 1025, 2000])
def test_outlying_first_parameter(gbs, N):
    import torch
    r = np.random.default_rng(N).uniform(0.5, 0.5001, size=N)
    r[0] = 1.5
    feat = torch.zeros(1, gbs.GBS_SUR_RECORD, dtype=torch.float64, device="cuda")
    gbs.gbs_surrogate_features([N], [N], [0.95], [4096], [0], [r], feat.data_ptr())
    f = feat.cpu().numpy()[0]
    x = r.astype(np.longdouble)
    mean = x.mean()
    sd = np.sqrt(((x - mean) ** 2).mean())
    assert abs(f[2] - float(mean)) <= 1e-13 * abs(float(mean))
    assert abs(f[3] - float(sd)) <= 1e-13 * float(sd)
    assert f[4] == r.min() and f[5] == r.max()
    sh2 = np.sinh(x) ** 2
    eta = np.longdouble(0.95) ** 2
    mu, var = eta * sh2.sum(), (eta * sh2 + eta**2 * sh2 * np.cosh(2 * x)).sum()
    assert abs(f[10] - float(mu)) <= 1e-13 * float(mu)
    assert abs(f[11] - float(np.sqrt(var))) <= 1e-13 * float(np.sqrt(var))
