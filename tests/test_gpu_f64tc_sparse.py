"""FP64 networks whose rows of T have few entries, where the digits of the
samples are the only rounding of the propagation."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_12749_gb300 as g
    g.build()
    return g


@pytest.mark.parametrize("N", [16, 40, 200])
def test_amplitudes_keep_their_bits(gbs, N):
    """One squeezed input (r = 1) and T = 1 / 2: n is alpha beta rounded once,
    the occupation alpha beta / 4 rounded once if alpha and beta pass the digits
    exactly, so four times it is n to the bit.  The samples' standard deviation
    is 1.347, their scale 2^4 (8.67 times that, rounded up to a power of two) and
    their digits 58 bits of it: amplitudes above 1/4 are exact, 85 % of each, and
    so are both in more than 70 % of the trajectories (binomial spread of 4000:
    0.7 %)."""
    r = np.zeros(N)
    j = N // 3
    r[j] = 1.0
    net = gbs.gbs_make_network(0.5 * np.eye(N), r, "fp64", 0)
    n, _ = gbs.gbs_debug_samples(net, 31, 0, 4000)
    occ = gbs.gbs_debug_occupations(net, 31, 0, 4000)
    gbs.gbs_free_network(net)
    assert np.mean(4.0 * occ[j].real == n) >= 0.68
    assert np.all(np.delete(occ, j, axis=0) == 0.0)
