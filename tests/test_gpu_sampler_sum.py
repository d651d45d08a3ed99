"""The FP64 sampler's n = sum_j alpha_j beta_j: its sum's rounding against that of
32 interleaved chains joined in a tree, formed here from the same products."""
import math

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


@pytest.mark.parametrize("N", [17, 33, 64, 130, 200, 400])
def test_sum_of_the_warps(gbs, N):
    """With T = 1/2 an occupation is alpha_j beta_j / 4 (amplitudes below 1/32 of
    their scale, 2^-59 of it off, weigh nothing here).  4000 trajectories: the
    ratio of two root mean squares spreads by 1.6 %."""
    cnt = 4000
    r = np.linspace(0.6, 1.1, N)
    net = gbs.gbs_make_network(0.5 * np.eye(N), r, "fp64", 0)
    n, _ = gbs.gbs_debug_samples(net, 4242, 0, cnt)
    p = 4.0 * gbs.gbs_debug_occupations(net, 4242, 0, cnt).real
    gbs.gbs_free_network(net)
    chains = np.zeros((32, cnt))
    for j in range(N):
        chains[j % 32] += p[j]
    while chains.shape[0] > 1:
        chains = chains[::2] + chains[1::2]
    err = np.zeros((2, cnt))
    for i in range(cnt):
        size = math.fsum(np.abs(p[:, i]))
        for q, v in enumerate((n[i], chains[0, i])):
            err[q, i] = math.fsum([v, *(-p[:, i])]) / size
    rms = np.sqrt((err**2).mean(axis=1))
    assert rms[0] <= 1.05 * rms[1], rms
