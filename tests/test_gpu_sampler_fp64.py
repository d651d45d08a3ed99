"""The FP64 sampler (digit tiles, FP32 tiles, plain rows) against the oracle's
n = sum_j alpha_j beta_j at the edges of its work split: modes around 8 (a
lane's group), 16 (a K block), 32 (a warp's pass) and every number of warps per
group of trajectories; trajectories around 8, 32 and a block's turn.

Bound: both sides' normals err by at most 4 2^-53 of the radius rho (log, sqrt,
sine and cosine to an ulp each, one product), so with Q = |q+| + |q-| each of
alpha, beta errs by (8 + 4) 2^-53 Q rho between the sides, their product by
24 2^-53 Q^2 rho^2 + 2^-53 |alpha beta|, and the sums of N terms by N 2^-53 each of
sum |alpha beta| <= sum Q^2 rho^2: (25 + 2 N) 2^-53 sum_j Q_j^2 rho_j^2.
"""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,count", [(1, 70), (7, 33), (15, 9), (16, 1), (17, 65), (32, 63), (33, 129),
                                     (64, 31), (65, 17), (129, 40), (200, 8)])
def test_n_matches_oracle(gbs, precision, N, count):
    e0, seed = 2**32 - 3, 2503 + N  # the trajectory index crosses 32 bits
    d = wl.small_network(N, r=np.linspace(0.1, 1.6, N), t2=0.9, seed=N)
    net = gbs.gbs_make_network(d.T, d.r, precision, 0)
    n, _ = gbs.gbs_debug_samples(net, seed, e0, count)
    gbs.gbs_free_network(net)
    Q = np.sqrt(0.5 * np.sinh(d.r)) * (np.exp(0.5 * d.r) + np.exp(-0.5 * d.r))
    for i in range(count):
        a, b = oracle.sample_inputs(d.r, seed, e0 + i)[:2]
        w = np.array([oracle.normals(seed, e0 + i, j) for j in range(N)])
        tol = (25 + 2 * N) * 2.0**-53 * np.sum(Q**2 * np.sum(w**2, axis=1))
        assert abs(n[i] - np.sum(a * b)) <= tol, (i, n[i] - np.sum(a * b), tol)
