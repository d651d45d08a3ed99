"""The FP64 generating-function kernel against the oracle's sums on the same
(n, n_S): every split of a sub-ensemble over half-warps and cluster blocks
(1, 2, 4, 8), ragged ends, mirror pairs (n_S real) and general n_S, windows
that cover the circle and that do not.

Bound per term e^{L}: the phase and exponent are products of |n_S| with factors
of at most 2 in FP64 on both sides, each rounded at most three times, and the
exponential, sine and cosine add a few ulp: (8 |n_S| + 32) 2^-52 of the term,
and 2^-60 where it is skipped.  Terms have |e^{L}| at most max(1, the oracle's
sum of |terms|), taken here as the largest |G| of the trajectory, and the
summation adds cnt 2^-52 of the sum of the terms.
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


@pytest.mark.parametrize("N,M,r,general,E,n_sub,K1,e0", [
    (6, 6, 0.5, False, 300, 300, 8, 0),      # one trajectory each
    (16, 16, 1.0, False, 2048, 16, 64, 0),   # 16 per half-warp and block
    (16, 16, 1.0, False, 5003, 2, 64, 3),    # 8 blocks a cluster, ragged
    (12, 9, 0.8, True, 5003, 3, 128, 1),
    (40, 40, 0.9, False, 1100, 4, 512, 7),   # window smaller than the circle
    (40, 33, 0.9, True, 700, 2, 512, 7),
    (5, 5, 0.3, False, 40, 1, 2, 0),         # the two self-paired points
    (20, 20, 0.7, True, 9, 4, 32, 2),        # fewer trajectories than half-warps
])
def test_sums_match_oracle(gbs, N, M, r, general, E, n_sub, K1, e0):
    d = wl.small_network(N, M=M, r=r, t2=0.9, seed=N + K1, general_loss=general)
    for precision in ("fp64", "fp32"):
        net = gbs.gbs_make_network(d.T, d.r, precision, 0)
        gbs.gbs_sample(net, d.seed_s, e0, E, n_sub, K1)
        _, _, acc, cnt = gbs.gbs_get_accumulators(net)
        n, nS = gbs.gbs_debug_samples(net, d.seed_s, e0, E)
        gbs.gbs_free_network(net)
        want, wcnt = oracle.accumulate_gf(n, nS, e0, n_sub, K1)
        assert np.array_equal(cnt, wcnt)
        th = 2 * np.pi * np.arange(K1) / K1
        L = (np.cos(th) - 1)[None, :] * nS.real[:, None] - np.sin(th)[None, :] * nS.imag[:, None]
        plus = np.exp(L)
        mat = (np.exp(L + np.minimum(0, 2 * n)[:, None])
               + np.exp(-L - 2 * np.maximum(n, 0)[:, None])) / (1 + np.exp(-2 * np.abs(n)))[:, None]
        for est, size in ((0, mat), (1, plus)):
            for q in range(n_sub):
                e = np.arange(E)[(np.arange(E) + e0) % n_sub == q]
                tol = np.sum(size[e] * ((8 * np.abs(nS[e]) + 32 + len(e)) * 2.0**-52)[:, None], axis=0)
                tol += len(e) * 2.0**-59
                err = np.abs(acc[est, q] - want[est, q])
                assert np.all(err <= tol), (precision, est, q, np.max(err / tol))
