"""The joint generating functions as digit contractions against the
outer-product kernel on the same trajectories: the same trajectories in few
sub-ensembles (contractions) and in many of 13 (FP64: 3) trajectories each
(outer products, FP64: a thread per grid point) have the same mean P.  Grids with ragged windows, three and
four bins, trajectories that need the (rA - 1) term, and ones left to the
outer-product kernel (few modes: exponents above the contractions' range).

Bound: with n_b = |n_Sb| and M = sum_b max(0, max_theta Re (z_b - 1) n_Sb) of a
trajectory, both sides evaluate factors of at most e^M whose exponents and
phases, up to 2 sum_b n_b, carry 2^-45 relative, whose double-float functions err by
2^-44, and sum them with 2^-44; resolution of the digits 2^-47 of e^5.5 at
most.  P is the mean over the grid of sums of such terms (two for matrix-P) times
phases, so |dP| <= mean_e 2 e^M (4 sum_b n_b + 8) 2^-44 + 2^-39, both sides.  FP64
networks: exponents, phases and functions carry 2^-52, resolutions 2^-55 of factors
below 2, sums of at most 3 terms on the other side: 2^-49 and 2^-50.
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


def _bound(d, bins, e0, E, eps):
    B = max(bins) + 1
    th = 2 * np.pi * np.arange(256) / 256
    z1 = np.exp(1j * th) - 1
    out = 0.0
    for e in range(E):
        _, _, a, b = oracle.sample_amplitudes(d.T, d.r, d.seed_s, e0 + e)
        nS = np.array([np.sum((a * b)[np.asarray(bins) == q]) for q in range(B)])
        M = np.max((z1[None, :] * nS[:, None]).real, axis=1).clip(0).sum()
        # e^{-L + c2}: the matrix-P partner term, at most e^{M'} with the same shape
        n = nS.real.sum()
        Mp = np.max((-z1[None, :] * nS[:, None]).real, axis=1).clip(0).sum() - 2 * max(n, 0)
        out += 2 * np.exp(max(M, Mp, 0)) * (4 * np.abs(nS).sum() + 8) * eps
    return out / E


@pytest.mark.parametrize("precision", ["bf16x3", "fp64"])
@pytest.mark.parametrize("N,M,r,t2,bins,K,ns", [
    (40, 40, 0.5, 1.0, 2, (128, 128), (9, 99)),   # lossless: B terms everywhere
    (40, 37, 0.6, 0.9, 2, (64, 256), (9, 99)),
    (4, 4, 0.6, 0.95, 2, (64, 64), (9, 99)),      # wide factors, rA != 1
    (8, 12, 0.4, 1.0, 2, (256, 64), (1, 99)),     # one sub-ensemble
    (12, 12, 0.5, 0.95, 3, (8, 8, 64), (3, 99)),
    (10, 10, 0.5, 1.0, 4, (4, 4, 4, 64), (11, 99)),
    (10, 14, 0.5, 0.9, 3, (8, 16, 32), (9, 99)),  # half a tile of columns
    (100, 100, 0.8, 0.8, 2, (64, 64), (13, 99)),  # windows smaller than the circles
])
def test_matches_general_kernels(gbs, precision, N, M, r, t2, bins, K, ns):
    E, e0, fp64 = 1287, 5, precision == "fp64"
    ns = (ns[0], 429 if fp64 else ns[1])
    d = wl.small_network(N, M=M, r=r, t2=t2, seed=300 + N)
    b = (np.arange(M) * bins // M).astype(np.int32)
    P = []
    for n_sub in ns:
        net = gbs.gbs_make_network_binned(d.T, d.r, b, precision, 0)
        gbs.gbs_sample_nd(net, d.seed_s, e0, E, n_sub, K)
        P.append(gbs.gbs_binned_counts_nd(net, K))
        gbs.gbs_free_network(net)
    tol = _bound(d, b, e0, E, 2.0**-49 if fp64 else 2.0**-44) + 2.0**(-50 if fp64 else -39)
    for est in (0, 2):
        assert np.all(np.isfinite(P[0][est])) and np.any(P[0][est] != 0)
        assert np.max(np.abs(P[0][est] - P[1][est])) <= tol, (est, np.max(np.abs(P[0][est] - P[1][est])), tol)
