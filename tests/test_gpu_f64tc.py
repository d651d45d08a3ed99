"""The FP64 GEMM on the tensor cores (digit products) against the oracle at
the edges of its tiles, and the networks it leaves to the SIMT kernel.

Bound on alpha'_i (beta'_i alike), with S_i = sum_j |T_ij| c_j, c_j the
sampler's bound 8.67 hypot(q+_j, q-_j) on |alpha_j|: the operands are rounded
to 2^-56 of bounds that exceed max_j |T_ij| 2^{e_j} and c_j by less than 2
each, so with W_i = max_j |T_ij| c_j and 2^{e_j} <= 2 c_j the product of the
two scales is below 4 W_i 2 and each of the N terms errs by at most 2^-55 of
it (2^-61 more from the digit pairs left out): N 8 W_i 2^-55.  The oracle's
own FP64 sums and samples: (N + 32) 2^-53 S_i.
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


def _check(gbs, T, r, count, seed=91):
    M, N = T.shape
    net = gbs.gbs_make_network(T, r, "fp64", 0)
    occ = gbs.gbs_debug_occupations(net, seed, 5, count)
    n, nS = gbs.gbs_debug_samples(net, seed, 5, count)
    gbs.gbs_free_network(net)
    q = np.sqrt(0.5 * np.sinh(r) * np.exp(np.abs(r))), np.sqrt(0.5 * np.sinh(r) * np.exp(-r))
    c = 8.67 * np.hypot(*q)
    err = 0.0
    for A in (T.real, T.imag):
        W = np.max(np.abs(A) * c[None, :], axis=1)
        S = np.sum(np.abs(A) * c[None, :], axis=1)
        err = err + N * 8 * W * 2.0**-55 + (N + 32) * 2.0**-53 * S
    for i in sorted({0, count - 1, count // 2}):
        _, _, ap, bp = oracle.sample_amplitudes(T, r, seed, 5 + i)
        want = ap * bp
        tol = err * (np.abs(ap) + np.abs(bp)) + 2 * err * err + 2.0**-50 * np.abs(want)
        assert np.all(np.abs(occ[:, i] - want) <= tol), (i, np.max(np.abs(occ[:, i] - want) / tol))
        assert abs(nS[i] - want.sum()) <= tol.sum() + M * 2.0**-53 * np.abs(want).sum()


@pytest.mark.parametrize("N,M,count", [(15, 3, 5), (16, 1, 1), (17, 63, 15), (31, 64, 16),
                                       (64, 65, 17), (65, 129, 33), (127, 40, 31), (128, 64, 32),
                                       (129, 200, 40), (257, 577, 65), (300, 64, 5000)])
def test_tile_edges(gbs, N, M, count):
    d = wl.small_network(N, M=M, r=np.linspace(0.1, 1.6, N), t2=0.9, seed=N, general_loss=True)
    _check(gbs, d.T, d.r, count)


@pytest.mark.parametrize("kind", ["vacuum", "rows", "columns", "beyond"])
def test_uneven_scales(gbs, kind):
    """Vacuum inputs and zero rows; rows of very different size; columns that
    the squeezing scales back; a row beyond the digits' range (SIMT kernel)."""
    N, M = 48, 70
    d = wl.small_network(N, M=M, r=np.linspace(0.2, 1.2, N), t2=0.9, seed=4)
    T, r = d.T.copy(), d.r.copy()
    if kind == "vacuum":
        r[::5] = 0.0
        T[7] = 0.0
    elif kind == "rows":
        T *= 10.0 ** np.linspace(-12, 3, M)[:, None]
    elif kind == "columns":
        r = np.linspace(1e-6, 6.0, N)
    else:
        T[3] *= 1e-140
    _check(gbs, T, r, 40)
