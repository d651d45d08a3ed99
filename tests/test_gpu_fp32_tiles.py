"""The FP32 GEMM at the edges of its tiles (64 modes, 64 trajectories, 16 input
modes, 4-stage ring) against an emulation of its arithmetic: T and the samples
rounded to FP32 and N fused multiply-adds in FP32 in the order of the input
modes, each formed here as the exact FP64 product plus the accumulator, rounded
to FP32 (double rounding moves a result by at most one FP32 ulp of the
accumulator and is rare, hence half an ulp per step of slack on A_i = sum_j
|T_ij| |alpha_j| instead of bitwise equality: far below the N-ulp error of another
order or precision at these sizes)."""
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


def _chain(T, x):
    acc = np.zeros(T.shape[0], dtype=np.float32)
    for j in range(T.shape[1]):
        acc = (T[:, j].astype(np.float64) * float(x[j]) + acc.astype(np.float64)).astype(np.float32)
    return acc.astype(np.float64)


@pytest.mark.parametrize("N,M,count", [(1, 1, 1), (15, 63, 63), (16, 64, 64), (17, 65, 65),
                                       (64, 1, 129), (65, 130, 33), (80, 64, 64), (333, 70, 200)])
def test_tile_edges(gbs, N, M, count):
    d = wl.small_network(N, M=M, r=np.linspace(0.2, 1.3, N), t2=0.9, seed=N + 3, general_loss=True)
    net = gbs.gbs_make_network(d.T, d.r, "fp32", 0)
    occ = gbs.gbs_debug_occupations(net, 17, 9, count)
    n, nS = gbs.gbs_debug_samples(net, 17, 9, count)
    gbs.gbs_free_network(net)
    Tr, Ti = d.T.real.astype(np.float32), d.T.imag.astype(np.float32)
    for i in sorted({0, count // 2, count - 1}):
        al, be, _, _ = oracle.sample_amplitudes(d.T, d.r, 17, 9 + i)
        a, b = al.astype(np.float32), be.astype(np.float32)
        ar, ai, br, bi = _chain(Tr, a), _chain(Ti, a), _chain(Tr, b), _chain(Ti, b)
        want = (ar * br + ai * bi) + 1j * (ai * br - ar * bi)
        A, B = np.abs(d.T) @ np.abs(al), np.abs(d.T) @ np.abs(be)
        tol = 2.0 * 2.0**-24 * A * B  # an ulp of one accumulator on either side
        assert np.all(np.abs(occ[:, i] - want) <= tol), np.max(np.abs(occ[:, i] - want) / tol)
        assert abs(nS[i] - occ[:, i].sum()) <= (M + 4) * 2.0**-52 * np.abs(occ[:, i]).sum()
        assert abs(n[i] - float(al @ be)) <= (N + 8) * 2.0**-52 * float(np.abs(al) @ np.abs(be))
