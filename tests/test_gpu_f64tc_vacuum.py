"""An output mode that is coupled to vacuum inputs alone, however weakly, is
zero and leaves the other modes' path as it is."""
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


@pytest.mark.parametrize("entry", [0.3, 1e-200, 1e200])
def test_rows_of_vacuum_inputs(gbs, entry):
    """Against the same network with that row zero: bitwise, since a row's
    digits depend on nothing outside it (the FP64 FMA kernel, taken for
    networks outside the digits' range, rounds differently)."""
    N, M = 48, 70
    d = wl.small_network(N, M=M, r=np.linspace(0.2, 1.2, N), t2=0.9, seed=4)
    r = d.r.copy()
    r[::3] = 0.0
    occ = []
    for v in (0.0, entry):
        T = d.T.copy()
        T[7] = 0.0
        T[7, ::3] = v * (1 - 0.5j)
        net = gbs.gbs_make_network(T, r, "fp64", 0)
        occ.append(gbs.gbs_debug_occupations(net, 91, 5, 300))
        gbs.gbs_free_network(net)
    assert np.all(occ[1][7] == 0.0)
    assert np.array_equal(occ[0], occ[1])
