"""Every entry point that returns sampled data reports a kernel that gave up
waiting (GBS_ETIMEOUT) and clears the flag; the wait limit of 0 makes the GEMM
give up without a fault (test_gpu_failures.py)."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

N, M, E, N_SUB, K1 = 40, 70, 500, 4, 64


@pytest.fixture(scope="module")
def gbs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_12749_gb300 as g
    g.build()
    return g


def _read(gbs, net, what, seed):
    if what == "histogram":
        return gbs.gbs_histogram(net, seed, 0, E, [0, 2], -1.0, 1.0, 16)
    if what == "samples":
        return np.concatenate(gbs.gbs_debug_samples(net, seed, 0, E)).view(np.float64)
    if what == "occupations":
        return gbs.gbs_debug_occupations(net, seed, 0, E).view(np.float64)
    if what == "windows":
        return gbs.gbs_debug_windows(net, seed, 0, E)
    gbs.gbs_reset(net)
    gbs.gbs_sample(net, seed, 0, E, N_SUB, K1)
    return gbs.gbs_get_accumulators(net)[2].view(np.float64)


@pytest.mark.parametrize("what", ["histogram", "samples", "occupations", "windows", "accumulators"])
@pytest.mark.parametrize("precision", ["bf16x3", "fp64", "fp32"])
def test_timeout_is_reported(gbs, precision, what):
    d = wl.small_network(N, M=M, r=0.7, t2=0.9, seed=47)
    net = gbs.gbs_make_network(d.T, d.r, precision, 0)
    gbs.gbs_sample(net, d.seed_s, 0, E, N_SUB, K1)  # windows are those of its K1
    want = _read(gbs, net, what, d.seed_s)
    gbs.gbs_set_wait_limit(net, 0)
    with pytest.raises(gbs.GbsError) as ei:
        _read(gbs, net, what, d.seed_s)
    assert ei.value.code == gbs.GBS_ETIMEOUT
    gbs.gbs_set_wait_limit(net, 2_000_000_000)
    assert np.array_equal(_read(gbs, net, what, d.seed_s), want)  # the flag was cleared
    gbs.gbs_free_network(net)
