"""The pipelines of the FP32 GEMM, the FP64 GEMM on the tensor cores and the joint
generating functions' contraction when they give up waiting.

As in test_gpu_failures.py nothing faults: a wait limit of 0 makes the kernel
first wait on a barrier that nothing arrives on.  It gives up, raises the
network's flag, takes no stage, lets the loads it issued land and returns.
"""
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


@pytest.fixture(scope="module")
def stream():
    import torch
    return torch.cuda.Stream().cuda_stream


def _sums(gbs, net, seed, E, n_sub, K1):
    gbs.gbs_sample(net, seed, 0, E, n_sub, K1)
    P = gbs.gbs_binned_counts(net, 0, K1)
    _, _, acc, _ = gbs.gbs_get_accumulators(net)
    return [acc.view(np.float64), *P]


# fewer K blocks than the ring has stages, and several turns of it
@pytest.mark.parametrize("precision,N", [("fp32", 40), ("fp32", 200), ("fp64", 16), ("fp64", 300)])
def test_gemm_wait_timeout(gbs, stream, precision, N):
    d = wl.small_network(N, M=160, r=0.7, t2=0.9, seed=41)
    E, n_sub, K1 = 6000, 8, 512
    ref = gbs.gbs_make_network(d.T, d.r, precision, stream)
    want = _sums(gbs, ref, d.seed_s, E, n_sub, K1)
    gbs.gbs_free_network(ref)

    net = gbs.gbs_make_network(d.T, d.r, precision, stream)
    gbs.gbs_set_wait_limit(net, 0)
    gbs.gbs_sample(net, d.seed_s, 0, E, n_sub, K1)
    with pytest.raises(gbs.GbsError) as ei:
        gbs.gbs_binned_counts(net, 0, K1)
    assert ei.value.code == gbs.GBS_ETIMEOUT
    gbs.gbs_set_wait_limit(net, 2_000_000_000)
    gbs.gbs_reset(net)
    got = _sums(gbs, net, d.seed_s, E, n_sub, K1)
    gbs.gbs_free_network(net)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16x3"])
def test_joint_contraction_wait_timeout(gbs, stream, precision):
    """The digit contraction of the joint generating functions (750 trajectories
    per sub-ensemble on 64 x 64 points)."""
    d = wl.small_network(40, M=70, r=0.5, t2=0.9, seed=43)
    bins = (np.arange(70) >= 30).astype(np.int32)
    E, n_sub, K = 6000, 8, [64, 64]
    net = gbs.gbs_make_network_binned(d.T, d.r, bins, precision, stream)
    gbs.gbs_sample_nd(net, d.seed_s, 0, E, n_sub, K)
    want = gbs.gbs_binned_counts_nd(net, K)
    gbs.gbs_reset(net)
    gbs.gbs_set_wait_limit(net, 0)
    gbs.gbs_sample_nd(net, d.seed_s, 0, E, n_sub, K)
    with pytest.raises(gbs.GbsError) as ei:
        gbs.gbs_binned_counts_nd(net, K)
    assert ei.value.code == gbs.GBS_ETIMEOUT
    gbs.gbs_set_wait_limit(net, 2_000_000_000)
    gbs.gbs_reset(net)
    gbs.gbs_sample_nd(net, d.seed_s, 0, E, n_sub, K)
    got = gbs.gbs_binned_counts_nd(net, K)
    gbs.gbs_free_network(net)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
