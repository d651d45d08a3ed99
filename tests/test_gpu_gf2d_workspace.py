"""The joint generating functions' work space belongs to the call: a captured
gbs_sample_nd allocates and releases it inside its graph, and eager calls
before and after it find their own."""
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


@pytest.mark.parametrize("precision", ["fp64", "bf16x3"])
def test_capture_after_a_smaller_call(gbs, precision):
    """A first call too small for the contraction, a captured one that takes it,
    an eager one of another size: bitwise the three calls made eagerly."""
    import torch
    d = wl.small_network(40, M=70, r=0.5, t2=0.9, seed=53)
    bins = (np.arange(70) >= 30).astype(np.int32)
    n_sub, K, parts = 16, [64, 64], [64, 4096, 9000]
    stream = torch.cuda.Stream()

    def network():
        net = gbs.gbs_make_network_binned(d.T, d.r, bins, precision, stream.cuda_stream)
        if precision == "bf16x3":
            gbs.gbs_set_gemm_config(net, 1, 0, 0)
        return net

    def call(net, i):
        gbs.gbs_sample_nd(net, d.seed_s, sum(parts[:i]), parts[i], n_sub, K)

    ref = network()
    for i in range(3):
        call(ref, i)
    want = gbs.gbs_binned_counts_nd(ref, K)
    gbs.gbs_free_network(ref)

    net = network()
    call(net, 0)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call(net, 1)
    with torch.cuda.stream(stream):
        graph.replay()
    call(net, 2)
    got = gbs.gbs_binned_counts_nd(net, K)
    del graph
    gbs.gbs_free_network(net)
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
