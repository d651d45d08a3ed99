"""The MLP GEMMs at the edges of their tiles (128 batch rows, 64 and 128 weight
columns, splits of the batch) against the oracle, with the tolerances of
test_gpu_surrogate.py (BF16 hi + lo operands, FP32 accumulation)."""
import numpy as np
import pytest

import oracle.surrogate as sur
from test_gpu_surrogate import _init_params, _oracle_params, _pack, _unpack, gbs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_dim,width,out_dim,layers,batch", [
    (1, 256, 256, 2, 1),       # one row: 127 padding rows
    (32, 256, 512, 3, 127),
    (10, 512, 512, 4, 129),    # second row tile with one row
    (5, 768, 256, 3, 640),     # 6 column tiles of the weight gradients, uneven splits
    (10, 512, 512, 5, 1800),
])
def test_gradients_at_tile_edges(gbs, in_dim, width, out_dim, layers, batch):  # noqa: F811
    import torch
    dims = [in_dim] + [width] * (layers - 1) + [out_dim]
    params = _init_params(300 + batch, dims)
    mlp = gbs.gbs_mlp_create(in_dim, width, out_dim, layers, max(batch, 700))
    gbs.gbs_mlp_set_params(mlp, _pack(params))
    rng = np.random.default_rng(batch)
    X = rng.normal(size=(batch, in_dim)).astype(np.float32)
    T = rng.normal(size=(batch, out_dim)).astype(np.float32)
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    loss, grad = gbs.gbs_mlp_gradients(mlp, Xd.data_ptr(), Td.data_ptr(), batch)
    Yd = torch.zeros(batch, out_dim, dtype=torch.float32, device="cuda")
    gbs.gbs_mlp_forward(mlp, Xd.data_ptr(), batch, Yd.data_ptr())
    torch.cuda.synchronize()
    po = _oracle_params(params)
    Yo, cache = sur.forward(po, X.astype(np.float64))
    assert np.max(np.abs(Yd.cpu().numpy() - Yo)) < 1e-4 * np.max(np.abs(Yo))
    lo = sur.loss(Yo, T.astype(np.float64))
    assert abs(loss - lo) < 1e-5 * lo
    go = sur.backward(po, cache, Yo, T.astype(np.float64))
    gg = _unpack(grad.astype(np.float64), dims)
    for l in range(layers):
        for w in (0, 1):
            a, b = gg[l][w], go[l][w]
            assert np.linalg.norm(a - b) < 5e-4 * np.linalg.norm(b), (l, w)
            assert np.max(np.abs(a - b)) < 2e-3 * np.max(np.abs(b)), (l, w)
    # the training step's first loss is the same sum
    hist = gbs.gbs_mlp_train(mlp, Xd.data_ptr(), Td.data_ptr(), batch,
                             np.full(3, 1e-4, dtype=np.float32))
    assert abs(hist[0] - loss) <= 2.0**-23 * loss and np.all(np.isfinite(hist))
    gbs.gbs_mlp_free(mlp)
