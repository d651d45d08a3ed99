"""The MLP's long sums."""
import numpy as np
import pytest

from test_gpu_surrogate import _init_params, _oracle_params, _pack, _unpack, gbs  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,batch", [(512, 16384), (1024, 32768)])
def test_weight_gradient_of_a_large_batch(gbs, width, batch):  # noqa: F811
    """Targets far below the outputs make every row's term of dW = dY^T H for the
    last layer nearly alike in sign, so that a tensor core's truncation of its
    FP32 accumulator (below 2^-23 of it at every product of 16 rows) adds up: by
    at most n / 2 2^-23 over n products into one accumulator, as the sum grows
    evenly.  The batch is summed in at least eight parts, of three products
    (hi hi, hi lo, lo hi) per 16 rows each.  The rest (operands of 16 bits and
    more, the forward pass's own chains of 2 width / 16 products) is below 1e-5."""
    import torch
    dims = [10, width, width, width, 256]
    params = _init_params(7 + width, dims)
    mlp = gbs.gbs_mlp_create(10, width, 256, 4, batch)
    gbs.gbs_mlp_set_params(mlp, _pack(params))
    rng = np.random.default_rng(batch)
    X = torch.from_numpy(rng.normal(size=(batch, 10)).astype(np.float32)).cuda()
    T = torch.full((batch, 256), -1000.0, dtype=torch.float32, device="cuda")
    _, grad = gbs.gbs_mlp_gradients(mlp, X.data_ptr(), T.data_ptr(), batch)
    gbs.gbs_mlp_free(mlp)
    h = X.double()
    po = [(torch.from_numpy(np.asarray(W)).cuda().double(), torch.from_numpy(np.asarray(b)).cuda().double())
          for W, b in _oracle_params(params)]
    for W, b in po[:-1]:
        z = h @ W.T + b
        h = z * torch.sigmoid(z)
    y = h @ po[-1][0].T + po[-1][1]
    want = (2.0 * (y - T.double()) / (batch * 256)).T @ h
    got = torch.from_numpy(_unpack(grad.astype(np.float64), dims)[-1][0]).cuda()
    n = 3 * (batch // 8 // 16)
    loss = ((want - got) / want).median().item()
    assert abs(loss) <= n / 2 * 2.0**-23 + 1e-5, loss

def test_loss_of_equal_errors(gbs):  # noqa: F811
    """With zero weights and equal targets every squared error is the same FP32
    number c.  Sums of 2, 4, .. 32 of them are exact in FP32, and so is the mean."""
    import torch
    dims = [10, 512, 512, 512]
    params = [(np.zeros((dims[i + 1], dims[i])), np.zeros(dims[i + 1])) for i in range(3)]
    mlp = gbs.gbs_mlp_create(10, 512, 512, 3, 1024)
    gbs.gbs_mlp_set_params(mlp, np.concatenate([np.concatenate([W.ravel(), b]) for W, b in params]).astype(np.float32))
    X = torch.randn(640, 10, device="cuda")
    t = np.float32(1.2345678)
    T = torch.full((640, 512), float(t), device="cuda")
    loss, _ = gbs.gbs_mlp_gradients(mlp, X.data_ptr(), T.data_ptr(), 640)
    gbs.gbs_mlp_free(mlp)
    c = float(np.float32(t * t))
    assert abs(loss - c) <= 2.0**-50 * c
