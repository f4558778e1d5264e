"""The network's products at the edges of their tiles (32 outputs) and k slices (64): sizes of
one, one below, at and above, and batches and widths that leave remainders, against the
oracle's FP64 chain rule; a single layer with the output written over the input."""
import numpy as np
import pytest

from oracle import taps_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_13933_gb300 import build, taps
    import os
    if not os.path.exists(taps.LIB_PATH):
        build.build()
    taps.lib()
    return taps


@pytest.mark.parametrize("dims,B", [([1, 1, 1], 1), ([31, 33, 32], 63), ([64, 65, 65, 1], 64), ([2, 128, 128, 127], 65),
                                    ([129, 32], 129)])
def test_forward_and_gradients_at_tile_edges(T, dims, B):
    rng = np.random.default_rng(sum(dims) + B)
    n = sum(i * o + o for i, o in zip(dims[:-1], dims[1:]))
    p = rng.normal(0, 0.3, n).astype(np.float32)
    X = rng.normal(0, 1, (B, dims[0])).astype(np.float32)
    Y = rng.normal(0, 1, (B, dims[-1])).astype(np.float32)
    net = T.MLP(dims[0], dims[1] if len(dims) > 2 else 1, len(dims) - 2, dims[-1])
    net.set_params(p)
    xd, td = torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda")
    loss, g = net.grad(xd, td)
    lo, go = O.mlp_loss_grad(p.astype(float), dims, X.astype(float), Y.astype(float))
    # FP32 chains of up to 129 products through three layers: 129 * 3 * 2^-24 = 2.3e-5
    assert abs(loss - lo) <= 2.5e-5 * lo
    assert np.linalg.norm(g - go) <= 1e-4 * np.linalg.norm(go)
    y = torch.empty((B, dims[-1]), dtype=torch.float32, device="cuda")
    net.forward(xd, y)
    torch.cuda.synchronize()
    yo = O.mlp_forward(p.astype(float), dims, X.astype(float))[-1]
    assert np.max(np.abs(y.cpu().numpy() - yo)) <= 2.5e-5 * max(1.0, np.max(np.abs(yo)))


def test_single_layer_in_place(T):
    rng = np.random.default_rng(5)
    p = rng.normal(0, 0.3, 40 * 40 + 40).astype(np.float32)
    X = rng.normal(0, 1, (70, 40)).astype(np.float32)
    net = T.MLP(40, 1, 0, 40)
    net.set_params(p)
    x, y = torch.tensor(X, device="cuda"), torch.empty((70, 40), dtype=torch.float32, device="cuda")
    net.forward(x, y)
    net.forward(x, x)
    torch.cuda.synchronize()
    assert torch.equal(x, y)
