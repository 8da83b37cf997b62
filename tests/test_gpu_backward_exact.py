"""The products of the dense and convolution backward passes at the edges of their tiles, on small
integers: every product and sum is exact in FP32, so the results equal FP64's bit for bit (needs a GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gwx():
    import paper_2407_19048_gb300 as m
    from paper_2407_19048_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    m.init()
    return m


def _ints(rng, *shape):
    return torch.from_numpy(rng.integers(-2, 3, shape).astype(np.float64))


# smallest sizes, one past and one short of a tile (128 rows, 64 / 128 / 256 columns), a batch that is split
# with a ragged last slice, an output of few columns, an output of many tiles
@pytest.mark.parametrize("M,N,K", [(8, 8, 8), (136, 72, 200), (128, 64, 64), (120, 136, 264), (2056, 8, 256),
                                   (4104, 256, 72), (520, 1032, 1096)])
@pytest.mark.parametrize("act", ["none", "relu"])
def test_dense_backward(gwx, M, N, K, act):
    rng = np.random.default_rng(M + N + K)
    X, W, dY = _ints(rng, M, K), _ints(rng, N, K), _ints(rng, M, N)
    b = _ints(rng, N) + 0.5
    dz = dY * ((X @ W.T + b) > 0) if act == "relu" else dY
    dX, dW, db = gwx.dense_bf16_backward(X.bfloat16().cuda(), W.bfloat16().cuda(), b.float().cuda(), dY.float().cuda(),
                                         gwx.ACT_RELU if act == "relu" else gwx.ACT_NONE)
    assert torch.equal(dX.double().cpu(), dz @ W)
    assert torch.equal(dW.double().cpu(), dz.T @ X)
    assert torch.equal(db.double().cpu(), dz.sum(0))


@pytest.mark.parametrize("B,T,C,O,k", [(1, 128, 64, 64, 1), (3, 256, 64, 128, 5), (2, 128, 192, 64, 3),
                                       (9, 384, 128, 320, 5)])
def test_conv_backward(gwx, B, T, C, O, k):
    rng = np.random.default_rng(B * T + C + O + k)
    x, W, dz = _ints(rng, B, T, C), _ints(rng, O, k, C), _ints(rng, B, T, O)
    p = (k - 1) // 2
    xp = torch.nn.functional.pad(x, (0, 0, p, p))
    zp = torch.nn.functional.pad(dz, (0, 0, p, p))
    dW = torch.stack([torch.einsum("bto,btc->oc", dz, xp[:, j:j + T]) for j in range(k)], 1)
    dx = sum(zp[:, k - 1 - j:k - 1 - j + T] @ W[:, j] for j in range(k))
    got_dx, got_dW = gwx.conv1d_bf16_backward(dz.float().cuda(), x.bfloat16().cuda(),
                                              W.reshape(O, k * C).bfloat16().cuda(), k)
    assert torch.equal(got_dx.double().cpu(), dx)
    assert torch.equal(got_dW.double().cpu(), dW.reshape(O, k * C))
