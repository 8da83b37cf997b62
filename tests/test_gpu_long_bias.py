"""Bias gradients of batches whose partial column sums come in more than one slice (more than 8192 rows), on small
integers: every partial sum is an integer below 2^24, so the results equal FP64's bit for bit (needs a GPU)."""
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


# two slices with a ragged last one; as many slices as there are, with a ragged last partial
@pytest.mark.parametrize("M,N", [(8200, 40), (64 * 256 * 32 + 8, 8)])
@pytest.mark.parametrize("act", ["none", "relu"])
def test_bias_gradients_of_long_batches(gwx, M, N, act):
    rng = np.random.default_rng(M)
    K = 8
    X, W, dY = (torch.from_numpy(rng.integers(-2, 3, s).astype(np.float64)) for s in ((M, K), (N, K), (M, N)))
    b = 0.5 + torch.arange(N, dtype=torch.float64) % 3
    dz = dY * ((X @ W.T + b) > 0) if act == "relu" else dY
    _, dW, db = gwx.dense_bf16_backward(X.bfloat16().cuda(), W.bfloat16().cuda(), b.float().cuda(), dY.float().cuda(),
                                        gwx.ACT_RELU if act == "relu" else gwx.ACT_NONE)
    assert torch.equal(db.double().cpu(), dz.sum(0))
    assert torch.equal(dW.double().cpu(), dz.T @ X)
