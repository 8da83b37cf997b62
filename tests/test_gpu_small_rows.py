"""The stem's im2col rows, the mean over time and the flow's targets at the edges of their blocks (needs a GPU):
copies and sums in a fixed order, compared bit for bit; targets (FP64, rounded once) to one FP32 rounding."""
import numpy as np
import pytest

import workloads

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


# one time, one short of, exactly and one past the 32 times in flight; odd channel counts take the scalar kernel
@pytest.mark.parametrize("B,T,C", [(1, 1, 2), (3, 31, 8), (2, 32, 7), (5, 33, 130), (2, 257, 64)])
def test_mean_over_time(gwx, B, T, C):
    from paper_2407_19048_gb300 import _lib
    x = torch.randn((B, T, C), generator=torch.Generator().manual_seed(T)).bfloat16()
    want = torch.zeros((B, C))
    for t in range(T):
        want += x[:, t].float()
    want = (want / T).bfloat16()
    xd, m = x.cuda(), torch.empty((B, C), dtype=torch.bfloat16, device="cuda")
    gwx._check(_lib.load().gwx_mean_time(gwx._ptr(xd), B, T, C, gwx._ptr(m), gwx._stream()))
    assert torch.equal(m.cpu(), want)


# taps that fill the padded row, leave a part of it or of its 8-column pieces; a row that is no multiple of 8
@pytest.mark.parametrize("D,k,s,K,N", [(2, 7, 2, 16, 100), (3, 7, 2, 24, 65), (1, 3, 1, 8, 9), (2, 4, 2, 8, 64),
                                       (2, 3, 1, 6, 31)])
def test_stem_rows(gwx, D, k, s, K, N):
    from paper_2407_19048_gb300 import _lib
    B, p = 3, (k - 1) // 2
    y = torch.randn((B, D, N), generator=torch.Generator().manual_seed(N))
    To = (N + 2 * p - k) // s + 1
    want = torch.zeros((B, To, K))
    yp = torch.nn.functional.pad(y, (p, p + k))
    for j in range(k):
        want[:, :, j * D:(j + 1) * D] = yp[:, :, j:j + s * To:s][:, :, :To].transpose(1, 2)
    yd, cols = y.cuda(), torch.empty((B, To, K), dtype=torch.bfloat16, device="cuda")
    gwx._check(_lib.load().gwx_im2col_cf(gwx._ptr(yd), B, D, N, k, s, p, K, gwx._ptr(cols), gwx._stream()))
    assert torch.equal(cols.cpu(), want.bfloat16())


@pytest.mark.parametrize("B", [1, 31, 32, 33, 100])
def test_flow_targets(gwx, B):
    theta = workloads.random_theta(B, B, workloads.workload("small")["prior"])
    m1, m2 = theta[0], theta[1]
    r = np.stack([(m1 * m2) ** 0.6 / (m1 + m2) ** 0.2, np.minimum(m1, m2) / np.maximum(m1, m2), theta[4],
                  np.cos(theta[7]), theta[9], np.sin(theta[10]), theta[8], theta[6]], axis=1)
    mean, scale = np.arange(8) * 0.3, 1.0 + np.arange(8) * 0.5
    got = gwx.flow_targets(torch.from_numpy(theta).cuda(), list(mean), list(scale)).cpu().numpy()
    want = (r - mean) / scale
    assert np.all(np.abs(got - want) <= 2.0 ** -23 * np.abs(want) + 1e-12 * (np.abs(r) + 1))
