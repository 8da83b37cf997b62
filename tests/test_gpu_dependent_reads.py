"""Chains of kernels launched under the end of their predecessors whose reads follow the producer directly (needs a
GPU): group norm, the convolution's rows of its output and their product; the masked rows of a dense layer, the column
sums of more than one slice and the kernel that finishes them; rows folded back onto an addend.  The bits of the
same calls with a synchronisation after each."""
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


def _chain(gwx, z0, W, steps, sync):
    """Norm, rows, product, gradient of the product, rows folded back onto the input: the result is the next input."""
    from paper_2407_19048_gb300 import _lib
    lib, st, p = _lib.load(), gwx._stream(), gwx._ptr
    B, T, C = z0.shape
    one, zero = torch.ones(C, device="cuda"), torch.zeros(C, device="cuda")
    z, keep = z0.clone(), []
    x = torch.empty((B, T, C), dtype=torch.bfloat16, device="cuda")
    ms, cols = torch.empty((B, 8, 2), device="cuda"), torch.empty((B * T, 5 * C), dtype=torch.bfloat16, device="cuda")
    dx = torch.empty_like(z)
    for _ in range(steps):
        gwx._check(lib.gwx_group_norm(p(z), B, T, C, 8, p(one), p(zero), None, None, 1, p(x), None, p(ms), st))
        sync()
        gwx._check(lib.gwx_im2col(p(x), B, T, C, 5, 1, 2, 5 * C, p(cols), st))
        sync()
        y = gwx.dense_bf16(cols, W, None, gwx.ACT_NONE)
        sync()
        dcols, dW, db = gwx.dense_bf16_backward(cols, W, zero, y, gwx.ACT_RELU)
        sync()
        gwx._check(lib.gwx_col2im(p(dcols), B, T, C, 5, 1, 2, 5 * C, p(z), p(dx), st))
        sync()
        z, dx = dx, z
        keep += [dW, db]
    return keep + [z, x]


@pytest.mark.parametrize("B,T,C", [(33, 256, 64), (4, 130, 32)])   # 264 partials of 32 rows are two slices; one
def test_chain_keeps_its_bits(gwx, B, T, C):
    g = torch.Generator(device="cuda").manual_seed(B)
    z = torch.randn((B, T, C), generator=g, device="cuda")
    W = (0.1 * torch.randn((C, 5 * C), generator=g, device="cuda")).bfloat16()
    want = _chain(gwx, z, W, 4, torch.cuda.synchronize)
    for _ in range(3):
        got = _chain(gwx, z, W, 4, lambda: None)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
    gwx.device_status()
