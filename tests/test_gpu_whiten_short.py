"""Whitening of windows shorter than a warp's share (needs a GPU): one window a block for a few, several side by side for
many.  Which form a window takes depends on how many there are, not what comes out: the bits of each are those of the
window among few, whatever the place in its block, with a last block that is not full, for detectors whose filters
differ, from rows of either alignment, and in place."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FS, F_LO, SEG = 2048.0, 20.0, 256


@pytest.fixture(scope="module")
def gwx():
    import paper_2407_19048_gb300 as m
    from paper_2407_19048_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    m.init()
    return m


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("N,D,B", [(256, 1, 1029), (256, 3, 701), (256, 4, 5000), (512, 1, 1029), (512, 2, 400)])
def test_many_windows_have_the_bits_of_few(gwx, N, D, B, aligned):
    g = torch.Generator(device="cuda").manual_seed(N + D)
    buf = 1e-21 * torch.randn(B * D * N + 2, generator=g, device="cuda")
    x = buf[: B * D * N].view(B, D, N) if aligned else buf[2:].view(B, D, N)
    psd = 1e-46 * (1.0 + torch.rand((D, SEG // 2 + 1), generator=g, device="cuda", dtype=torch.float64))
    few = max(1, 64 // D)   # far fewer than windows share blocks
    want = torch.cat([gwx.whiten(x[i:i + few].contiguous(), psd, SEG, FS, F_LO) for i in range(0, B, few)])
    got = gwx.whiten(x, psd, SEG, FS, F_LO)
    assert torch.equal(got, want)
    gwx.whiten(x, psd, SEG, FS, F_LO, out=x)
    assert torch.equal(x, want)
    gwx.device_status()
