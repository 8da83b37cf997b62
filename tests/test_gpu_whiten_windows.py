"""Whitening in the fused kernel's own windows (needs a GPU): every window size, one to four detectors, fewer
windows than blocks and more, rows that are not 16-byte aligned (no bulk copies), in place.

Tolerance: two single-precision transforms of N/2 points with exactly rounded constants stay within
(2 log2 N + 6) 2^-24 of the exact result in the 2-norm (one rounding a butterfly level and transform, and the filter,
the packing and the 1/n products), as a share of the largest whitened window."""
import math

import numpy as np
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


def _exact(x, psd, unwhiten):
    from oracle import spectral
    f = spectral.unwhiten if unwhiten else spectral.whiten
    return f(x.cpu().numpy().astype(np.float64), psd.cpu().numpy(), SEG, FS, F_LO)


@pytest.mark.parametrize("unwhiten", [False, True])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("N,D,B", [(256, 4, 1), (256, 3, 700), (512, 1, 5), (1024, 2, 333), (2048, 4, 77),
                                   (4096, 3, 1), (8192, 3, 131), (16384, 4, 41), (16384, 1, 1)])
def test_windows_against_the_oracle(gwx, N, D, B, aligned, unwhiten):
    g = torch.Generator(device="cuda").manual_seed(N + 7 * D + B)
    buf = torch.randn(B * D * N + 2, generator=g, device="cuda")
    if not unwhiten:
        buf *= 1e-21
    x = buf[: B * D * N].view(B, D, N) if aligned else buf[2:].view(B, D, N)
    psd = 1e-46 * (1.0 + torch.rand((D, SEG // 2 + 1), generator=g, device="cuda", dtype=torch.float64))
    ref = _exact(x, psd, unwhiten)
    f = gwx.unwhiten if unwhiten else gwx.whiten
    got = f(x, psd, SEG, FS, F_LO)
    tol = (2 * math.log2(N) + 6) * 2.0 ** -24
    err = np.linalg.norm(got.cpu().numpy() - ref, axis=-1)
    assert np.all(err <= tol * np.linalg.norm(ref, axis=-1).max())
    f(x, psd, SEG, FS, F_LO, out=x)   # in place: the same bits
    assert torch.equal(x, got)
    gwx.device_status()
