"""gwx_group_norm_backward with scratch that is aligned for doubles and no further (needs a GPU): the bits of the
call with aligned scratch, for the parameter sums that come out of the pass over the samples and for those that have a
kernel of their own."""
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


@pytest.mark.parametrize("B,T,C", [(3, 40, 64), (3, 40, 24)])
def test_scratch_at_eight_bytes(gwx, B, T, C):
    from paper_2407_19048_gb300 import _lib
    lib, p, G = _lib.load(), gwx._ptr, 8
    g = torch.Generator(device="cuda").manual_seed(C)
    z, dy = torch.randn((B, T, C), generator=g, device="cuda"), torch.randn((B, T, C), generator=g, device="cuda")
    gamma, ms = torch.ones(C, device="cuda"), torch.rand((B, G, 2), generator=g, device="cuda")
    nb, got = lib.gwx_group_norm_backward_scratch(B, C, G), []
    for shift in (0, 8):
        buf = torch.empty(nb + 256 + shift, dtype=torch.uint8, device="cuda")
        scratch = buf[(-buf.data_ptr()) % 256 + shift:]
        out = [torch.empty_like(z), torch.empty(C, device="cuda"), torch.empty(C, device="cuda")]
        gwx._check(lib.gwx_group_norm_backward(p(dy), p(z), B, T, C, G, p(ms), p(gamma), p(scratch), *map(p, out),
                                               gwx._stream()))
        got.append(out)
    assert all(torch.equal(a, b) for a, b in zip(*got))
