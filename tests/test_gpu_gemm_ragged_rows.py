"""Products whose rows are not multiples of four values (needs a GPU): the bits of the same product with its columns
filled up to a multiple of four, in both output types, with and without bias and activation, for narrow and wide
products, chunks of 32 columns that are full, half full and nearly empty, and rows that end in the middle of a warp's 32."""
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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M,N,K", [(130, 1, 64), (1, 2, 8), (77, 7, 72), (130, 9, 64), (259, 33, 128), (40, 41, 8),
                                   (130, 66, 64), (1000, 257, 136), (513, 1002, 64), (4100, 2559, 1024)])
def test_ragged_rows(gwx, M, N, K, dtype):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn((M, K), generator=g, device="cuda").bfloat16()
    full = -(-N // 4) * 4
    B = torch.randn((full, K), generator=g, device="cuda").bfloat16()
    b = torch.randn(full, generator=g, device="cuda")
    for bias, act in ((None, gwx.ACT_NONE), (b, gwx.ACT_NONE), (b, gwx.ACT_RELU), (b, gwx.ACT_GELU)):
        want = gwx.dense_bf16(A, B, bias, act, out_dtype=dtype)[:, :N]
        buf = torch.full((M * N + 64,), 7.0, dtype=dtype, device="cuda")
        got = buf[: M * N].view(M, N)
        gwx.dense_bf16(A, B[:N].contiguous(), None if bias is None else bias[:N].contiguous(), act, out=got, out_dtype=dtype)
        assert torch.equal(got, want)
        assert (buf[M * N:] == 7.0).all()
