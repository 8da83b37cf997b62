"""Kernels launched under the end of their predecessors (needs a GPU): a chain of calls over the same buffers gives
the bits of the same calls with a synchronisation after each, on one stream, on two at once, and replayed as a
graph."""
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


def _state(seed, M, K, N):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return {"x": torch.randn((M, K), generator=g, device="cuda").bfloat16(),
            "w": (0.1 * torch.randn((N, K), generator=g, device="cuda")).bfloat16(),
            "v": (0.1 * torch.randn((K, N), generator=g, device="cuda")).bfloat16(),
            "b": torch.randn(N, generator=g, device="cuda"), "c": torch.zeros(K, device="cuda"),
            "strain": 1e-21 * torch.randn((3, 2, 2048), generator=g, device="cuda"),
            "psd": torch.full((2, 513), 1e-46, dtype=torch.float64, device="cuda")}


def _chain(gwx, s, steps, sync):
    """Each step's products feed the next, through buffers that are written again every step."""
    keep = []
    x, y = s["x"].clone(), s["strain"].clone()
    for _ in range(steps):
        h = gwx.dense_bf16(x, s["w"], s["b"], gwx.ACT_RELU, out_dtype=torch.bfloat16)
        sync()
        dX, dW, db = gwx.dense_bf16_backward(x, s["w"], s["b"], h.float(), gwx.ACT_RELU)
        sync()
        x.copy_(torch.tanh(gwx.dense_bf16(h, s["v"], s["c"], gwx.ACT_NONE)).bfloat16())
        gwx.whiten(y, s["psd"], 1024, 2048.0, 20.0, out=y)
        sync()
        y.mul_(1e-21)
        keep += [dX, dW, db]
    return keep + [x, y]


@pytest.mark.parametrize("M,K,N", [(8, 64, 64), (200, 136, 72), (2056, 264, 520)])
def test_chains_keep_their_bits(gwx, M, K, N):
    a, b = _state(1, M, K, N), _state(2, M, K, N)
    want = [_chain(gwx, s, 6, torch.cuda.synchronize) for s in (a, b)]
    nothing = lambda: None  # noqa: E731
    for w, s in zip(want, (a, b)):
        assert all(torch.equal(p, q) for p, q in zip(w, _chain(gwx, s, 6, nothing)))
    streams, got = [torch.cuda.Stream(), torch.cuda.Stream()], []
    torch.cuda.synchronize()
    for s, st in zip((a, b), streams):
        with torch.cuda.stream(st):
            got.append(_chain(gwx, s, 6, nothing))
    torch.cuda.synchronize()
    for w, r in zip(want, got):
        assert all(torch.equal(p, q) for p, q in zip(w, r))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = _chain(gwx, a, 3, nothing)
    ref = _chain(gwx, a, 3, torch.cuda.synchronize)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(p, q) for p, q in zip(ref, out))
    gwx.device_status()
