"""gwx_group_norm_backward_src (the gradient masked, routed back through the max pool or spread over
time on the fly) and the products from bfloat16 dz, against the same steps as passes of their own
(needs a GPU).  Equal operations in another order only across FP64 sums: the FP32 gradient equal, dz
its bfloat16 rounding up to the rounding of the group means (2^-8 of an element where that moves it
across a boundary, in few), parameter gradients to FP32 rounding."""
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


# every column-quad layout (8, 16, 32 and 256 quads), times that fill less than one run of rows, an odd
# number of them, more runs than slices
@pytest.mark.parametrize("B,T,C", [(1, 1, 32), (3, 37, 64), (2, 514, 64), (5, 130, 128), (2, 9, 1024)])
@pytest.mark.parametrize("kind", [0, 1, 2, 3])
def test_against_separate_passes(gwx, B, T, C, kind):
    from paper_2407_19048_gb300 import _lib
    lib, st, G = _lib.load(), gwx._stream(), 8
    g = torch.Generator(device="cuda").manual_seed(B + T + C + kind)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    z, gamma, beta = 2.0 + rnd(B, T, C), 1.0 + 0.1 * rnd(C), 0.1 * rnd(C)
    out, ms = torch.empty((B, T, C), dtype=torch.bfloat16, device="cuda"), torch.empty((B, G, 2), device="cuda")
    gwx._check(lib.gwx_group_norm(gwx._ptr(z), B, T, C, G, gwx._ptr(gamma), gwx._ptr(beta), None, None, 1, gwx._ptr(out),
                                  None, gwx._ptr(ms), st))
    To, arg = (T - 1) // 2 + 1, None
    dy = rnd(B, T, C)
    d = dy
    if kind == 2:
        pooled, arg = torch.empty((B, To, C), dtype=torch.bfloat16, device="cuda"), \
            torch.empty((B, To, C), dtype=torch.uint8, device="cuda")
        gwx._check(lib.gwx_maxpool(gwx._ptr(out), B, T, C, gwx._ptr(pooled), gwx._ptr(arg), st))
        assert torch.equal(pooled.float(), torch.nn.functional.max_pool1d(out.float().transpose(1, 2), 3, 2, 1).transpose(1, 2))
        dy, d = rnd(B, To, C), torch.empty((B, T, C), device="cuda")
        gwx._check(lib.gwx_maxpool_backward(gwx._ptr(dy), gwx._ptr(arg), B, T, C, gwx._ptr(d), st))
    elif kind == 3:
        dy, d = rnd(B, C), torch.empty((B, T, C), device="cuda")
        gwx._check(lib.gwx_mean_time_backward(gwx._ptr(dy), B, T, C, gwx._ptr(d), st))
    if kind:
        m = torch.empty_like(d)
        gwx._check(lib.gwx_relu_mask(gwx._ptr(d), gwx._ptr(out), d.numel(), gwx._ptr(m), st))
        d = m
    x = lambda *s, dt=torch.float32: torch.empty(s, dtype=dt, device="cuda")  # noqa: E731
    dz, dg, db = x(B, T, C), x(C), x(C)
    scratch = x(lib.gwx_group_norm_backward_scratch(B, C, G), dt=torch.uint8)
    gwx._check(lib.gwx_group_norm_backward(gwx._ptr(d), gwx._ptr(z), B, T, C, G, gwx._ptr(ms), gwx._ptr(gamma),
                                           gwx._ptr(scratch), gwx._ptr(dz), gwx._ptr(dg), gwx._ptr(db), st))
    dz16, dsum, dg2, db2 = x(B, T, C, dt=torch.bfloat16), x(B, T, C), x(C), x(C)
    scratch = x(lib.gwx_group_norm_backward_src_scratch(B, C, G), dt=torch.uint8)
    gwx._check(lib.gwx_group_norm_backward_src(kind, gwx._ptr(dy), gwx._ptr(out), gwx._ptr(arg), gwx._ptr(z), B, T, C, G,
                                               gwx._ptr(ms), gwx._ptr(gamma), gwx._ptr(scratch), gwx._ptr(dz16),
                                               gwx._ptr(dsum), gwx._ptr(dg2), gwx._ptr(db2), st))
    assert torch.equal(dsum, d)
    want = dz.bfloat16().float()
    diff = (dz16.float() - want).abs()
    assert (diff <= 2.0 ** -7 * want.abs() + 1e-6).all() and (diff > 0).float().mean() <= 1e-3
    for p, q in ((dg2, dg), (db2, db)):
        assert (p - q).abs().max() <= 1e-6 * (1.0 + q.abs().max())


def test_refusals(gwx):
    from paper_2407_19048_gb300 import _lib
    lib, t = _lib.load(), torch.zeros(1 << 16, device="cuda")
    p = gwx._ptr(t)
    for kind, C, out, arg in ((1, 24, p, None), (4, 64, p, None), (1, 64, None, None), (2, 64, p, None)):
        assert lib.gwx_group_norm_backward_src(kind, p, out, arg, p, 1, 8, C, 8, p, p, p, p, None, p, p, None) != 0
    assert lib.gwx_conv1d_bf16_backward_dz(p, p, p, 1, 128, 64, 64, 5, None, p, p, p, 0, None) != 0
    assert lib.gwx_dense_bf16_backward_dz(p, p, p, 8, 8, 12, p, p, p, 1 << 16, None) != 0
