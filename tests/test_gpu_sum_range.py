"""Sums in two-float arithmetic (csrc/sum2.cuh) against FP64: the group norm's statistics, output and gradients at every
layout of a block, and totals beyond FP32's range, where FP64 sums are finite (needs a GPU).

Bounds, u = 2^-24: a run of 16 rows of four channels is summed in FP32 (a difference, two levels of the four, 16
additions: 19 roundings, and up to four more for the products of a term), the runs with their errors kept.  So a mean of
terms t is off by at most 24 u mean|t|, a mean of products by 28 u; a variance, from the mean square q of z - z_0 and the
square of its mean, by 70 u q."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U, G, EPS = 2.0 ** -24, 8, 1e-5


@pytest.fixture(scope="module")
def gwx():
    import paper_2407_19048_gb300 as m
    from paper_2407_19048_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    m.init()
    return m


def _empty(*s, dt=torch.float32):
    return torch.empty(s, dtype=dt, device="cuda")


def _forward(gwx, z, gamma, beta):
    from paper_2407_19048_gb300 import _lib
    B, T, C = z.shape
    out, ms, p = _empty(B, T, C, dt=torch.bfloat16), _empty(B, G, 2), gwx._ptr
    gwx._check(_lib.load().gwx_group_norm(p(z), B, T, C, G, p(gamma), p(beta), None, None, 1, p(out), None, p(ms),
                                          gwx._stream()))
    return out, ms


def _backward(gwx, dy, z, ms, gamma, out):
    """(dz, dgamma, dbeta) of dy as given, and the same of dy [out > 0] by the entry that masks."""
    from paper_2407_19048_gb300 import _lib
    lib, p, (B, T, C), st = _lib.load(), gwx._ptr, z.shape, gwx._stream()
    plain = [_empty(B, T, C), _empty(C), _empty(C)]
    ws = _empty(lib.gwx_group_norm_backward_scratch(B, C, G), dt=torch.uint8)
    gwx._check(lib.gwx_group_norm_backward(p(dy), p(z), B, T, C, G, p(ms), p(gamma), p(ws), *map(p, plain), st))
    masked = [_empty(B, T, C, dt=torch.bfloat16), _empty(C), _empty(C)]
    ws = _empty(lib.gwx_group_norm_backward_src_scratch(B, C, G), dt=torch.uint8)
    gwx._check(lib.gwx_group_norm_backward_src(1, p(dy), p(out), None, p(z), B, T, C, G, p(ms), p(gamma), p(ws),
                                               p(masked[0]), None, p(masked[1]), p(masked[2]), st))
    return plain, masked


def _groups(x):
    """[B][T][C] as [B][T][G][C / G], and the mean over time and a group's channels, shaped to subtract."""
    return x.view(*x.shape[:2], G, -1)


def _mean(x):
    return _groups(x).mean((1, 3), keepdim=True)


def _check_gradients(got, d, z, ms, gamma, rounding):
    x, dg = _groups(z), _groups(d * gamma)
    mean, rstd = (ms.double()[:, None, :, i, None] for i in (0, 1))
    xhat = (x - mean) * rstd
    m1, m2 = dg.mean((1, 3), keepdim=True), (dg * xhat).mean((1, 3), keepdim=True)
    dz = rstd * (dg - m1 - xhat * m2)
    tol = rstd * (4 * U * (dg.abs() + m1.abs() + 3 * (xhat * m2).abs()) + 24 * U * dg.abs().mean((1, 3), keepdim=True)
                  + 28 * U * xhat.abs() * (dg * xhat).abs().mean((1, 3), keepdim=True))
    assert ((_groups(got[0].double()) - dz).abs() <= tol + rounding * dz.abs()).all()
    flat = xhat.reshape(z.shape)
    for g, t, k in ((got[1], d * flat, 28), (got[2], d, 24)):
        total = t.sum((0, 1))
        assert ((g.double() - total).abs() <= k * U * t.abs().sum((0, 1)) + 2 * U * total.abs()).all()


# column quads from 8 to 256 a sample (C = 32 .. 1024), less than one run of rows, odd numbers of them, several runs
@pytest.mark.parametrize("B,T,C", [(1, 1, 32), (3, 37, 64), (2, 514, 64), (5, 130, 128), (2, 9, 1024), (3, 700, 256)])
def test_group_norm_against_fp64(gwx, B, T, C):
    g = torch.Generator(device="cuda").manual_seed(B + T + C)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    z, gamma, beta, dy = 2.0 + r(B, T, C), 1.0 + 0.1 * r(C), 0.1 * r(C), r(B, T, C)
    out, ms = _forward(gwx, z, gamma, beta)
    z64 = z.double()
    d0 = _groups(z64) - _groups(z64)[:, :1, :, :1]
    mean, var, q = _mean(z64), (_groups(z64) - _mean(z64)).square().mean((1, 3), keepdim=True), \
        d0.square().mean((1, 3), keepdim=True)
    got_mean, got_rstd = (ms.double()[:, None, :, i, None] for i in (0, 1))
    assert ((got_mean - mean).abs() <= 24 * U * d0.abs().mean((1, 3), keepdim=True) + 2 * U * mean.abs()).all()
    rstd = (var + EPS).rsqrt()
    assert ((got_rstd / rstd - 1).abs() <= 35 * U * q / (var + EPS) + 2 * U).all()
    n = ((_groups(z64) - got_mean) * got_rstd).reshape(B, T, C) * gamma.double()
    y = torch.relu(n + beta.double())
    assert ((out.double() - y).abs() <= 2.0 ** -8 * y + 4 * U * (n.abs() + beta.double().abs())).all()
    plain, masked = _backward(gwx, dy, z, ms, gamma, out)
    _check_gradients(plain, dy.double(), z64, ms, gamma.double(), U)
    _check_gradients(masked, (dy * (out > 0)).double(), z64, ms, gamma.double(), 2.0 ** -8)


def test_gradient_sums_beyond_fp32(gwx):
    """Sums of a sample of 5e38 and 4e39, group means of 1e36, totals over the samples that cancel."""
    B, T, C = 2, 514, 64
    g = torch.Generator(device="cuda").manual_seed(3)
    z, gamma = torch.randn((B, T, C), generator=g, device="cuda"), torch.ones(C, device="cuda")
    out, ms = _forward(gwx, z, gamma, torch.zeros(C, device="cuda") + 9.0)   # (no output is masked)
    dy = 1e36 * (0.9 + 0.2 * torch.rand((B, T, C), generator=g, device="cuda"))
    dy[1] *= -1.0
    for got, rounding in zip(_backward(gwx, dy, z, ms, gamma, out), (U, 2.0 ** -8)):
        assert all(torch.isfinite(x).all() for x in got)
        _check_gradients(got, dy.double(), z.double(), ms, gamma.double(), rounding)


def test_mean_of_values_whose_sum_is_beyond_fp32(gwx):
    """Squares beyond FP32 make the deviation infinite (output beta); the mean is finite in FP64 sums."""
    B, T, C = 2, 514, 64
    g = torch.Generator(device="cuda").manual_seed(4)
    z = 2e36 * torch.rand((B, T, C), generator=g, device="cuda")
    z[:, 0] = 0.0
    out, ms = _forward(gwx, z, torch.ones(C, device="cuda"), torch.full((C,), 0.5, device="cuda"))
    mean = _mean(z.double())[:, 0, :, 0]
    assert ((ms[..., 0].double() - mean).abs() <= 26 * U * mean).all()
    assert (ms[..., 1] == 0).all() and (out == 0.5).all()


@pytest.mark.parametrize("M", [4096, 8200])   # one slice of partial sums, two
def test_bias_gradient_beyond_fp32(gwx, M):
    """Integers times 2^118, exact in every partial sum: column sums of 10^40 that cancel down to FP32; infinities."""
    N, K, g = 40, 8, torch.Generator(device="cuda").manual_seed(M)
    a = torch.randint(1, 5, (M // 2, N), generator=g, device="cuda").double()
    e = torch.randint(-1, 2, (M // 2, N), generator=g, device="cuda").double()
    dY = (torch.cat([a, e - a]) * 2.0 ** 118).float()
    X, W = torch.zeros((M, K), device="cuda").bfloat16(), torch.zeros((N, K), device="cuda").bfloat16()
    b = torch.zeros(N, device="cuda")
    db = gwx.dense_bf16_backward(X, W, b, dY, gwx.ACT_NONE)[2]
    assert torch.equal(db.double(), e.sum(0) * 2.0 ** 118)
    dY[5, 1], dY[M - 1, 2], dY[7, 3], dY[M - 7, 3] = float("inf"), float("-inf"), float("inf"), float("-inf")
    bad = gwx.dense_bf16_backward(X, W, b, dY, gwx.ACT_NONE)[2]
    assert bad[1] == float("inf") and bad[2] == float("-inf") and bad[3].isnan()
    assert torch.equal(bad[[0] + list(range(4, N))], db[[0] + list(range(4, N))])
