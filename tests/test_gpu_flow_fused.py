"""The flow's fused density and training kernels against the same passes layer by layer through the
library's stage entries (needs a GPU).

Both round at the same places and sum in the same order, so ln q and the context's gradient are equal bit
for bit.  Weight and bias gradients are FP32 sums over n rows in another order: a sum of n terms differs by
at most n 2^-24 sum |t|, and sum |t| <= sqrt(n) |t|_2, so per tensor the 2-norm of the difference stays
below n^1.5 2^-24 of the gradient's for terms that do not cancel; the loss is an FP64 sum (1e-12)."""
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


WL = workloads.workload("small")
MEAN, SCALE = [20.0, 0.6, 1000.0, 0.0, 3.0, 0.0, 3.0, 3.0], [8.0, 0.3, 500.0, 0.6, 1.8, 0.6, 1.8, 1.8]
F_FEAT = 1968


def _setup(gwx, C, H, K, n, seed):
    shape = workloads.flow_shape(features=F_FEAT, group=4, embed_hidden=64, context=C, layers=K, hidden=H)
    size, offs = gwx.flow_layout(shape)
    params = torch.zeros(size, device="cuda")
    tensors = workloads.random_flow_params(seed, shape)
    for o, a in zip(offs, tensors):
        params[o:o + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
    p16 = params.bfloat16()
    view = [(p16 if a.ndim == 2 else params)[o:o + a.size].view(a.shape) for o, a in zip(offs, tensors)]
    rng = np.random.default_rng(seed)
    ctx = torch.from_numpy(rng.normal(0, 1, (n, C))).cuda().bfloat16()
    theta = torch.from_numpy(workloads.random_theta(seed, n, WL["prior"])).cuda()
    y = torch.zeros((n, 2, WL["N"]), device="cuda")
    return shape, params, p16, offs, view, ctx, theta, y


def _density(gwx, view, K, x, ctx):
    tape, ss = [None] * K, torch.empty(x.shape[0], device="cuda")
    for l in reversed(range(K)):
        w = view[6 + 6 * l:12 + 6 * l]
        X = gwx.flow_conditioner_input(l, x, ctx)
        g1 = gwx.dense_bf16(X, w[0], w[1], gwx.ACT_RELU, out_dtype=torch.bfloat16)
        g2 = gwx.dense_bf16(g1, w[2], w[3], gwx.ACT_RELU, out_dtype=torch.bfloat16)
        o = gwx.dense_bf16(g2, w[4], w[5])
        x = gwx.flow_coupling(l, -1, x, o, ss, l == K - 1)
        tape[l] = (X, g1, g2, o, x)
    return x, ss, tape


# widths and contexts of the rule's range (one and two 128-column parts, 64 columns of input or more), rows
# that fill a part of a tile, exactly one, and one more row group than tiles
@pytest.mark.parametrize("C,H,K,n", [(8, 128, 1, 8), (64, 256, 5, 136), (56, 256, 2, 128), (32, 128, 4, 264),
                                     (64, 256, 3, 1000)])
def test_training_equals_layers(gwx, C, H, K, n):
    shape, params, p16, offs, view, ctx, theta, y = _setup(gwx, C, H, K, n, 5 * C + H + n)
    z, ss, tape = _density(gwx, view, K, gwx.flow_targets(theta, MEAN, SCALE), ctx)
    _, loss, g = gwx.flow_nll(z, ss)
    want, dctx = {}, torch.empty((n, C), device="cuda")
    for l in range(K):
        X, g1, g2, o, w = tape[l]
        v = view[6 + 6 * l:12 + 6 * l]
        d, gu = gwx.flow_coupling_backward(l, w, o, g, 1.0 / n)
        for t, (inp, act) in ((4, (g2, gwx.ACT_NONE)), (2, (g1, gwx.ACT_RELU)), (0, (X, gwx.ACT_RELU))):
            d, want[6 + 6 * l + t], want[7 + 6 * l + t] = gwx.dense_bf16_backward(inp, v[t], v[t + 1], d, act)
        gwx.flow_input_backward(l, d, gu, dctx, l == 0)
        g = gu
    grads, got_dctx = torch.full_like(params, 7.0), torch.empty((n, C), device="cuda")
    got = gwx.flow_train_step(shape, params, p16, grads, _zeros(params), _zeros(params), 0, 1e-3, MEAN, SCALE, y,
                              theta, WL["fs"], WL["f_lo"], ctx=ctx, d_ctx=got_dctx)
    gwx.device_status()
    assert torch.equal(got_dctx, dctx)
    assert abs(got.item() - loss.item()) <= 1e-12 * abs(loss.item())
    for t, a in want.items():
        b = grads[offs[t]:offs[t] + a.numel()].view(a.shape).double()
        assert (b - a.double()).norm() <= n ** 1.5 * 2.0 ** -24 * a.double().norm(), t
    assert not grads[:offs[6]].any()          # the caller's summary: no gradients of the built-in one


def _zeros(t):
    return torch.zeros_like(t)


@pytest.mark.parametrize("C,H,K,n", [(120, 256, 3, 130), (64, 128, 4, 77), (16, 256, 16, 1)])
def test_log_prob_equals_layers(gwx, C, H, K, n):
    shape, params, p16, offs, view, ctx, theta, y = _setup(gwx, C, H, K, n, C + H + n)
    z, ss, _ = _density(gwx, view, K, gwx.flow_targets(theta, MEAN, SCALE), ctx)
    want = (-0.5 * (z.double() ** 2).sum(1) - 4.0 * np.log(2.0 * np.pi) - sum(np.log(SCALE)) - ss.double()).cpu().numpy()
    got = gwx.flow_log_prob(shape, params, p16, MEAN, SCALE, y, theta, WL["fs"], WL["f_lo"], ctx=ctx).cpu().numpy()
    assert np.allclose(got, want, rtol=1e-13, atol=1e-12)
