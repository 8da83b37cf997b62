"""The fused sampling kernel against the same pass layer by layer through the library's stage entries (needs a
GPU).  Both round the draws at the same places, so these are equal bit for bit.  The log scales (each at most 3)
are FP32 sums of 4 K terms, one after the other in the fused kernel and layer by layer in the stages: an order's
error is at most 4 K 2^-24 of the sum of magnitudes, 12 K, so ln q differs by at most 96 K^2 2^-24."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WL = workloads.workload("small")
MEAN, SCALE = [20.0, 0.6, 1000.0, 0.0, 3.0, 0.0, 3.0, 3.0], [8.0, 0.3, 500.0, 0.6, 1.8, 0.6, 1.8, 1.8]


@pytest.fixture(scope="module")
def gwx():
    import paper_2407_19048_gb300 as m
    from paper_2407_19048_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    m.init()
    return m


# both hidden widths; context widths at the first K step, the edges of the second K-block and the widest; one
# layer, the parity of the bias buffers, all four splits; one draw, a tile less and more one, two rounds of tiles
@pytest.mark.parametrize("C,H,K,S", [(8, 128, 1, 1), (8, 256, 2, 127), (56, 256, 5, 129), (64, 256, 3, 300),
                                     (72, 128, 4, 257), (120, 256, 7, 128), (120, 128, 9, 40), (64, 256, 2, 19600)])
def test_fused_draws_equal_the_layered_pass(gwx, C, H, K, S):
    shape = workloads.flow_shape(features=1968, group=4, embed_hidden=64, context=C, layers=K, hidden=H)
    size, offs = gwx.flow_layout(shape)
    params = torch.zeros(size, device="cuda")
    tensors = workloads.random_flow_params(C + H + K, shape)
    for o, a in zip(offs, tensors):
        params[o:o + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
    p16 = params.bfloat16()
    view = [(p16 if a.ndim == 2 else params)[o:o + a.size].view(a.shape) for o, a in zip(offs, tensors)]
    E = 3
    ctx = torch.from_numpy(np.random.default_rng(C).normal(0, 1, (E, C))).cuda().bfloat16()
    ev = torch.tensor([0, S // 3, S // 3, S], dtype=torch.int64, device="cuda")
    y = torch.zeros((E, 2, WL["N"]), device="cuda")
    got = gwx.sample_posterior(shape, params, p16, MEAN, SCALE, WL["prior"], y, WL["fs"], WL["f_lo"], ev, 31, 7,
                               ctx=ctx)
    z = gwx.flow_base(31, 7, 0, S)
    x, ss = z, torch.empty(S, device="cuda")
    for l in range(K):
        w = view[6 + 6 * l:12 + 6 * l]
        X = gwx.flow_conditioner_input(l, x, ctx, ev)
        g1 = gwx.dense_bf16(X, w[0], w[1], gwx.ACT_RELU, out_dtype=torch.bfloat16)
        g2 = gwx.dense_bf16(g1, w[2], w[3], gwx.ACT_RELU, out_dtype=torch.bfloat16)
        x = gwx.flow_coupling(l, 1, x, gwx.dense_bf16(g2, w[4], w[5]), ss, l == 0)
    ref = gwx.flow_proposal(x, z, ss, MEAN, SCALE, WL["prior"], 31, 7)
    assert torch.equal(got[0], ref[0])
    assert torch.isfinite(got[1]).all() and torch.equal(torch.isfinite(got[2]), torch.isfinite(ref[2]))
    tol = 96 * K * K * 2.0 ** -24 if K > 1 else 0.0
    for a, b in zip(got[1:], ref[1:]):
        ok = torch.isfinite(b)
        assert ((a - b)[ok].abs() <= tol).all()
    gwx.device_status()
