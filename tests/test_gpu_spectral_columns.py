"""The flow's feature rows made in one pass over the spectra against the three kernels that make them kind by kind
(needs a GPU): the same sums in the same order, so the flow's density given the windows equals, bit for bit, its
density given the context that the separate calls lead to."""
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


# one to four detectors, groups that leave a remainder, a group a bin, fewer groups than a block's 128
@pytest.mark.parametrize("D,G,extra", [(1, 4, 0), (1, 4, 2), (2, 4, 3), (2, 5, 1), (3, 7, 3), (4, 3, 3), (2, 1, 2),
                                       (3, 64, 3)])
@pytest.mark.parametrize("B", [1, 9])
def test_rows_in_one_pass(gwx, D, G, extra, B):
    N, fs, f_lo = WL["N"], WL["fs"], WL["f_lo"]
    k_lo = int(-(-f_lo * N // fs))
    ng = (N // 2 - k_lo) // G
    used = D * ng + (D * (D - 1) * ng if extra & 1 else 0) + (2 * D * ng if extra & 2 else 0)
    F = (used + 7) // 8 * 8 + 8
    shape = workloads.flow_shape(features=F, group=G, embed_hidden=64, context=32, layers=2, hidden=64)
    shape["extra"] = extra
    size, offs = gwx.flow_layout(shape)
    params = torch.zeros(size, device="cuda")
    tensors = workloads.random_flow_params(D + G, shape)
    for o, a in zip(offs, tensors):
        params[o:o + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
    p16 = params.bfloat16()
    y = torch.randn((B, D, N), generator=torch.Generator(device="cuda").manual_seed(G), device="cuda")
    theta = torch.from_numpy(workloads.random_theta(3, B, WL["prior"])).cuda()
    got = gwx.flow_log_prob(shape, params, p16, MEAN, SCALE, y, theta, fs, f_lo)
    feat = gwx.spectral_features(y, fs, f_lo, G, F)
    col = D * ng
    if extra & 1:
        if D > 1:
            gwx.cross_features(y, fs, f_lo, G, F, col, feat)
        col += D * (D - 1) * ng
    if extra & 2:
        gwx.lag_features(y, fs, f_lo, G, F, col, feat)
    h = feat
    for t, act in ((0, gwx.ACT_RELU), (2, gwx.ACT_RELU), (4, gwx.ACT_NONE)):
        w = p16[offs[t]:offs[t] + tensors[t].size].view(tensors[t].shape)
        b = params[offs[t + 1]:offs[t + 1] + tensors[t + 1].size]
        h = gwx.dense_bf16(h, w, b, act, out_dtype=torch.bfloat16)
    want = gwx.flow_log_prob(shape, params, p16, MEAN, SCALE, y, theta, fs, f_lo, ctx=h)
    assert torch.equal(got, want)
    assert torch.isfinite(got).all()
