"""A batch's preparation in one launch and the fused pass over single windows (needs a GPU).

A draw depends on its index, the seed and the step alone, so a small batch (whose windows are dealt out one by
one) equals the head of a large one (dealt out by draws) bit for bit; the preparation equals the prior draws and
the set-up of given parameters."""
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


DETS = ("H1", "L1", "V1", "H1")


def _run(gwx, N, D, L, B):
    wl = workloads.workload("hl3")
    g = torch.Generator(device="cuda").manual_seed(N + D)
    noise = 1e-21 * torch.randn((D, L), generator=g, device="cuda")
    psd = torch.full((D, 513), 1e-46, dtype=torch.float64, device="cuda")
    return gwx.simulate_batch(wl["prior"], 11, 2, noise, psd, 1024, 2048.0, 20.0, DETS[:D], 0.3, B, N)


# the smallest window, one block and several blocks an SM, the staged shapes, a background whose rows are neither
# 16- nor 8-byte aligned; batches of one draw, of a part of a set-up block, one draw more than a block
@pytest.mark.parametrize("N,D,L,big", [(256, 4, 4096, 3000), (2048, 2, 4099, 2500), (8192, 3, 16384, 700),
                                       (16384, 3, 32770, 470), (16384, 1, 32768, 470)])
def test_small_batch_is_the_head_of_a_large_one(gwx, N, D, L, big):
    y, theta, off = _run(gwx, N, D, L, big)
    for B in (1, 5, 33):
        ys, ts, os_ = _run(gwx, N, D, L, B)
        assert torch.equal(ys, y[:B]) and torch.equal(ts, theta[:, :B]) and torch.equal(os_, off[:B])
    gwx.device_status()


@pytest.mark.parametrize("D", [1, 2, 3, 4])
def test_preparation_equals_prior_and_given_parameters(gwx, D):
    from paper_2407_19048_gb300 import _lib
    lib, wl = _lib.load(), workloads.workload("hl3")
    N, L, B = 1024, 4096, 77
    y, theta, off = _run(gwx, N, D, L, B)
    t2, o2 = gwx.sample_prior(wl["prior"], 11, 2, B, L, N)
    assert torch.equal(theta, t2) and torch.equal(off, o2)
    g = torch.Generator(device="cuda").manual_seed(N + D)
    noise = 1e-21 * torch.randn((D, L), generator=g, device="cuda")
    psd = torch.full((D, 513), 1e-46, dtype=torch.float64, device="cuda")
    ids, _ = gwx._det_ids(DETS[:D])
    b = gwx.SimulateBuffers(B, D, N)
    p = gwx._ptr
    gwx._check(lib.gwx_prepare_theta(p(theta), L, N, 2048.0, 20.0, ids, D, 0.3, B, p(b.ws), b.ws_bytes, gwx._stream()))
    gwx._check(lib.gwx_simulate_prepared(p(noise), L, p(psd), 1024, 2048.0, 20.0, D, B, N, p(off), p(b.y), 0, p(b.ws),
                                         b.ws_bytes, gwx._stream()))
    assert torch.equal(b.y, y)
