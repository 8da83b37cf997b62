"""The marginal likelihood's first pass reads only the table blocks that a template's last bin
reaches: templates ending on either side of every block boundary, against the FP64 oracle
(needs a GPU).  Tolerance: |Delta ln L| <= 1e-3, as for the marginal likelihood itself."""
import math

import numpy as np
import pytest

import workloads
from oracle import constants as C
from oracle import likelihood, pipeline

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


# (workload, sampling rate, window, u, n_tc): transforms of n = 2^10, 2^9 (last radix 16 and
# two) and 2^12 points; the block of the tables is n/16 bins
@pytest.mark.parametrize("name,fs,T,u,n_tc", [("small", 1024, 2.0, 4, 512), ("small", 512, 2.0, 2, 65),
                                              ("hl3", 2048, 4.0, 2, 40)])
@pytest.mark.parametrize("S", [1, 33])
def test_templates_around_the_block_edges(gwx, name, fs, T, u, n_tc, S):
    wl = workloads.resampled(name, fs, T)
    ev = pipeline.simulate_batch(dict(wl, B=2), 0)
    n, df = wl["N"] // 2, fs / wl["N"]
    th = workloads.random_theta(91, S, wl["prior"])
    k_lo = math.ceil(wl["f_lo"] / df)
    edges = [e for m in range(1, 8) for e in (m * n // 16 - 1, m * n // 16)] + [k_lo - 1, n - 1]
    for s in range(S):
        last = edges[(s + 2) % len(edges)]
        total = 1.0 / (6.0 ** 1.5 * math.pi * C.MTSUN_S * df * (last + 0.5))   # f_isco half a bin past `last`
        th[C.M1, s], th[C.M2, s] = 0.55 * total, 0.45 * total
    offs = np.array([0, S // 2, S])
    args = (wl["seg_len"], wl["fs"], wl["f_lo"])
    y = ev["y"].astype(np.float32)
    ref = likelihood.log_likelihood_tmarg(y.astype(np.float64), ev["psd"], *args, th, offs, wl["dets"], 0.5 * T, n_tc, u)
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    got = gwx.log_likelihood_tmarg(cuda(y), cuda(ev["psd"]), *args, wl["dets"], 0.0, 0.5 * T, n_tc, u, cuda(th),
                                   cuda(offs)).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-3
