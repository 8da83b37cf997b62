"""The work this framework is run for, as measurable cases: simulated training batches, the background they
are drawn on, whitening of caller strain, the likelihoods that judge posterior samples, the flow that draws
them and the networks it is trained through.

A case is a dict of plain values with a "kind"; prepare() makes what a program holds before the call, run()
makes one pass through the public entry points, exact() restates the pass in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

import paper_2407_19048_gb300 as gwx
from paper_2407_19048_gb300.flow import FlowPosterior
from paper_2407_19048_gb300.resnet import ResNet1D

DETS = ("H1", "L1", "V1")
F_LO = 20.0

# (masses, spins, distance) boxes of the repository's workloads: "small" and "sweep" share the first, "hl3" has
# the second, the learned part the third
PRIORS = {"small": ((10.0, 50.0), (-0.5, 0.5), (200.0, 2000.0)),
          "hl3": ((5.0, 100.0), (-0.99, 0.99), (100.0, 3000.0)),
          "nonspinning": ((10.0, 50.0), (0.0, 0.0), (200.0, 2000.0))}


def listed():
    return [
        # a training batch of the two-detector 2 s workload at its own 64 draws: all launch latency
        {"name": "simulate_64x2x2s", "kind": "simulate", "prior": "small", "fs": 1024, "T": 2, "D": 2, "B": 64,
         "seconds": 16, "seg": 1},
        # the three-detector 4 s workload's batch, an ordinary training step's data
        {"name": "simulate_2048x3x4s", "kind": "simulate", "prior": "hl3", "fs": 2048, "T": 4, "D": 3, "B": 2048,
         "seconds": 64, "seg": 2},
        # the throughput sweep's batch, the largest window and the headline of the benchmark
        {"name": "simulate_8192x3x8s", "kind": "simulate", "prior": "small", "fs": 2048, "T": 8, "D": 3, "B": 8192,
         "seconds": 128, "seg": 2},
        # a fresh background chunk and its power spectrum, made once every few batches
        {"name": "background_3x64s", "kind": "background", "fs": 2048, "D": 3, "seconds": 64, "seg": 2},
        # strain that a program brings along (recorded windows), whitened; an odd number of windows
        {"name": "whiten_1001x3x4s", "kind": "whiten", "fs": 2048, "T": 4, "D": 3, "B": 1001, "seconds": 64, "seg": 2},
        # the likelihood of 64 events' samples, uneven counts, three detectors
        {"name": "loglike_64_events", "kind": "loglike", "prior": "hl3", "fs": 2048, "T": 4, "D": 3, "E": 64,
         "lo": 2000, "hi": 50000, "counts": 9, "seconds": 64, "seg": 2},
        # the importance-sampling judge: merger time integrated out, 64 events, uneven counts
        {"name": "tmarg_64_events", "kind": "tmarg", "prior": "nonspinning", "fs": 1024, "T": 2, "D": 2, "E": 64,
         "lo": 2000, "hi": 50000, "counts": 9, "u": 16, "seconds": 16, "seg": 1},
        # one event of a stream with a few thousand samples: the latency of the judge
        {"name": "tmarg_1_event", "kind": "tmarg", "prior": "nonspinning", "fs": 1024, "T": 2, "D": 2, "E": 1,
         "lo": 7001, "hi": 7001, "counts": 1, "u": 16, "seconds": 16, "seg": 1},
        # 20,000 posterior draws of one event, the paper's inference
        {"name": "posterior_20000", "kind": "posterior", "fs": 1024, "T": 2, "D": 2, "E": 1, "S": 20000, "layers": 16,
         "hidden": 256, "seconds": 16, "seg": 1},
        # loss and gradients of the flow on a training batch (forward and backward of the whole estimator)
        {"name": "flow_gradients_4096", "kind": "flow", "fs": 1024, "T": 2, "D": 2, "B": 4096, "layers": 16,
         "hidden": 256, "seconds": 16, "seg": 1},
        # the ResNet-1D summary's stem, a 64-channel block and a strided 128-channel block, forward and backward
        {"name": "resnet_blocks_512", "kind": "resnet", "B": 512, "D": 2, "N": 2048, "stages": "64x1,128x1/2",
         "out": 64},
        # the embedding's first dense layer, forward and backward
        {"name": "dense_4096x1968x512", "kind": "dense", "M": 4096, "K": 1968, "N": 512, "act": "relu"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate", "simulate", "simulate", "background", "whiten", "loglike", "tmarg", "tmarg",
                       "posterior", "flow", "resnet", "dense"])
    fs = rng.choice([1024, 2048])
    if kind == "simulate":
        T, D = rng.choice([2, 4, 8]), rng.randint(1, 3)
        N = fs * T
        B = min(_log_int(rng, 1, 8192), (8192 * 3 * 16384) // (D * N))
        return {"kind": kind, "prior": rng.choice(["small", "hl3"]), "fs": fs, "T": T, "D": D, "B": B,
                "seconds": rng.choice([16, 64, 128]), "seg": rng.choice([1, 2])}
    if kind == "background":
        return {"kind": kind, "fs": fs, "D": rng.randint(1, 3), "seconds": rng.choice([16, 32, 64, 128]),
                "seg": rng.choice([1, 2])}
    if kind == "whiten":
        return {"kind": kind, "fs": fs, "T": rng.choice([2, 4, 8]), "D": rng.randint(1, 3), "B": _log_int(rng, 1, 2048),
                "seconds": 64, "seg": rng.choice([1, 2])}
    if kind == "loglike":
        lo = _log_int(rng, 100, 5000)
        return {"kind": kind, "prior": rng.choice(["small", "hl3"]), "fs": fs, "T": rng.choice([2, 4, 8]),
                "D": rng.randint(1, 3), "E": _log_int(rng, 1, 64), "lo": lo, "hi": lo * rng.randint(1, 10),
                "counts": rng.randint(1, 10000), "seconds": 64, "seg": rng.choice([1, 2])}
    if kind == "tmarg":
        lo = _log_int(rng, 100, 5000)
        return {"kind": kind, "prior": rng.choice(["small", "nonspinning"]), "fs": 1024, "T": rng.choice([2, 4]),
                "D": rng.randint(2, 3), "E": _log_int(rng, 1, 16), "lo": lo, "hi": lo * rng.randint(1, 4),
                "counts": rng.randint(1, 10000), "u": rng.choice([4, 8, 16]), "seconds": 16, "seg": 1}
    if kind == "posterior":
        E = _log_int(rng, 1, 32)
        return {"kind": kind, "fs": 1024, "T": 2, "D": rng.randint(1, 3), "E": E, "S": _log_int(rng, max(E, 500), 200000),
                "layers": rng.choice([8, 16]), "hidden": rng.choice([128, 256]), "seconds": 16, "seg": 1}
    if kind == "flow":
        return {"kind": kind, "fs": 1024, "T": 2, "D": rng.randint(1, 3), "B": 8 * _log_int(rng, 8, 512),
                "layers": rng.choice([8, 16]), "hidden": rng.choice([128, 256]), "seconds": 16, "seg": 1}
    if kind == "resnet":
        return {"kind": kind, "B": 8 * _log_int(rng, 2, 64), "D": rng.randint(1, 3), "N": rng.choice([2048, 4096]),
                "stages": rng.choice(["64x1", "64x1,128x1/2", "64x2"]), "out": 64}
    return {"kind": "dense", "M": 8 * _log_int(rng, 16, 1024), "K": 8 * _log_int(rng, 9, 256),
            "N": 8 * _log_int(rng, 4, 128), "act": rng.choice(["none", "relu"])}


# ---------------------------------------------------------------- what a program holds

def _prior(case):
    m, chi, d = PRIORS[case.get("prior", "nonspinning")]
    T = float(case["T"])
    return {"m_lo": m[0], "m_hi": m[1], "chi_lo": chi[0], "chi_hi": chi[1], "d_lo": d[0], "d_hi": d[1],
            "tc_lo": 0.5 * T, "tc_hi": 0.75 * T, "phi_lo": 0.0, "phi_hi": 2.0 * math.pi, "psi_lo": 0.0,
            "psi_hi": 2.0 * math.pi}


def _sizes(case):
    """(window samples, background samples, Welch segment length)"""
    fs = case["fs"]
    return fs * case.get("T", 0), fs * case["seconds"], fs * case["seg"]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 1000003)


def _psd_aligo(f):
    x = f / 215.0
    return 1e-49 * (x ** -4.14 - 5.0 * x ** -2 + 111.0 * (1.0 - x ** 2 + 0.5 * x ** 4) / (1.0 + 0.5 * x ** 2))


def _strain(seed, rows, L, fs):
    """Gaussian strain [rows][L] (float32) coloured by the analytic aLIGO spectrum, flat below 20 Hz."""
    f = torch.arange(L // 2 + 1, device="cuda", dtype=torch.float64) * (fs / L)
    s = torch.sqrt(L * fs * _psd_aligo(f.clamp(min=F_LO)) / 4.0)
    g = _gen(seed)
    out = torch.empty((rows, L), dtype=torch.float32, device="cuda")
    for i in range(0, rows, 256):
        n = min(256, rows - i)
        x = torch.randn((n, L // 2 + 1, 2), generator=g, device="cuda").double() * s[:, None]
        out[i:i + n] = torch.fft.irfft(torch.view_as_complex(x), n=L).float()
    return out


def _background(case, seed):
    """(strain [D][L], its power spectrum), as a program keeps them from its data."""
    _, L, M = _sizes(case)
    noise = _strain(seed, case["D"], L, case["fs"])
    return noise, gwx.welch_psd(noise, float(case["fs"]), M, M // 2)


def _batch(case, seed, B, prior=None):
    """Simulated whitened windows [B][D][N] and their parameters."""
    N, _, M = _sizes(case)
    noise, psd = _background(case, seed)
    y, theta, _ = gwx.simulate_batch(prior or _prior(case), seed, 0, noise, psd, M, float(case["fs"]), F_LO,
                                     DETS[:case["D"]], 0.0, B, N)
    return y, theta, psd


def _counts(case):
    return np.random.default_rng(case["counts"]).integers(case["lo"], case["hi"] + 1, case["E"]).astype(np.int64)


def _n_tc(case):
    return int(0.25 * case["T"] * case["fs"])


def _workload(case):
    N, L, M = _sizes(case)
    return {"name": "learned", "B": case.get("B", 512), "dets": DETS[:case["D"]], "fs": float(case["fs"]),
            "T": float(case["T"]), "N": N, "L": L, "seg_len": M, "seg_stride": M // 2, "f_lo": F_LO, "gmst": 0.0,
            "param_seed": 1, "noise_seed": 2, "prior": _prior(case)}


def _flow(case, seed):
    """A flow with weights as a trained one has them: every layer moves its coordinates."""
    fl = FlowPosterior(_workload(case), layers=case["layers"], hidden=case["hidden"], seed=seed)
    g = _gen(seed + 1)
    arrays = []
    for t, s in enumerate(fl.tensor_shapes()):
        if len(s) == 2:
            gain = 0.3 if (t >= 6 and t % 6 == 4) else 1.0
            arrays.append(torch.randn(s, generator=g, device="cuda") * (gain / math.sqrt(s[1])))
        else:
            arrays.append(torch.randn(s, generator=g, device="cuda") * 0.1)
    fl.set_tensors(arrays)
    return fl


def _stages(case):
    out = []
    for part in case["stages"].split(","):
        head, _, s = part.partition("/")
        c, n = head.split("x")
        out.append((int(c), int(n), int(s or 1)))
    return tuple(out)


ACTS = {"none": gwx.ACT_NONE, "relu": gwx.ACT_RELU}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": int(seed)}
    if kind == "background":
        return st
    if kind == "resnet":
        net = ResNet1D(case["D"], case["out"], stages=_stages(case), seed=seed)
        g = _gen(seed)
        st.update(net=net, y=torch.randn((case["B"], case["D"], case["N"]), generator=g, device="cuda"),
                  dc=torch.randn((case["B"], case["out"]), generator=g, device="cuda") / case["B"])
        return st
    if kind == "dense":
        g = _gen(seed)
        M, N, K = case["M"], case["N"], case["K"]

        def r(*s):
            return torch.randn(s, generator=g, device="cuda")

        st.update(X=r(M, K).bfloat16(), W=(r(N, K) / math.sqrt(K)).bfloat16(), b=0.1 * r(N), dY=r(M, N) / M)
        return st
    N, L, M = _sizes(case)
    if kind == "simulate":
        noise, psd = _background(case, seed)
        st.update(noise=noise, psd=psd, prior=_prior(case), bufs=gwx.SimulateBuffers(case["B"], case["D"], N))
    elif kind == "whiten":
        _, psd = _background(case, seed)
        d = _strain(seed + 7, case["B"] * case["D"], N, case["fs"]).view(case["B"], case["D"], N)
        st.update(d=d, psd=psd)
    elif kind in ("loglike", "tmarg"):
        y, truth, psd = _batch(case, seed, case["E"])
        c = _counts(case)
        offs = torch.from_numpy(np.concatenate([[0], np.cumsum(c)])).cuda()
        S = int(c.sum())
        theta, _ = gwx.sample_prior(_prior(case), seed + 5, 1, S, L, N)
        # every other sample lies near its event's source, as a posterior's samples do
        ev = torch.repeat_interleave(torch.arange(case["E"], device="cuda"), torch.from_numpy(c).cuda())
        near = torch.arange(S, device="cuda") % 2 == 1
        g = _gen(seed + 3)
        for p, w in ((0, 0.01), (1, 0.01), (4, 0.1), (7, 0.05), (9, 0.02), (10, 0.02), (5, 0.0), (2, 0.0), (3, 0.0)):
            t = truth[p][ev] * (1.0 + w * torch.randn(S, generator=g, device="cuda", dtype=torch.float64))
            theta[p] = torch.where(near, t, theta[p])
        st.update(y=y, psd=psd, theta=theta.contiguous(), offs=offs)
    elif kind == "posterior":
        y, _, _ = _batch(case, seed, case["E"])
        cuts = np.sort(np.random.default_rng(seed).integers(0, case["S"] + 1, case["E"] - 1))
        offs = torch.from_numpy(np.concatenate([[0], cuts, [case["S"]]]).astype(np.int64)).cuda()
        st.update(y=y, offs=offs, flow=_flow(case, seed))
    elif kind == "flow":
        y, theta, _ = _batch(case, seed, case["B"])
        st.update(y=y, theta=theta, flow=_flow(case, seed))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "resnet":
        c = st["net"].forward(st["y"])
        return {"c": c, "grads": st["net"].backward(st["dc"])}
    if kind == "dense":
        act = ACTS[case["act"]]
        Y = gwx.dense_bf16(st["X"], st["W"], st["b"], act, out_dtype=torch.bfloat16)
        dX, dW, db = gwx.dense_bf16_backward(st["X"], st["W"], st["b"], st["dY"], act)
        return {"Y": Y, "dX": dX, "dW": dW, "db": db}
    N, L, M = _sizes(case)
    fs, dets = float(case["fs"]), DETS[:case["D"]]
    if kind == "background":
        n = gwx.colored_noise(st["seed"], 3, case["D"], L, fs, F_LO)
        return {"noise": n, "psd": gwx.welch_psd(n, fs, M, M // 2)}
    if kind == "simulate":
        y, theta, offsets = gwx.simulate_batch(st["prior"], st["seed"], 3, st["noise"], st["psd"], M, fs, F_LO, dets,
                                               0.0, case["B"], N, buffers=st["bufs"])
        return {"y": y, "theta": theta, "offsets": offsets}
    if kind == "whiten":
        return {"y": gwx.whiten(st["d"], st["psd"], M, fs, F_LO)}
    if kind == "loglike":
        return {"lnl": gwx.log_likelihood(st["y"], st["psd"], M, fs, F_LO, dets, 0.0, st["theta"], st["offs"])}
    if kind == "tmarg":
        return {"lnl": gwx.log_likelihood_tmarg(st["y"], st["psd"], M, fs, F_LO, dets, 0.0, 0.5 * case["T"],
                                                _n_tc(case), case["u"], st["theta"], st["offs"])}
    if kind == "posterior":
        theta, log_q, log_ratio = st["flow"].sample(st["y"], st["offs"], st["seed"], 4, S=case["S"])
        return {"theta": theta, "log_q": log_q, "log_ratio": log_ratio}
    loss = st["flow"].train_step(st["y"], st["theta"], update=False)
    return {"loss": loss, "grads": st["flow"].grads}


# ---------------------------------------------------------------- what a pass cannot do without

def _mean_bins(case):
    """Mean number of waveform bins of a draw of the case's prior."""
    (lo, hi), _, _ = PRIORS[case.get("prior", "nonspinning")]
    m = np.random.default_rng(0).uniform(lo, hi, (2, 4096)).sum(axis=0)
    k = np.minimum(1.0 / (6.0 ** 1.5 * math.pi * m * 4.925490947641267e-6), case["fs"] / 2) - F_LO
    return float(np.maximum(k, 0.0).mean() * case["T"])


def _flow_flops(case):
    C, H, K = 64, case["hidden"], case["layers"]
    return 2.0 * K * ((8 + C) * H + H * H + 8 * H)


def work(case):
    kind = case["kind"]
    if kind == "dense":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * M * K + 2 * N * K + 4 * N + 2 * M * N + 4 * M * N + 4 * M * K + 4 * N * K + 4 * N,
                "flops": 6.0 * M * N * K}
    if kind == "resnet":
        B, N = case["B"], case["N"]
        T, cin = N // 2, _stages(case)[0][0]
        flops, params = 6.0 * B * T * 7 * case["D"] * cin, 7 * case["D"] * cin
        T //= 2
        for c, n, s in _stages(case):
            for i in range(n):
                T = T // s if i == 0 else T
                w = 5 * cin * c + 5 * c * c + (cin * c if i == 0 and (s > 1 or cin != c) else 0)
                flops += 6.0 * B * T * w
                params += w
                cin = c
        return {"bytes": 4 * B * case["D"] * N + 8 * B * case["out"] + 6 * params, "flops": flops}
    N, L, M = _sizes(case)
    D = case["D"]
    if kind == "background":
        segs = 2 * (L // M) - 1
        return {"bytes": 4 * D * L + 8 * D * (M // 2 + 1),
                "flops": D * (2.5 * L * math.log2(L) + 15.0 * L + segs * (2.5 * M * math.log2(M) + 3.0 * M))}
    fft = 2.5 * N * math.log2(N)
    if kind == "simulate":
        return {"bytes": 4 * case["B"] * D * N + 8 * D * (M // 2 + 1) + 4 * D * L + 96 * case["B"],
                "flops": case["B"] * (D * (2 * fft + 3.0 * N) + _mean_bins(case) * (150 + 60 * D))}
    if kind == "whiten":
        return {"bytes": 8 * case["B"] * D * N + 8 * D * (M // 2 + 1), "flops": case["B"] * D * (2 * fft + 3.0 * N)}
    if kind in ("loglike", "tmarg"):
        S = float(_counts(case).sum())
        per = _mean_bins(case) * (150 + 60 * D)
        if kind == "tmarg":
            J = case["u"] * _n_tc(case)
            per += 2.5 * J * math.log2(J) + 4.0 * J
        return {"bytes": 4 * case["E"] * D * N + 96 * S, "flops": S * per + case["E"] * D * fft}
    if kind == "posterior":
        return {"bytes": 4 * case["E"] * D * N + 13 * 8 * case["S"], "flops": case["S"] * (_flow_flops(case) + 300)}
    k_lo = math.ceil(F_LO * N / case["fs"])
    F = D * ((N // 2 - k_lo) // 4) * (1 + (D - 1) + 2)
    embed = 2.0 * (F * 512 + 512 * 512 + 512 * 64)
    return {"bytes": 4 * case["B"] * D * N + 88 * case["B"] + 6 * (_flow_flops(case) + embed) / 2,
            "flops": case["B"] * (3 * (_flow_flops(case) + embed) + D * fft)}


# ---------------------------------------------------------------- the same in 64 bits

F64, I64 = torch.float64, torch.int64
MASK = 0xFFFFFFFF


def _philox(c, k0, k1):
    """Ten Philox4x32 rounds on four int64 tensors holding 32-bit words."""
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & MASK) ^ c[1] ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c[3] ^ k1, p0 & MASK]
    return c


def _words(index, block, tag, step, seed):
    z = torch.zeros_like(index)
    return _philox([index & MASK, z + block, z + tag, z + (step & MASK)], seed & MASK, (seed >> 32) & MASK)


def _uniform52(hi, lo):
    return (((hi << 20) | (lo >> 12)).to(F64) + 0.5) * 2.0 ** -52


def _arange(n, dtype=F64):
    return torch.arange(n, device="cuda", dtype=dtype)


def _prior_draws(p, seed, step, B, L, N):
    i = _arange(B, I64)
    u = []
    for j in range(6):
        w = _words(i, j, 1, step, seed)
        u += [_uniform52(w[0], w[1])] + ([_uniform52(w[2], w[3])] if j < 5 else [])
    off = (w[2] * (L - N + 1)) >> 32
    lin = lambda a, b, x: p[a] + (p[b] - p[a]) * x  # noqa: E731
    th = torch.stack([lin("m_lo", "m_hi", u[0]), lin("m_lo", "m_hi", u[1]), lin("chi_lo", "chi_hi", u[2]),
                      lin("chi_lo", "chi_hi", u[3]), lin("d_lo", "d_hi", u[4]), lin("tc_lo", "tc_hi", u[5]),
                      lin("phi_lo", "phi_hi", u[6]), torch.arccos(1.0 - 2.0 * u[7]), lin("psi_lo", "psi_hi", u[8]),
                      2.0 * math.pi * u[9], torch.arcsin(2.0 * u[10] - 1.0)])
    return th, off


SITES = ((46.455147, -119.407657, 142.554, 324.0, 234.0), (30.562894, -90.774240, -6.574, 252.2835, 162.2835),
         (43.631415, 10.504497, 51.884, 19.4326, 289.4326))


def _site(d):
    lat, lon, h, xaz, yaz = SITES[d]
    phi, lam = math.radians(lat), math.radians(lon)
    north = np.array([-math.sin(phi) * math.cos(lam), -math.sin(phi) * math.sin(lam), math.cos(phi)])
    east = np.array([-math.sin(lam), math.cos(lam), 0.0])
    x, y = (math.cos(math.radians(a)) * north + math.sin(math.radians(a)) * east for a in (xaz, yaz))
    f = 1.0 / 298.257223563
    e2 = f * (2.0 - f)
    n = 6378137.0 / math.sqrt(1.0 - e2 * math.sin(phi) ** 2)
    r = np.array([(n + h) * math.cos(phi) * math.cos(lam), (n + h) * math.cos(phi) * math.sin(lam),
                  (n * (1.0 - e2) + h) * math.sin(phi)])
    return torch.from_numpy(0.5 * (np.outer(x, x) - np.outer(y, y))).cuda(), torch.from_numpy(r).cuda()


MTSUN = 4.925490947641267e-6


def _last_bin(th, df):
    return torch.floor(1.0 / (6.0 ** 1.5 * math.pi * (th[0] + th[1]) * MTSUN) / df)


def _templates(th, fs, N, D, K, tc=None):
    """fs h_d on bins 0 .. K-1 of the window's grid, complex128 [S][D][K]: TaylorF2 3.5PN with the 1.5PN
    spin-orbit term, f_isco cut, projected and shifted by tc + dt_d."""
    df, pi = fs / N, math.pi
    m1, m2, chi1, chi2, dist, tc0, phic, iota, psi, ra, dec = th
    M, eta, delta = (m1 + m2) * MTSUN, m1 * m2 / (m1 + m2) ** 2, (m1 - m2) / (m1 + m2)
    cs, ca = 0.5 * (chi1 + chi2), 0.5 * (chi1 - chi2)
    k = _arange(K)
    f = (k * df).clamp(min=df)
    v = (pi * M[:, None] * f) ** (1.0 / 3.0)
    lv = torch.log(v)
    g = 0.5772156649015329
    col = lambda x: x[:, None]  # noqa: E731
    s = 1.0 + col(3715.0 / 756.0 + 55.0 * eta / 9.0) * v ** 2
    s = s + col(-16.0 * pi + 113.0 / 3.0 * delta * ca + (113.0 / 3.0 - 76.0 * eta / 3.0) * cs) * v ** 3
    s = s + col(15293365.0 / 508032.0 + 27145.0 * eta / 504.0 + 3085.0 * eta ** 2 / 72.0) * v ** 4
    s = s + col(pi * (38645.0 / 756.0 - 65.0 * eta / 9.0)) * (1.0 + 3.0 * lv) * v ** 5
    a6 = (11583231236531.0 / 4694215680.0 - 640.0 * pi ** 2 / 3.0 - 6848.0 * g / 21.0 - 6848.0 * math.log(4.0) / 21.0
          + (-15737765635.0 / 3048192.0 + 2255.0 * pi ** 2 / 12.0) * eta + 76055.0 * eta ** 2 / 1728.0
          - 127825.0 * eta ** 3 / 1296.0)
    s = s + (col(a6) - 6848.0 / 21.0 * lv) * v ** 6
    s = s + col(pi * (77096675.0 / 254016.0 + 378515.0 * eta / 1512.0 - 74045.0 * eta ** 2 / 756.0)) * v ** 7
    ph = -col(phic) - pi / 4.0 + 3.0 / (128.0 * col(eta)) * v ** -5 * s
    amp = (math.sqrt(5.0 / 24.0) * pi ** (-2.0 / 3.0)
           * col((M * eta ** 0.6) ** (5.0 / 6.0) / (dist * 3.085677581491367e22 / 299792458.0)) * f ** (-7.0 / 6.0))
    on = (k >= math.ceil(F_LO / df)) & (k <= col(_last_bin(th, df)))
    base = torch.polar(torch.where(on, fs * amp, torch.zeros_like(amp)), -ph)
    ci = torch.cos(iota)
    sd, cd, sp, cp = torch.sin(dec), torch.cos(dec), torch.sin(ra), torch.cos(ra)
    n = torch.stack([cd * cp, cd * sp, sd])
    eth, eph = torch.stack([sd * cp, sd * sp, -cd]), torch.stack([-sp, cp, torch.zeros_like(sp)])
    X, Y = torch.cos(psi) * eth + torch.sin(psi) * eph, torch.sin(psi) * eth - torch.cos(psi) * eph
    t0 = tc0 if tc is None else torch.full_like(tc0, tc)
    out = torch.empty((th.shape[1], D, K), dtype=torch.complex128, device="cuda")
    for d in range(D):
        T, r = _site(d)
        fp = (X * (T @ X)).sum(0) - (Y * (T @ Y)).sum(0)
        fc = (X * (T @ Y)).sum(0) + (Y * (T @ X)).sum(0)
        x = col(t0 - (r @ n) / 299792458.0) * (df * k)
        shift = torch.polar(torch.ones_like(x), -2.0 * pi * (x - torch.round(x)))
        out[:, d] = base * col(torch.complex(fp * 0.5 * (1.0 + ci ** 2), -fc * ci)) * shift
    return out


def _filter(psd, M, fs, N):
    """Whitening filter [D][N/2+1]."""
    k = _arange(N // 2 + 1, I64)
    j0, fr = (k * M) // N, ((k * M) % N).to(F64) / N
    s = psd[:, j0] + (psd[:, (j0 + 1).clamp(max=M // 2)] - psd[:, j0]) * fr
    on = (k >= math.ceil(F_LO / (fs / N))) & (k < N // 2)
    return torch.where(on, 1.0 / torch.sqrt(s * fs / 2.0), torch.zeros_like(s))


def _exact_simulate(case, st):
    N, L, M = _sizes(case)
    B, D, fs = case["B"], case["D"], float(case["fs"])
    th, off = _prior_draws(st["prior"], st["seed"], 3, B, L, N)
    W, K = _filter(st["psd"], M, fs, N), N // 2 + 1
    noise = st["noise"].double()
    y = torch.empty((B, D, N), dtype=F64, device="cuda")
    step = max(1, (1 << 22) // N)
    for i in range(0, B, step):
        j = min(B, i + step)
        d = noise[:, off[i:j, None] + _arange(N, I64)].transpose(0, 1)
        X = torch.fft.rfft(d)
        kk = min(K, int(_last_bin(th[:, i:j], fs / N).max().item()) + 1)
        X[..., :kk] += _templates(th[:, i:j], fs, N, D, kk)
        y[i:j] = torch.fft.irfft(X * W, n=N)
    return {"y": y, "theta": th, "offsets": None}


def _exact_background(case, st):
    _, L, M = _sizes(case)
    D, fs = case["D"], float(case["fs"])
    K = L // 2 + 1
    j = _arange((K + 1) // 2, I64)
    f = _arange(K) * fs / L
    sig = torch.sqrt(L * fs * _psd_aligo(f.clamp(min=F_LO)) / 4.0)
    n = torch.empty((D, L), dtype=F64, device="cuda")
    u24 = lambda w: ((w >> 8).to(F64) + 0.5) * 2.0 ** -24  # noqa: E731
    for d in range(D):
        w = _words(j, d, 2, 3, st["seed"])
        g = []
        for a, b in ((w[0], w[1]), (w[2], w[3])):
            r, t = torch.sqrt(-2.0 * torch.log(u24(a))), 2.0 * math.pi * u24(b)
            g.append(torch.complex(r * torch.cos(t), r * torch.sin(t)))
        X = torch.stack(g, 1).reshape(-1)[:K] * sig
        X[0] = 0.0
        X[-1] = X[-1].real * math.sqrt(2.0)
        n[d] = torch.fft.irfft(X, n=L)
    w = 0.5 - 0.5 * torch.cos(2.0 * math.pi * _arange(M) / M)
    P = (torch.fft.rfft(n.unfold(1, M, M // 2) * w).abs() ** 2).mean(1) / (fs * (w * w).sum())
    P[:, 1:-1] *= 2.0
    return {"noise": n, "psd": P}


def _exact_lnl(case, st):
    N, _, M = _sizes(case)
    E, D, fs = case["E"], case["D"], float(case["fs"])
    W, df = _filter(st["psd"], M, fs, N), fs / N
    Y = torch.fft.rfft(st["y"].double())
    band = W[0] > 0
    yy = (Y[..., band].abs() ** 2).sum((1, 2))
    th, S = st["theta"], st["theta"].shape[1]
    ev = torch.bucketize(_arange(S, I64), st["offs"], right=True).clamp(max=E) - 1
    last = _last_bin(th, df).clamp(max=N // 2 - 1)
    order = torch.argsort(last)
    out = torch.empty(S, dtype=F64, device="cuda")
    tm = case["kind"] == "tmarg"
    tc_lo, J, u = 0.5 * case["T"], case.get("u", 1) * _n_tc(case), case.get("u", 1)
    i = 0
    while i < S:
        j = min(S, i + 4096)
        K = int(last[order[j - 1]].item()) + 1
        at = order[i:j]
        G = _templates(th[:, at], fs, N, D, K, tc_lo if tm else None) * W[:, :K]
        Ye = Y[ev[at], :, :K]
        if tm:
            c = (Ye * G.conj()).sum(1) * (2.0 / N)
            base = -(yy[ev[at]] + (G.abs() ** 2).sum((1, 2))) / N
            z = torch.fft.irfft(c, n=N * u)[:, :J] * (0.5 * N * u)
            out[at] = base + torch.logsumexp(z, 1) - math.log(J)
        else:
            out[at] = -(yy[ev[at]] + (G.abs() ** 2 - 2.0 * (Ye.conj() * G).real).sum((1, 2))) / N
        i = j
    return {"lnl": out}


def _features(y, fs, F):
    """Log group powers, cross spectra and lag-one products of whitened windows, in the flow's column order."""
    B, D, N = y.shape
    Y = torch.fft.rfft(y)
    k_lo, G = math.ceil(F_LO * N / fs), 4
    ng = (N // 2 - k_lo) // G
    a, b = (Y[..., k_lo + o:k_lo + o + ng * G].reshape(B, D, ng, G) for o in (0, 1))
    pw = lambda x: (x.abs() ** 2).sum(-1)  # noqa: E731
    cols = [torch.log(pw(a) / (G * N)).reshape(B, -1)]
    for i in range(D):
        for j in range(i + 1, D):
            r = (a[:, i] * a[:, j].conj()).sum(-1) / torch.sqrt(pw(a[:, i]) * pw(a[:, j]))
            cols += [r.real, r.imag]
    for i in range(D):
        r = (a[:, i] * b[:, i].conj()).sum(-1) / torch.sqrt(pw(a[:, i]) * pw(b[:, i]))
        cols += [r.real, r.imag]
    f = torch.cat(cols, 1)
    return torch.cat([f, f.new_zeros(B, F - f.shape[1])], 1)


SPLITS = (((0, 1, 2, 3), (4, 5, 6, 7)), ((4, 5, 6, 7), (0, 1, 2, 3)), ((0, 2, 4, 6), (1, 3, 5, 7)),
          ((1, 3, 5, 7), (0, 2, 4, 6)))


def _tensors(fl):
    """The flow's parameters as the products use them (weights from the bfloat16 copy), in 64 bits."""
    return [fl.tensor(t, bf16=len(s) == 2).double() for t, s in enumerate(fl.tensor_shapes())]


def _net(x, w):
    h = torch.relu(x @ w[0].T + w[1])
    h = torch.relu(h @ w[2].T + w[3])
    return h @ w[4].T + w[5]


def _coupling(v, c, w, l, sampling):
    a, b = SPLITS[l % 4]
    o = _net(torch.cat([v[:, a], torch.zeros_like(v[:, a]), c], 1), w)
    s = 3.0 * torch.tanh(o[:, 4:] / 3.0)
    out = v.clone()
    out[:, b] = v[:, b] * torch.exp(s) + o[:, :4] if sampling else (v[:, b] - o[:, :4]) * torch.exp(-s)
    return out, s.sum(1)


def _coords(th):
    m1, m2 = th[0], th[1]
    mc = (m1 * m2) ** 0.6 / (m1 + m2) ** 0.2
    return torch.stack([mc, torch.minimum(m1, m2) / torch.maximum(m1, m2), th[4], torch.cos(th[7]), th[9],
                        torch.sin(th[10]), th[8], th[6]], 1)


def _exact_flow(case, st):
    fl = st["flow"]
    ts = [t.clone().requires_grad_(True) for t in _tensors(fl)]
    f = _features(st["y"].double(), float(case["fs"]), fl.shape["features"])
    mean, scale = (torch.tensor(v, dtype=F64, device="cuda") for v in (fl.mean, fl.scale))
    v, c, tot = (_coords(st["theta"]) - mean) / scale, _net(f, ts[:6]), 0.0
    for l in reversed(range(case["layers"])):
        v, s = _coupling(v, c, ts[6 + 6 * l:12 + 6 * l], l, False)
        tot = tot + s
    loss = (0.5 * (v * v).sum(1) + 4.0 * math.log(2.0 * math.pi) + tot).mean()
    grads = torch.zeros(fl.n_params, dtype=F64, device="cuda")
    for g, o in zip(torch.autograd.grad(loss, ts), fl.offsets):
        grads[o:o + g.numel()] = g.reshape(-1)
    return {"loss": loss.detach().reshape(1), "grads": grads}


def _exact_posterior(case, st):
    fl, S, p = st["flow"], case["S"], _prior(case)
    ts, i = _tensors(fl), _arange(S, I64)
    u = []
    for j in range(6):
        w = _words(i, j, 4, 4, st["seed"])
        u += [_uniform52(w[0], w[1]), _uniform52(w[2], w[3])]
    z = []
    for j in range(4):
        r, t = torch.sqrt(-2.0 * torch.log(u[2 * j])), 2.0 * math.pi * u[2 * j + 1]
        z += [r * torch.cos(t), r * torch.sin(t)]
    z = torch.stack(z, 1)
    ev = torch.bucketize(i, st["offs"], right=True).clamp(max=case["E"]) - 1
    c = _net(_features(st["y"].double(), float(case["fs"]), fl.shape["features"]), ts[:6])[ev]
    v, tot = z, 0.0
    for l in range(case["layers"]):
        v, s = _coupling(v, c, ts[6 + 6 * l:12 + 6 * l], l, True)
        tot = tot + s
    mean, scale = (torch.tensor(x, dtype=F64, device="cuda") for x in (fl.mean, fl.scale))
    mc, q, dist, ct, ra, sd, psi, phi = (mean + scale * v).unbind(1)
    log_q = -0.5 * (z * z).sum(1) - 4.0 * math.log(2.0 * math.pi) - tot - torch.log(scale).sum()
    big = mc * (1.0 + q) ** 0.2 * q ** -0.6
    small = q * big
    ok = ((mc > 0) & (q > 0) & (q <= 1) & (small >= p["m_lo"]) & (big <= p["m_hi"]) & (dist >= p["d_lo"])
          & (dist <= p["d_hi"]) & (ct.abs() <= 1) & (ra >= 0) & (ra < 2.0 * math.pi) & (sd.abs() <= 1)
          & (psi >= p["psi_lo"]) & (psi <= p["psi_hi"]) & (phi >= p["phi_lo"]) & (phi <= p["phi_hi"]))
    lp = (math.log(2.0) + 2.0 * torch.log(big) - torch.log(mc) - 2.0 * math.log(p["m_hi"] - p["m_lo"])
          - math.log(p["d_hi"] - p["d_lo"]) - math.log(8.0 * math.pi) - math.log(p["psi_hi"] - p["psi_lo"])
          - math.log(p["phi_hi"] - p["phi_lo"]))
    swap = u[8] < 0.5
    lo = torch.full_like(mc, p["m_lo"])
    lin = lambda a, b, x: p[a] + (p[b] - p[a]) * x  # noqa: E731
    th = torch.stack([torch.where(ok, torch.where(swap, small, big), lo), torch.where(ok, torch.where(swap, big, small), lo),
                      lin("chi_lo", "chi_hi", u[10]), lin("chi_lo", "chi_hi", u[11]),
                      torch.where(ok, dist, torch.full_like(mc, p["d_lo"])), lin("tc_lo", "tc_hi", u[9]), phi,
                      torch.arccos(ct.clamp(-1, 1)), psi, ra, torch.arcsin(sd.clamp(-1, 1))])
    return {"theta": th, "log_q": log_q, "log_ratio": torch.where(ok, lp - log_q, torch.full_like(mc, -math.inf))}


def _exact_resnet(case, st):
    net, D = st["net"], case["D"]
    P = {}

    def leaf(name, x):
        P[name] = x.double().clone().requires_grad_(True)
        return P[name]

    def conv(x, W, k, s, pad):
        cin = x.shape[1]
        w = W[:, :k * cin].reshape(W.shape[0], k, cin).permute(0, 2, 1)
        cols = torch.nn.functional.pad(x, (pad, pad)).unfold(2, k, s)
        return torch.einsum("bctk,ock->bot", cols, w)

    def gn(x, g, b):
        return torch.nn.functional.group_norm(x, 8, g, b, 1e-5)

    named = {n: (w32 if w16 is None else w16) for n, w32, w16 in net.tensors()}
    L = {n: leaf(n, w) for n, w in named.items()}
    h = torch.relu(gn(conv(st["y"].double(), L["W0"], 7, 2, 3), L["g0"], L["b0"]))
    h = torch.nn.functional.max_pool1d(h, 3, 2, 1)
    i = 0
    for c, n, s in _stages(case):
        for b in range(n):
            q = "%d." % i
            s_ = s if b == 0 else 1
            o = torch.relu(gn(conv(h, L[q + "W1"], 5, s_, 2), L[q + "g1"], L[q + "b1"]))
            o = gn(conv(o, L[q + "W2"], 5, 1, 2), L[q + "g2"], L[q + "b2"])
            if q + "Wd" in L:
                h = gn(conv(h, L[q + "Wd"], 1, s_, 0), L[q + "gd"], L[q + "bd"])
            h = torch.relu(o + h)
            i += 1
    c = h.mean(2) @ L["Wf"].T + L["bf"]
    g = torch.autograd.grad(c, list(L.values()), st["dc"].double())
    return {"c": c.detach(), "grads": dict(zip(L.keys(), g))}


def _exact_dense(case, st):
    X, W, b = (st[k].double().requires_grad_(True) for k in ("X", "W", "b"))
    z = X @ W.T + b
    Y = torch.relu(z) if case["act"] == "relu" else z
    dX, dW, db = torch.autograd.grad(Y, (X, W, b), st["dY"].double())
    return {"Y": Y.detach(), "dX": dX, "dW": dW, "db": db}


def exact(case, seed):
    kind, st = case["kind"], prepare(case, seed)
    if kind == "whiten":
        N, _, M = _sizes(case)
        W = _filter(st["psd"], M, float(case["fs"]), N)
        return {"y": torch.fft.irfft(torch.fft.rfft(st["d"].double()) * W, n=N)}
    if kind in ("loglike", "tmarg"):
        return _exact_lnl(case, st)
    return {"simulate": _exact_simulate, "background": _exact_background, "posterior": _exact_posterior,
            "flow": _exact_flow, "resnet": _exact_resnet, "dense": _exact_dense}[kind](case, st)
