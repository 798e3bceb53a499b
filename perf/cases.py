"""Performance cases of the correlator: what a user's program asks of it, at the sizes it is used at.

Each case is one pass through the public binding (`paper_0906_1887_gb300.corr`) on device memory: the
X stage on packed 4/8-bit samples, on float samples (BF16x3 and FP32), the F stage and the polyphase
filterbank, the fused X + dump step, and a batch of uneven jobs.  The calls on host buffers
(`corr_xengine_run_host`, the serving loop) are these stages beside copies over the host link, so they
are stood for by the stages.  The FP32 engine on 4/8-bit samples is the plain form that the exact
tensor-core engine is compared with, not a path for earnest use, and has no case.

Sizes are those of the benchmark's workloads (the 32-antenna prototype dump, the 64-input stream, the
1024-input array, the uneven batch, the serving streams), or lie in the ranges they are drawn from.
"""
import math

import numpy as np
import torch

from paper_0906_1887_gb300 import corr

DEV = "cuda"

# ---- the listed cases ------------------------------------------------------------------------


def listed():
    return [
        # the paper's prototype: 32 dual-pol antennas, 128 channels, 512 samples, one dump of 4-bit
        # samples: the smallest call, where launches and latency count
        dict(name="proto_dump_4bit", kind="x", n=64, c=128, t=512, bits=4, dumps=1, acc=False),
        # the streamed correlator: 64 inputs, 768 channels, 1000 samples a dump, 8-bit, several dumps a call
        dict(name="stream64_8bit", kind="x", n=64, c=768, t=1000, bits=8, dumps=8, acc=False),
        # the large array: 512 dual-pol antennas, 1536 channels, 256 samples: 12.9 GB of visibilities a dump
        dict(name="array1024_8bit", kind="x", n=1024, c=1536, t=256, bits=8, dumps=1, acc=False),
        # a long dump of a 256-antenna array, the compute-heavy end of the uneven batch
        dict(name="long512_8bit", kind="x", n=512, c=128, t=2048, bits=8, dumps=1, acc=False),
        # one job of a serving stream: a 200-antenna array, 4-bit, added into its accumulators
        dict(name="serve400_4bit_acc", kind="x", n=400, c=613, t=472, bits=4, dumps=1, acc=True),
        # an array whose packed rows are no whole 16-byte pieces (75 inputs, odd channels and samples)
        dict(name="ragged75_8bit", kind="x", n=75, c=333, t=777, bits=8, dumps=2, acc=False),
        # the stream on float samples, as an F stage outside hands them over
        dict(name="stream64_bf16x3", kind="xf", n=64, c=768, t=1000, dumps=2, engine="bf16x3"),
        # float samples where BF16x3's 1e-5 is not enough
        dict(name="stream64_fp32", kind="xf", n=64, c=768, t=1000, dumps=1, engine="fp32"),
        # the prototype's whole chain on one second of data: 8-tap filterbank, then the X stage
        dict(name="fx_pfb8_proto", kind="fx", n=64, c=128, frames=10000, fkind="c8", taps=8),
        # F stage of real samples (voltages of a single-sideband receiver), long transforms
        dict(name="fstage_real8", kind="f", n=128, c=1024, frames=512, fkind="r8", taps=0),
        # X stage with the dump step fused: averaged and phase-corrected float32 straight from the samples
        dict(name="fused_dump256", kind="xd", n=256, c=512, t=500, bits=8),
        # sub-arrays of 16..256 dual-pol antennas in one tuned launch
        dict(name="batch15", kind="batch", jobs=15, sizes=4000),
    ]


# ---- drawn cases -----------------------------------------------------------------------------


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _inputs(rng, lo, hi):
    """Arrays come in all sizes; most have rows that are whole 16-byte pieces."""
    n = _logint(rng, lo, hi)
    return min(hi, (n + 15) // 16 * 16) if rng.random() < 0.6 else n


def _fit(case, key, max_bytes, max_flops):
    """The case with `key` (channels, frames) cut until it costs no more than the largest listed one."""
    while True:
        w = work(case)
        over = max(w["bytes"] / max_bytes, w["flops"] / max_flops)
        if over <= 1.0 or case[key] <= 1:
            return case
        case[key] = max(1, int(case[key] / over * 0.98))


def draw(rng):
    kind = rng.choices(["x", "xf", "fx", "f", "xd", "batch"], [10, 3, 1, 2, 2, 1])[0]
    if kind == "x":
        c = dict(kind="x", n=_inputs(rng, 8, 1024), c=_logint(rng, 64, 1536), t=_logint(rng, 64, 2048),
                 bits=rng.choice([4, 8]), dumps=rng.randint(1, 4), acc=rng.random() < 0.3)
        return _fit(c, "c", 8e9, 8e11)
    if kind == "xf":
        c = dict(kind="xf", n=_inputs(rng, 8, 256), c=_logint(rng, 64, 1024), t=_logint(rng, 100, 2000),
                 dumps=rng.randint(1, 3), engine=rng.choice(["bf16x3", "bf16x3", "fp32"]))
        return _fit(c, "c", 4e9, 5e10)
    if kind == "fx":
        fk = rng.choice(["c8", "c4", "r8"])
        c = dict(kind="fx", n=_inputs(rng, 8, 128), c=rng.choice([64, 128, 256]), frames=_logint(rng, 1000, 10000),
                 fkind=fk, taps=rng.choice([0, 4, 8]))
        return _fit(c, "frames", 2e9, 1e11)
    if kind == "f":
        taps = rng.choice([0, 0, 4, 8])
        c = dict(kind="f", n=_inputs(rng, 8, 512), c=2 ** rng.randint(5, 10 if taps else 11),
                 frames=_logint(rng, 50, 10000), fkind=rng.choice(["c8", "c4", "r8"]), taps=taps)
        return _fit(c, "frames", 2e9, 1e11)
    if kind == "xd":
        c = dict(kind="xd", n=(_inputs(rng, 16, 1024) + 15) // 16 * 16, c=_logint(rng, 64, 1024),
                 t=_logint(rng, 64, 1024), bits=rng.choice([4, 8]))
        return _fit(c, "c", 4e9, 2e11)
    return dict(kind="batch", jobs=rng.randint(5, 12), sizes=rng.randint(1, 10 ** 6))


# ---- inputs ----------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _packed(g, dumps, t, c, n, bits):
    """Packed samples [dumps][t][c][n]: 8-bit Gaussian noise (sigma 16, clipped to +-127) with a part common
    to all inputs (rho 0.1) as (re, im) bytes; 4-bit uniform -7..7, re in the high nibble."""
    if bits == 4:
        v = torch.randint(-7, 8, (dumps, t, c, n, 2), generator=g, device=DEV, dtype=torch.int8)
        return (((v[..., 0] & 15) << 4) | (v[..., 1] & 15)).view(torch.uint8).contiguous()
    out = torch.empty((dumps, t, c, n, 2), dtype=torch.int8, device=DEV)
    step = max(1, (1 << 28) // max(1, c * n * 2))
    for d in range(dumps):
        for t0 in range(0, t, step):
            s = (min(step, t - t0), c, n, 2)
            z = torch.randn(s, generator=g, device=DEV).mul_(math.sqrt(0.9))
            z += torch.randn((s[0], c, 1, 2), generator=g, device=DEV).mul_(math.sqrt(0.1))
            out[d, t0:t0 + s[0]] = z.mul_(16.0).round_().clamp_(-127, 127).to(torch.int8)
    return out.view(torch.uint8)


def _floats(g, dumps, t, c, n):
    z = torch.randn((dumps, t, c, n, 2), generator=g, device=DEV).mul_(math.sqrt(0.9))
    z += torch.randn((dumps, t, c, 1, 2), generator=g, device=DEV).mul_(math.sqrt(0.1))
    return z.mul_(16.0)


def _time_samples(g, case):
    """Packed time samples [time][input] of an F-stage case, and its taps (a windowed sinc, or None)."""
    n, L, taps = case["n"], case["c"] * (2 if case["fkind"] == "r8" else 1), case["taps"]
    total = (case["frames"] + max(0, taps - 1)) * L
    if case["fkind"] == "c4":
        x = _packed(g, 1, total, 1, n, 4)
    elif case["fkind"] == "c8":
        x = _packed(g, 1, total, 1, n, 8)
    else:
        x = torch.randn((total, n), generator=g, device=DEV).mul_(16.0).round_().clamp_(-127, 127)
        x = x.to(torch.int8).view(torch.uint8)
    h = None
    if taps:
        k = np.arange(taps * L, dtype=np.float64)
        h = (np.sinc((k - (taps * L - 1) / 2) / L) * np.hamming(taps * L)).astype(np.float32)
    return x.reshape(-1), h


def _delays(case, seed):
    """Geometric delays (s) of the inputs and the channels' sky frequencies (Hz)."""
    r = np.random.default_rng(seed)
    tau = torch.from_numpy(r.normal(0.0, 1e-6, case["n"])).to(DEV)
    nu = torch.from_numpy(1.5e8 + 1e4 * np.arange(case["c"])).to(DEV)
    return tau, nu


def _batch_sizes(case):
    """Uneven jobs as the benchmark's batch draws them: 16..256 dual-pol antennas, 64..1024 channels,
    128..2048 samples."""
    r = np.random.default_rng(case["sizes"])
    ants = (16, 32, 64, 128, 256)
    return [(2 * ants[k % 5], 64 * int(r.integers(1, 17)), 128 * int(r.integers(1, 17))) for k in range(case["jobs"])]


_ENGINES = {"bf16x3": corr.ENGINE_BF16X3, "fp32": corr.ENGINE_FP32}
_FKINDS = {"c8": corr.F_COMPLEX8, "c4": corr.F_COMPLEX4, "r8": corr.F_REAL8}


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("x", "xf"):
        n, c, t, d = case["n"], case["c"], case["t"], case["dumps"]
        bits = case["bits"] if kind == "x" else 32
        s["plan"] = plan = corr.Plan(n, c, t, bits)
        s["engine"] = corr.ENGINE_TC if kind == "x" else _ENGINES[case["engine"]]
        s["in"] = _packed(g, d, t, c, n, bits) if kind == "x" else _floats(g, d, t, c, n)
        s["vis"] = plan.empty_vis(d, DEV)
        if case.get("acc"):
            s["vis"].zero_()   # a new dump interval
        s["ws"] = plan.empty_workspace(s["engine"], d, DEV)
    elif kind == "xd":
        s["plan"] = plan = corr.Plan(case["n"], case["c"], case["t"], case["bits"])
        s["in"] = _packed(g, 1, case["t"], case["c"], case["n"], case["bits"])
        s["out"] = torch.empty((1, case["c"], plan.n_baselines, 2), dtype=torch.float32, device=DEV)
        s["tau"], s["nu"] = _delays(case, seed)
        s["ws"] = torch.empty(max(1, plan.dump_workspace_size()), dtype=torch.uint8, device=DEV)
    elif kind in ("f", "fx"):
        s["in"], h = _time_samples(g, case)
        s["fplan"] = corr.FPlan(case["n"], case["c"], _FKINDS[case["fkind"]], case["taps"], h)
        s["spec"] = s["fplan"].empty_spectra(case["frames"], DEV)
        if kind == "fx":
            s["plan"] = corr.Plan(case["n"], s["fplan"].n_out_chan, case["frames"], 32)
            s["vis"] = s["plan"].empty_vis(1, DEV)
            s["ws"] = s["plan"].empty_workspace(corr.ENGINE_BF16X3, 1, DEV)
    else:
        jobs = []
        for n, c, t in _batch_sizes(case):
            x = torch.randint(-60, 61, (t, c, n, 2), generator=g, device=DEV, dtype=torch.int8).view(torch.uint8)
            jobs.append((n, c, t, 8, x, torch.empty((c, n * (n + 1) // 2, 2), dtype=torch.int64, device=DEV)))
        s["vis"] = [j[5] for j in jobs]
        s["batch"] = corr.Batch(jobs, corr.BATCH_GRAPH | corr.BATCH_AUTOTUNE | corr.BATCH_PLANES)
    return s


def run(s):
    kind = s["kind"]
    if kind in ("x", "xf"):
        s["plan"].run(s["in"], s["vis"], s["ws"], accumulate=bool(s["case"].get("acc")), engine=s["engine"],
                      n_dumps=s["case"]["dumps"])
        return s["vis"]
    if kind == "xd":
        s["plan"].run_dump(s["in"], s["out"], s["case"]["t"], s["tau"], s["nu"], s["ws"])
        return s["out"]
    if kind == "batch":
        s["batch"].run()
        return s["vis"]
    s["fplan"].run(s["in"], s["spec"], s["case"]["frames"])
    if kind == "f":
        return s["spec"]
    s["plan"].run(s["spec"], s["vis"], s["ws"], engine=corr.ENGINE_BF16X3)
    return [s["spec"], s["vis"]]


# ---- what a pass cannot do without -----------------------------------------------------------


def _xwork(n, c, t, in_bytes, out_bytes):
    """Samples in once, visibilities out once; 4 real multiply-adds per complex one."""
    p = n * (n + 1) // 2
    return {"bytes": float(t * c * n * in_bytes + c * p * out_bytes), "flops": 8.0 * p * c * t}


def _fwork(case):
    n, taps = case["n"], case["taps"]
    L = case["c"] * (2 if case["fkind"] == "r8" else 1)
    n_out = case["c"] + (1 if case["fkind"] == "r8" else 0)
    frames = case["frames"]
    return {"bytes": float((frames + max(0, taps - 1)) * L * n * (2 if case["fkind"] == "c8" else 1) +
                           frames * n_out * n * 8),
            "flops": float(frames) * n * L * (5.0 * math.log2(L) + 4.0 * taps)}


def work(case):
    kind = case["kind"]
    if kind == "x":
        w = _xwork(case["n"], case["c"], case["t"], 2 if case["bits"] == 8 else 1, 32 if case["acc"] else 16)
        return {k: v * case["dumps"] for k, v in w.items()}
    if kind == "xf":
        w = _xwork(case["n"], case["c"], case["t"], 8, 8)
        return {k: v * case["dumps"] for k, v in w.items()}
    if kind == "xd":
        return _xwork(case["n"], case["c"], case["t"], 2 if case["bits"] == 8 else 1, 8)
    if kind == "batch":
        ws = [_xwork(n, c, t, 2, 16) for n, c, t in _batch_sizes(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    w = _fwork(case)
    if kind == "fx":   # the spectra are an output of the F stage and an input of the X stage
        x = _xwork(case["n"], case["c"] + (1 if case["fkind"] == "r8" else 0), case["frames"], 8, 8)
        w = {k: w[k] + x[k] for k in w}
    return w


# ---- the same results in 64 bits -------------------------------------------------------------


def _correlate(z):
    """z: complex128 [t][c][n] -> [c][P] sums over t of z_i conj(z_j), i <= j in row order."""
    z = z.permute(1, 2, 0)
    iu = torch.triu_indices(z.shape[1], z.shape[1], device=z.device)
    return (z @ z.conj().transpose(1, 2))[:, iu[0], iu[1]]


def _unpack(x, bits):
    """Packed samples [...][n](2) -> complex128."""
    if bits == 4:
        v = x.view(torch.int8)
        return torch.complex((v >> 4).double(), ((v << 4) >> 4).double())
    return torch.view_as_complex(x.view(torch.int8).double())


def _spectra(case, x, h):
    n, frames, taps, bits = case["n"], case["frames"], max(1, case["taps"]), {"c8": 8, "c4": 4, "r8": 0}[case["fkind"]]
    L = case["c"] * (2 if case["fkind"] == "r8" else 1)
    n_out = case["c"] + (1 if case["fkind"] == "r8" else 0)
    x = x.view(-1, L, n, 2) if bits == 8 else x.view(-1, L, n)
    w = torch.ones((1, L, 1), dtype=torch.float64, device=DEV)
    if h is not None:
        w = torch.from_numpy(h.astype(np.float64)).to(DEV).view(taps, L, 1)
    out = torch.empty((frames, n_out, n), dtype=torch.complex128, device=DEV)
    step = max(1, (1 << 25) // (L * n))
    for f0 in range(0, frames, step):
        f1 = min(frames, f0 + step)
        y = 0
        for m in range(taps):
            v = x[f0 + m:f1 + m]
            y = y + w[m] * (_unpack(v, bits) if bits else v.view(torch.int8).to(torch.complex128))
        out[f0:f1] = torch.fft.fft(y, dim=1)[:, :n_out]
    return out


def _xcorr_chunks(c, n, t, samples):
    """[c][P][2] float64; samples(c0, c1) gives complex128 [t][c1 - c0][n]."""
    out = torch.empty((c, n * (n + 1) // 2, 2), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 27) // max(n * n, t * n))
    for c0 in range(0, c, step):
        c1 = min(c, c0 + step)
        out[c0:c1] = torch.view_as_real(_correlate(samples(c0, c1)))
    return out


def exact(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind in ("x", "batch"):
        return None   # whole numbers
    if kind == "xf":
        x = torch.view_as_complex(_floats(g, case["dumps"], case["t"], case["c"], case["n"]))
        return torch.stack([_xcorr_chunks(case["c"], case["n"], case["t"],
                                          lambda a, b, d=d: x[d, :, a:b].to(torch.complex128))
                            for d in range(case["dumps"])])
    if kind == "xd":
        x = _packed(g, 1, case["t"], case["c"], case["n"], case["bits"])[0]
        tau, nu = _delays(case, seed)
        v = torch.view_as_complex(_xcorr_chunks(case["c"], case["n"], case["t"],
                                                lambda a, b: _unpack(x[:, a:b].contiguous(), case["bits"])))
        iu = torch.triu_indices(case["n"], case["n"], device=DEV)
        for c in range(case["c"]):
            v[c] *= torch.polar(torch.full_like(tau, 1.0)[iu[0]] / case["t"],
                                2.0 * math.pi * torch.remainder(nu[c] * (tau[iu[0]] - tau[iu[1]]), 1.0))
        return torch.view_as_real(v)[None]
    spec = _spectra(case, *_time_samples(g, case))
    if kind == "f":
        return torch.view_as_real(spec)
    vis = _xcorr_chunks(spec.shape[1], case["n"], case["frames"], lambda a, b: spec[:, a:b])
    return [torch.view_as_real(spec), vis[None]]
