"""The measured work of the correlator: what its users call, at their sizes.

``listed()`` holds the named cases and ``draw(rng)`` one more of the same
ranges.  A case is a dict of plain values:

    kind    "push"     one handle: device pushes, then the dump (an integration)
            "track"    the same with coarse sample delays and gain/delay corrections
            "host"     the same from page-locked host memory into host memory
            "noalloc"  corr_correlate_noalloc, the allocation-free one-shot call
            "batch"    CorrelatorBatch, one captured step replayed
            "grad"     autograd.visibilities, forward and backward
    N, K    antennas and transform length ("modes" = "N:K,N:K,..." for a batch)
    frames  spectra per antenna ("samples" = samples per antenna and mode for a batch)
    push    spectra per push
    dtype   X-engine precision (fp32, fp16, fp8, fp32_simt)

Inputs follow the signal model of the paper's load: 4-bit samples of Gaussian
noise (2 LSB rms) with a 1% common component that reaches every antenna with
its own integer delay, and a weak narrowband tone.
"""

import math

import numpy as np
import torch

from paper_1102_0148_gb300 import autograd, corr

_MAX_DELAY = 16       # integer delays of the common component, samples


def listed():
    return [
        # The paper's 44-element array, 2^17 samples per antenna in one call:
        # a short look (a fringe check, one pulsar phase bin).  Latency and
        # launches count here.
        dict(name="short-look-fp32", kind="push", N=44, K=512, frames=256, push=256, dtype="fp32"),
        # The allocation-free call of a real-time acquisition loop, on one
        # 2^20-sample block of the same array (CUDA-core X-engine).
        dict(name="oneshot-noalloc", kind="noalloc", N=44, K=512, frames=2048),
        # The real-time load: 1 s at 35 MS/s streamed in 2^20-sample pushes,
        # full precision.  68359 spectra are no multiple of any tile.
        dict(name="realtime-fp32", kind="push", N=44, K=512, frames=68359, push=2048, dtype="fp32"),
        # The full 40 MHz band, 1 s at 80 MS/s, with the FP16 X-engine: the
        # largest integration, more than one workspace pass.
        dict(name="fullband-fp16", kind="push", N=44, K=512, frames=156250, push=2048, dtype="fp16"),
        # The real-time load with the FP8 X-engine.
        dict(name="realtime-fp8", kind="push", N=44, K=512, frames=68359, push=2048, dtype="fp8"),
        # A dense array, 256 elements at K = 1024, 2^22 samples, full precision:
        # the cross-multiply dominates.
        dict(name="dense-fp32", kind="push", N=256, K=1024, frames=4096, push=4096, dtype="fp32"),
        # Four concurrent modes (sub-arrays of uneven N and K and the dense
        # array) as one captured step, replayed per integration.
        dict(name="batch-fp16", kind="batch", modes="44:512,22:2048,11:4096,256:1024",
             samples=1 << 22, dtype="fp16"),
        # Gain and delay calibration: the loss against the uncorrected
        # instrument, forward and backward, 2^20 samples.
        dict(name="gradient", kind="grad", N=44, K=512, frames=2048),
        # Delay tracking: coarse sample delays undo the geometric delays and
        # fractional delays and gains are applied in the F-engine; a stream in
        # 2^20-sample pushes whose last one is ragged.
        dict(name="tracking-fp32", kind="track", N=44, K=512, frames=17001, push=2048, dtype="fp32"),
        # Samples that arrive in host memory: 2^23 per antenna from
        # page-locked buffers, visibilities back to the host.
        dict(name="host-stream-fp32", kind="host", N=44, K=512, frames=16384, push=2048, dtype="fp32"),
        # Coarse channels at high time resolution: 64 elements, K = 256.
        dict(name="coarse-k256-fp32", kind="push", N=64, K=256, frames=16384, push=4096, dtype="fp32"),
        # Fine channels on an array that fills no tile (130 elements, 1500
        # spectra), FP16.
        dict(name="ragged-k2048-fp16", kind="push", N=130, K=2048, frames=1500, push=1500, dtype="fp16"),
    ]


# ----------------------------------------------------------------------------
# Drawn cases
# ----------------------------------------------------------------------------

_MAX_SAMPLES = 2.0e9      # antenna-samples of a drawn case (the full-band case has 3.5e9)
_MAX_XFLOPS = 3.0e11      # its cross-multiply (the dense case has 5.5e11)
_SHORT_K = 5.0e5          # short transforms (K <= 256) cost more per sample: samples / K at most


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _max_frames(N, K, samples=_MAX_SAMPLES, flops=_MAX_XFLOPS):
    if K <= 256:
        samples = min(samples, _SHORT_K * K)
    return max(64, int(min(samples / (N * K), flops / (4.0 * N * (N + 1) * (K // 2)))))


def draw(rng):
    kind = rng.choice(["push"] * 5 + ["noalloc", "batch", "grad", "track", "host"])
    K = 1 << rng.randint(4, 12)
    if rng.random() < 0.4:
        K = 512
    if kind == "noalloc":
        while True:
            N = _log_int(rng, 2, 64)
            if K * 8 + N * (N + 1) // 2 * (K // 2) * 24 + 128 * K * N * 4 < (31 << 20):
                break
            K = max(16, K // 2)
        frames = _log_int(rng, 33, _max_frames(N, K, 2e8, 2e10))
        return dict(kind=kind, N=N, K=K, frames=frames)
    if kind == "batch":
        modes = []
        for _ in range(rng.randint(2, 4)):
            modes.append("%d:%d" % (_log_int(rng, 2, 160), 1 << rng.randint(7, 12)))
        return dict(kind=kind, modes=",".join(modes), samples=4096 * _log_int(rng, 8, 512),
                    dtype=rng.choice(["fp32", "fp16", "fp8"]))
    if kind == "grad":
        N = _log_int(rng, 2, 128)
        K = max(64, K)
        return dict(kind=kind, N=N, K=K, frames=_log_int(rng, 64, _max_frames(N, K, 4e8, 2e10)))
    if kind in ("track", "host"):
        N = _log_int(rng, 2, 128)
        frames = _log_int(rng, 64, _max_frames(N, K, 5e8, 5e10))
        return dict(kind=kind, N=N, K=K, frames=frames, push=_log_int(rng, 33, frames) if frames > 33 else frames,
                    dtype=rng.choice(["fp32", "fp16", "fp8"]))
    N = _log_int(rng, 1, 512)
    dtype = rng.choice(["fp32", "fp32", "fp16", "fp8", "fp32_simt"])
    frames = _log_int(rng, 64, _max_frames(N, K) if dtype != "fp32_simt"
                      else _max_frames(N, K, 5e8, 3e10))
    push = rng.choice([frames, min(frames, 2048), _log_int(rng, 64, frames)])
    return dict(kind=kind, N=N, K=K, frames=frames, push=max(push, frames // 64), dtype=dtype)


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

def _modes(case):
    return [tuple(int(v) for v in m.split(":")) for m in case["modes"].split(",")]


def _samples(N, K, frames, seed):
    """Packed 4-bit samples [frames][N][K/2] (uint8, on the GPU) and the
    integer delays of the common component."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    d = torch.randint(0, _MAX_DELAY, (N,), generator=g, device=dev)
    out = torch.empty((frames, N, K // 2), dtype=torch.uint8, device=dev)
    prev = torch.zeros(_MAX_DELAY, device=dev)
    block = max(1, (1 << 26) // (N * K))
    for f0 in range(0, frames, block):
        f1 = min(frames, f0 + block)
        T = (f1 - f0) * K
        c = torch.cat([prev, 0.2 * torch.randn(T, generator=g, device=dev)])
        prev = c[-_MAX_DELAY:].clone()
        t = torch.arange(f0 * K, f1 * K, device=dev, dtype=torch.float64)
        tone = (0.5 * torch.cos(2.0 * math.pi * torch.remainder(t * (97.0 / 512.0), 1.0))).float()
        x = torch.randn((N, T), generator=g, device=dev).mul_(2.0)
        x += c.unfold(0, T, 1)[_MAX_DELAY - d]
        x += tone
        q = x.round_().clamp_(-8, 7).to(torch.int8)
        b = (q[:, 0::2] & 15) | (q[:, 1::2] << 4)
        out[f0:f1] = b.view(torch.uint8).view(N, f1 - f0, K // 2).transpose(0, 1)
    return out, d


def _gains_delays(N, seed):
    """Per-antenna complex gains ~ CN(1, 0.1^2) and fractional delays ~ U(-0.5, 0.5)."""
    rng = np.random.Generator(np.random.PCG64(seed + 17))
    g = 1.0 + 0.1 / math.sqrt(2.0) * (rng.normal(size=N) + 1j * rng.normal(size=N))
    return g.astype(np.complex64), rng.uniform(-0.5, 0.5, N).astype(np.float32)


def _pushes(case):
    f, step = case["frames"], case["push"]
    return [(a, min(f, a + step)) for a in range(0, f, step)]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "batch":
        modes = _modes(case)
        st["data"] = [_samples(N, K, case["samples"] // K, seed * 8 + m)[0].reshape(-1)
                      for m, (N, K) in enumerate(modes)]
        b = corr.CorrelatorBatch(modes, case["dtype"])
        for h, (N, K) in zip(b.handles, modes):
            corr.corr_set_chunk(h, case["samples"] // K)
        st["vis"] = [torch.empty((N * (N + 1) // 2, K // 2), dtype=torch.complex64, device="cuda")
                     for N, K in modes]
        torch.cuda.synchronize()
        b.capture(st["data"], st["vis"])
        st["batch"] = b
        return st
    N, K, frames = case["N"], case["K"], case["frames"]
    x, d = _samples(N, K, frames, seed)
    shape = (N * (N + 1) // 2, K // 2)
    if kind == "host":
        st["x"] = torch.empty(x.shape, dtype=torch.uint8, pin_memory=True).copy_(x)
        st["vis"] = torch.empty(shape, dtype=torch.complex64, pin_memory=True)
    else:
        st["x"] = x
        st["vis"] = torch.empty(shape, dtype=torch.complex64, device="cuda")
    if kind == "noalloc":
        return st
    st["c"] = c = corr.Correlator(N, K, case.get("dtype", "fp32"))
    if kind == "track":
        g, tau = _gains_delays(N, seed)
        c.set_corrections(g, tau)
        st["sample_delays"] = (d.max() - d).cpu().numpy().astype(np.int32) % (K + 1)
    if kind == "grad":
        g, tau = _gains_delays(N, seed)
        st["gains"] = torch.from_numpy(g).cuda().requires_grad_(True)
        st["delays"] = torch.from_numpy(tau).cuda().requires_grad_(True)
        st["model"] = _visibilities64(x, N, K)
    torch.cuda.synchronize()
    return st


# ----------------------------------------------------------------------------
# One pass
# ----------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        n = st["batch"].replay()
        st["batch"].sync()
        return {"vis": st["vis"], "n": n}
    if kind == "noalloc":
        x = st["x"]
        corr.corr_correlate_noalloc(x, case["frames"] * case["K"], case["N"], case["K"], st["vis"],
                                    torch.cuda.current_stream())
        return {"vis": st["vis"]}
    c, x = st["c"], st["x"]
    if kind == "grad":
        V = autograd.visibilities(st["gains"], st["delays"], x, c)
        loss = (V - st["model"]).abs().pow(2).sum()
        gg, gt = torch.autograd.grad(loss, (st["gains"], st["delays"]))
        return {"vis": V.detach(), "loss": loss.detach(), "grad_gains": gg, "grad_delays": gt}
    if kind == "track":
        # a new pointing: the stream starts over with its own delays
        c.set_sample_delays(None)
        c.set_sample_delays(st["sample_delays"])
    for a, b in _pushes(case):
        c.push(x[a:b])
    vis, n = c.dump(out=st["vis"])
    return {"vis": vis, "n": n}


# ----------------------------------------------------------------------------
# Accounting and the 64-bit values
# ----------------------------------------------------------------------------

def _work_one(N, K, frames, out_bytes):
    P, C = N * (N + 1) // 2, K // 2
    return (N * frames * (K // 2) + P * C * out_bytes,
            N * frames * 2.5 * K * math.log2(K) + 8.0 * P * C * frames)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_work_one(N, K, case["samples"] // K, 8) for N, K in _modes(case)]
        return {"bytes": float(sum(a for a, _ in w)), "flops": float(sum(b for _, b in w))}
    N, K, frames = case["N"], case["K"], case["frames"]
    P, C = N * (N + 1) // 2, K // 2
    if kind == "grad":
        # forward; backward from the samples again and from dL/dV (its closed
        # form: two complex products per pair, antenna and channel)
        b, f = _work_one(N, K, frames, 16)
        return {"bytes": float(2 * N * frames * (K // 2) + 2 * P * C * 16),
                "flops": float(2 * f + 32.0 * P * C)}
    b, f = _work_one(N, K, frames, 8)
    return {"bytes": float(b), "flops": float(f)}


def _unpack64(x, N, K):
    """uint8 [F][N][K/2] -> float64 [F][N][K]."""
    lo = (x & 15).to(torch.int16)
    hi = (x >> 4).to(torch.int16)
    s = torch.stack([lo, hi], dim=-1).reshape(x.shape[0], N, K)
    return torch.where(s >= 8, s - 16, s).double()


def _visibilities64(x, N, K, gains=None, delays=None, sample_delays=None):
    """Sum over frames of Y_i conj(Y_j), [P][C] complex128."""
    dev = x.device
    C = K // 2
    iu, ju = torch.triu_indices(N, N, device=dev)
    G = torch.zeros((C, N, N), dtype=torch.complex128, device=dev)
    a = None
    if gains is not None:
        k = torch.arange(C, dtype=torch.float64, device=dev)
        tau = torch.as_tensor(delays, device=dev).double()
        a = (torch.as_tensor(gains, device=dev).to(torch.complex128)[:, None]
             * torch.exp(-2j * math.pi * tau[:, None] * k[None, :] / K))
    prev = torch.zeros((N, K), dtype=torch.float64, device=dev)
    if sample_delays is not None:
        shift = torch.as_tensor(sample_delays, device=dev).long()
    block = max(1, (1 << 25) // (N * K))
    for f0 in range(0, x.shape[0], block):
        s = _unpack64(x[f0:f0 + block], N, K)
        if sample_delays is not None:
            F = s.shape[0]
            flat = torch.cat([prev, s.transpose(0, 1).reshape(N, F * K)], dim=1)
            prev = flat[:, -K:].clone()
            idx = torch.arange(F * K, device=dev)[None, :] + (K - shift)[:, None]
            s = flat.gather(1, idx).reshape(N, F, K).transpose(0, 1)
        Y = torch.fft.rfft(s, dim=-1)[..., :C]
        if a is not None:
            Y = Y * a
        Yk = Y.permute(2, 1, 0).contiguous()
        G += Yk @ Yk.conj().transpose(1, 2)
    return G[:, iu, ju].t().contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return {"vis": [_visibilities64(_samples(N, K, case["samples"] // K, seed * 8 + m)[0], N, K)
                        for m, (N, K) in enumerate(_modes(case))],
                "n": [case["samples"] // K for _, K in _modes(case)]}
    N, K, frames = case["N"], case["K"], case["frames"]
    x, d = _samples(N, K, frames, seed)
    if kind == "track":
        g, tau = _gains_delays(N, seed)
        D = (d.max() - d).cpu().numpy() % (K + 1)
        return {"vis": _visibilities64(x, N, K, g, tau, D), "n": frames}
    V = _visibilities64(x, N, K)
    if kind == "noalloc":
        return {"vis": V}
    if kind == "grad":
        g32, t32 = _gains_delays(N, seed)
        g = torch.from_numpy(g32).cuda().to(torch.complex128).requires_grad_(True)
        tau = torch.from_numpy(t32).cuda().double().requires_grad_(True)
        k = torch.arange(K // 2, dtype=torch.float64, device="cuda")
        a = g[:, None] * torch.exp(-2j * math.pi * tau[:, None] * k[None, :] / K)
        iu, ju = torch.triu_indices(N, N, device="cuda")
        W = a[iu] * a[ju].conj() * V
        loss = (W - V).abs().pow(2).sum()
        gg, gt = torch.autograd.grad(loss, (g, tau))
        return {"vis": W.detach(), "loss": loss.detach(), "grad_gains": gg, "grad_delays": gt}
    return {"vis": V, "n": frames}
