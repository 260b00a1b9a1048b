"""The workloads this library is timed on.

Each case is one pass of work that a user of the library has it do: an
integration period of one channel (in one call, or as it arrives in short
chunks), a period of many channels at once, a channel whose comb offset has no
short period, and a batch of tone DFTs.  Sample rates, combs, offsets and
lengths are those of the benchmark and the tests, and lengths of the same kind
between them: 10 ms recorder chunks, fractions of a second, whole seconds.

A case is a dict of plain values with a "kind":
  plan   one channel: fmt, fs, fc, fo, n samples, handed over in `calls` calls
         of equal length (the last takes the rest), starting `skew` elements
         into a 256-byte aligned buffer
  batch  `channels` channels drawn from `mix` (sample rates up to `fs_max`,
         2-bit and int8 alternating, lengths between lo_ms and hi_ms in steps
         of 10 ms), folded and finalized as two calls or as one graph replay
  rot    one channel whose offset is prime or not a whole number of hertz
  dft    C channels of an N-point tone DFT in one of the library's modes
"""
import math
import random

import numpy as np
import torch

import paper_2501_05993_gb300 as pcal

LEVELS = (-3.3359, -1.0, 1.0, 3.3359)  # 2-bit codes 0..3
MHZ = 1_000_000


def listed():
    return [
        # a recorder's 10 ms chunk of one 64 MHz channel, finalized at once: the smallest call
        {"name": "chunk_2bit", "kind": "plan", "fmt": "2bit", "fs": 64 * MHZ, "fc": MHZ, "fo": 10_000, "n": 640_000,
         "calls": 1, "skew": 0},
        # a quarter of a second of the 16 MHz float channel as it arrives: 25 chunks of 10 ms
        {"name": "live_f32", "kind": "plan", "fmt": "f32", "fs": 16 * MHZ, "fc": MHZ, "fo": 10_000, "n": 4_000_000,
         "calls": 25, "skew": 0},
        # 0.1 s of an int8 channel cut out of a longer recording: odd start, odd length
        {"name": "cut_i8", "kind": "plan", "fmt": "i8", "fs": 128 * MHZ, "fc": MHZ, "fo": 30_000, "n": 12_800_003,
         "calls": 1, "skew": 5},
        # one second of the 16 MHz float channel (16e6 samples)
        {"name": "second_f32", "kind": "plan", "fmt": "f32", "fs": 16 * MHZ, "fc": MHZ, "fo": 10_000, "n": 16_000_000,
         "calls": 1, "skew": 0},
        # eight seconds of a 64 MHz 2-bit channel (the benchmark's channel)
        {"name": "long_2bit", "kind": "plan", "fmt": "2bit", "fs": 64 * MHZ, "fc": MHZ, "fo": 10_000,
         "n": 512 * MHZ, "calls": 1, "skew": 0},
        # a wide band with many tones: 1024 MHz, 1024 tones, half a second of int8
        {"name": "wide_i8", "kind": "plan", "fmt": "i8", "fs": 1024 * MHZ, "fc": MHZ, "fo": 10_000, "n": 512 * MHZ + 11,
         "calls": 1, "skew": 0},
        # an offset of whole kilohertz, not tens: a period of 256,000 samples; one second of 2-bit
        {"name": "fine_2bit", "kind": "plan", "fmt": "2bit", "fs": 256 * MHZ, "fc": MHZ, "fo": 7_000, "n": 256 * MHZ,
         "calls": 1, "skew": 0},
        # 64 mixed channels of up to 0.8 s, folded together
        {"name": "batch_mixed", "kind": "batch", "channels": 64, "mix": 11, "fs_max": 256 * MHZ, "lo_ms": 50,
         "hi_ms": 800, "graph": False},
        # 64 live channels, one 10 ms chunk each, as one replayed step
        {"name": "batch_live", "kind": "batch", "channels": 64, "mix": 12, "fs_max": 1024 * MHZ, "lo_ms": 10,
         "hi_ms": 10, "graph": True},
        # a prime offset: no period to fold over; four seconds of int8
        {"name": "prime_i8", "kind": "rot", "fmt": "i8", "fs": 64 * MHZ, "fc": MHZ, "fo": 10_007.0, "n": 256 * MHZ},
        # an offset of a fraction of a hertz; one second of the float channel
        {"name": "fraction_f32", "kind": "rot", "fmt": "f32", "fs": 16 * MHZ, "fc": MHZ, "fo": 10_007.25,
         "n": 16_000_000},
        # the tones of 4096 channels at once, in the default mode
        {"name": "tones_1024", "kind": "dft", "C": 4096, "N": 1024, "mode": "tf32x3"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "plan", "batch", "rot", "dft"])
    if kind == "dft":
        N = rng.choice([16, 20, 32, 50, 64, 100, 128, 200, 250, 256, 500, 512, 1000, 1024])
        return {"kind": "dft", "C": _log_int(rng, 16, 4096), "N": N, "mode": rng.choice(["fp32", "tf32x3", "bf16x6"])}
    if kind == "batch":
        graph = rng.random() < 0.5
        lo = 10 if graph else rng.choice([10, 20, 50])
        return {"kind": "batch", "channels": rng.randint(4, 64), "mix": rng.randint(0, 10**6),
                "fs_max": rng.choice([64, 256, 1024] if graph else [64, 256]) * MHZ, "lo_ms": lo,
                "hi_ms": 10 if graph else lo + 10 * rng.randint(0, 50), "graph": graph}
    fmt = rng.choice(["2bit", "i8", "f32"])
    if kind == "rot":
        fs = rng.choice([16, 32, 64, 128, 256, 1024]) * MHZ
        top = {"2bit": 256, "i8": 256, "f32": 64}[fmt] * MHZ
        n = min(_log_int(rng, 160_000, top), top)
        return {"kind": "rot", "fmt": fmt, "fs": fs, "fc": MHZ, "fo": rng.randint(1, 16 * 500_000) / 16.0,
                "n": n // 4 * 4 if fmt == "2bit" else n}
    fs = rng.choice([16, 20, 32, 50, 64, 100, 128, 256, 512, 1024]) * MHZ
    fo = rng.choice([1000, 10_000, 10_000, 10_000]) * rng.randint(1, 49)
    top = {"2bit": 512, "i8": 512, "f32": 64}[fmt] * MHZ
    n = min(_log_int(rng, 160_000, top), top)
    calls = 1
    if rng.random() < 0.3:  # as it arrives: chunks of at least 10 ms
        calls = max(1, min(rng.randint(2, 32), n // (fs // 100)))
    return {"kind": "plan", "fmt": fmt, "fs": fs, "fc": MHZ, "fo": fo, "n": n // 4 * 4 if fmt == "2bit" else n,
            "calls": calls, "skew": rng.choice([0, 0, 1, 3])}


# ---- inputs: unit Gaussian noise plus a comb of N delayed tones --------------------------

AMP = 0.02


def _bytes_of(fmt, n):
    return {"2bit": n // 4, "i8": n, "f32": 4 * n}[fmt]


def _quantise(x, fmt, out):
    """x (float32, a multiple of four samples) into out: the format's elements."""
    if fmt == "f32":
        out.copy_(x)
    elif fmt == "i8":
        out.copy_(x.mul_(20.0).round_().clamp_(-128, 127))
    else:
        c = ((x >= -0.98).to(torch.uint8) + (x >= 0) + (x >= 0.98)).view(-1, 4)
        out.copy_(c[:, 0] | c[:, 1] << 2 | c[:, 2] << 4 | c[:, 3] << 6)


def _comb(fs, fc, fo, td, k):
    """sum_i sin(2 pi (i fc + fo)(k/fs + td)) for sample numbers k (float64), in float32."""
    N = fs // fc
    i = torch.arange(N, dtype=torch.float64, device="cuda")
    turns = torch.remainder(torch.outer(i, i) / N + i * (fc * td), 1.0)
    g = torch.polar(torch.ones_like(turns), 2 * math.pi * turns).sum(1).to(torch.complex64)
    ph = (2 * math.pi * torch.remainder(k * (fo / fs) + fo * td, 1.0)).float()
    gb = g[torch.remainder(k, N).long()]
    return torch.sin(ph) * gb.real + torch.cos(ph) * gb.imag


def _samples(fmt, fs, fc, fo, n, seed, skew=0, folds=True):
    """n samples on the GPU; folds: the comb repeats after L = fs / gcd samples."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    td = 3e-9 + 20e-9 * random.Random(seed).random()
    dtype = {"2bit": torch.uint8, "i8": torch.int8, "f32": torch.float32}[fmt]
    spe = 4 if fmt == "2bit" else 1  # samples per element
    buf = torch.empty(n // spe + skew, dtype=dtype, device="cuda")
    x = buf[skew:]
    if folds:
        L = fs // math.gcd(fs, fc, int(fo))
        comb = AMP * _comb(fs, fc, fo, td, torch.arange(L, dtype=torch.float64, device="cuda"))
        step = max(4, (1 << 25) // L // 4 * 4) * L
    else:
        step = 1 << 24
    for at in range(0, n, step):
        m = min(step, n - at)
        if folds:
            z = torch.randn(-(-m // (4 * L)) * 4, L, generator=gen, device="cuda").add_(comb).view(-1)[:m]
        else:
            z = torch.randn(m, generator=gen, device="cuda")
            z += AMP * _comb(fs, fc, fo, td, torch.arange(at, at + m, dtype=torch.float64, device="cuda"))
        _quantise(z, fmt, x[at // spe:(at + m) // spe])
    return x


def _mix(case):
    """The channels of a batch: (fs, fc, fo, fmt, samples)."""
    rng = random.Random(case["mix"])
    rates = [r * MHZ for r in (32, 64, 128, 256, 512, 1024) if r * MHZ <= case["fs_max"]]
    out = []
    for c in range(case["channels"]):
        fs = rng.choice(rates)
        ms = 10 * rng.randint(case["lo_ms"] // 10, case["hi_ms"] // 10)
        out.append((fs, MHZ, 10_000 * rng.randint(0, 99), "2bit" if c % 2 == 0 else "i8", fs // 1000 * ms))
    return out


def _pulse(case, seed):
    """Folded bins of C channels: noise of each channel's own level and a delayed pulse."""
    C, N = case["C"], case["N"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    P = torch.randn(C, N, dtype=torch.complex64, generator=gen, device="cuda")
    P *= torch.pow(10.0, 6 * torch.rand(C, 1, generator=gen, device="cuda") - 2)
    at = torch.randint(0, N, (C, 1), generator=gen, device="cuda")
    return P.scatter_add_(1, at, P.abs().amax(1, keepdim=True).to(torch.complex64) * 10)


class _Doubles:
    """A device address as an array of doubles; it keeps the object that owns the memory."""

    def __init__(self, owner, ptr, n):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (int(ptr), False), "shape": (n,), "typestr": "<f8", "version": 3}


def _device_doubles(owner, ptr, n):
    return torch.as_tensor(_Doubles(owner, ptr, n), device="cuda")


def _parts(res, N):
    """The result vector of a finalize by its parts (pcal.h: pcal_result_device, pcal_read_post)."""
    return {"phasors": res[:2 * N], "amp": res[2 * N:3 * N], "phase": res[3 * N:4 * N],
            "unwrapped": res[4 * N:5 * N], "td": res[5 * N:5 * N + 1], "sigma_td": res[5 * N + 1:5 * N + 2],
            "samples": res[5 * N + 2:5 * N + 3], "td_peak": res[5 * N + 3:5 * N + 4],
            "peak_bin": res[5 * N + 4:5 * N + 5], "bandpass_phase": res[5 * N + 5:6 * N + 5]}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "plan":
        fs, fc, fo, n, calls = (case[k] for k in ("fs", "fc", "fo", "n", "calls"))
        x = _samples(case["fmt"], fs, fc, fo, n, seed, case["skew"])
        spe = 4 if case["fmt"] == "2bit" else 1
        each = n // calls // spe * spe
        cuts = [c * each for c in range(calls)] + [n]
        plan = pcal.Plan(fs, fc, fo, case["fmt"])
        res = _device_doubles(plan, plan.result_device_ptr, 6 * plan.N + 5)
        return {"kind": kind, "plan": plan, "chunks": [x[a // spe:b // spe] for a, b in zip(cuts, cuts[1:])],
                "out": _parts(res, plan.N)}
    if kind == "batch":
        mix = _mix(case)
        xs = [_samples(fmt, fs, fc, fo, n, seed * 1000 + c) for c, (fs, fc, fo, fmt, n) in enumerate(mix)]
        batch = pcal.Batch([ch[:4] for ch in mix])
        out = [_device_doubles(batch, pcal.pcal_batch_result_device(batch.handle, c), 6 * int(g.N) + 5)
               for c, g in enumerate(batch.geometry)]
        return {"kind": kind, "batch": batch, "xs": xs, "ns": [ch[4] for ch in mix], "graph": case["graph"], "out": out}
    if kind == "rot":
        x = _samples(case["fmt"], case["fs"], case["fc"], case["fo"], case["n"], seed, folds=False)
        return {"kind": kind, "plan": pcal.RotPlan(case["fs"], case["fc"], case["fo"], case["fmt"]), "x": x,
                "n": case["n"]}
    P = _pulse(case, seed)
    return {"kind": kind, "dft": pcal.Dft(case["N"], case["mode"]), "P": P, "C": case["C"], "T": torch.empty_like(P)}


def run(state):
    kind = state["kind"]
    if kind == "plan":
        for x in state["chunks"]:
            state["plan"].accumulate(x)
        state["plan"].finalize_device()
        return state["out"]
    if kind == "batch":
        if state["graph"]:
            state["batch"].step_graph(state["xs"], state["ns"])
        else:
            state["batch"].accumulate(state["xs"], state["ns"])
            state["batch"].finalize_device()
        return state["out"]
    if kind == "rot":
        state["plan"].accumulate(state["x"], state["n"])
        state["plan"].finalize_device()
        return state["plan"].results()
    state["dft"].execute(state["P"], state["C"], state["T"])
    return state["T"]


def work(case):
    kind = case["kind"]
    if kind == "dft":  # P in, T out; a fast transform's operations
        C, N = case["C"], case["N"]
        return {"bytes": 16 * C * N, "flops": 5 * C * N * max(1.0, math.log2(N))}
    if kind == "batch":
        mix = _mix(case)
        return {"bytes": sum(_bytes_of(ch[3], ch[4]) + 8 * (6 * (ch[0] // ch[1]) + 5) for ch in mix),
                "flops": sum(ch[4] for ch in mix)}
    N = case["fs"] // case["fc"]
    # one addition a sample where the samples fold, one real-by-complex product and its sum where they do not
    return {"bytes": _bytes_of(case["fmt"], case["n"]) + 8 * (6 * N + 5), "flops": case["n"] * (1 if kind == "plan" else 4)}


# ---- the same in 64 bits, from the definitions ---------------------------------------------

def _decoded(x, fmt, at, m):
    """Samples at .. at + m of x as float64."""
    if fmt != "2bit":
        return x[at:at + m].double()
    lev = torch.tensor(LEVELS, dtype=torch.float64, device="cuda")
    b = x[at // 4:(at + m) // 4]
    return lev[torch.stack([(b >> s) & 3 for s in (0, 2, 4, 6)], 1).view(-1).long()]


def _folded_bins(x, fmt, fs, fc, fo, n):
    """P[b]: the samples rotated by exp(-j 2 pi fo n/fs) and folded modulo N, through the sums modulo L."""
    g = math.gcd(fs, fc, int(fo))
    L, N = fs // g, fs // fc
    S = torch.zeros(L, dtype=torch.float64, device="cuda")
    rows = max(4, (1 << 24) // L // 4 * 4)
    for at in range(0, n, rows * L):
        m = min(rows * L, n - at)
        v = _decoded(x, fmt, at, m)
        S += v[:m // L * L].view(-1, L).sum(0)
        S[:m % L] += v[m // L * L:]
    r = torch.arange(L, device="cuda") * (int(fo) // g) % L
    return (S * torch.polar(torch.ones_like(S), r.double() * (-2 * math.pi / L))).view(-1, N).sum(0)


def _rotated_bins(x, fmt, fs, fc, fo, n):
    """P[b] with every sample rotated; fo is a whole number of sixteenths of a hertz."""
    N = fs // fc
    num, den = int(fo * 16), fs * 16
    P = torch.zeros(N, dtype=torch.complex128, device="cuda")
    step = (1 << 23) // (4 * N) * (4 * N)
    for at in range(0, n, step):
        m = min(step, n - at)
        k = torch.arange(at, at + m, device="cuda")
        v = _decoded(x, fmt, at, m)
        v = v * torch.polar(torch.ones_like(v), (k * num % den).double() * (-2 * math.pi / den))
        P += v[:m // N * N].view(-1, N).sum(0)
        P[:m % N] += v[m // N * N:]
    return P


def _products(P, M, fs, fc):
    """Everything a finalize gives, from the folded bins P (complex128)."""
    P = P.cpu().numpy()
    N = len(P)
    T = np.fft.fft(P)
    wrap = lambda v: v - 2 * np.pi * np.floor((v + np.pi) / (2 * np.pi))  # noqa: E731
    psi = wrap(np.angle(T) + np.pi / 2)
    u = psi[0] + np.concatenate([[0.0], np.cumsum(wrap(np.diff(psi)))])
    w, i = np.abs(T) ** 2, np.arange(N)
    dx, du = i - (w * i).sum() / w.sum(), u - (w * u).sum() / w.sum()
    sxx = (w * dx * dx).sum()
    slope = (w * dx * du).sum() / sxx
    ssr = (w * (du - slope * dx) ** 2).sum()
    a = np.abs(P)
    b = int(np.argmax(a))
    ym, y0, yp = a[b - 1], a[b], a[(b + 1) % N]
    pos = b + 0.5 * (ym - yp) / (ym - 2 * y0 + yp)
    q = -pos - N * np.floor((-pos + N / 2) / N)
    return {"phasors": np.stack([T.real, T.imag], 1).reshape(-1), "amp": 2 * np.abs(T) / M, "phase": psi,
            "unwrapped": u, "td": np.array([slope / (2 * np.pi * fc)]),
            "sigma_td": np.array([np.sqrt(ssr / sxx / (N - 2)) / (2 * np.pi * fc)]), "samples": np.array([float(M)]),
            "td_peak": np.array([q / fs]), "peak_bin": np.array([pos]), "bandpass_phase": du - slope * dx}


def exact(case, seed):
    kind = case["kind"]
    if kind == "dft":
        return torch.fft.fft(_pulse(case, seed).to(torch.complex128), dim=1)
    if kind == "plan":
        fs, fc, fo, n, fmt = (case[k] for k in ("fs", "fc", "fo", "n", "fmt"))
        x = _samples(fmt, fs, fc, fo, n, seed, case["skew"])
        return _products(_folded_bins(x, fmt, fs, fc, fo, n), n, fs, fc)
    if kind == "batch":
        out = []
        for c, (fs, fc, fo, fmt, n) in enumerate(_mix(case)):
            x = _samples(fmt, fs, fc, fo, n, seed * 1000 + c)
            p = _products(_folded_bins(x, fmt, fs, fc, fo, n), n, fs, fc)
            out.append(np.concatenate([p[k] for k in _parts(np.zeros(0), 0)]))
        return out
    fs, fc, fo, n, fmt = (case[k] for k in ("fs", "fc", "fo", "n", "fmt"))
    x = _samples(fmt, fs, fc, fo, n, seed, folds=False)
    p = _products(_rotated_bins(x, fmt, fs, fc, fo, n), n, fs, fc)
    ph = p["phasors"]
    return {"phasors": ph[0::2] + 1j * ph[1::2], "amp": p["amp"], "phase": p["phase"], "unwrapped": p["unwrapped"],
            "td": float(p["td"][0]), "sigma_td": float(p["sigma_td"][0]), "td_peak": float(p["td_peak"][0]),
            "bandpass_phase": p["bandpass_phase"]}
