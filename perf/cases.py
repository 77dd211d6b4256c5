"""Timed cases of the library: what a program that estimates spectral correlation has it do.

Every case goes through the Python binding as a user's program calls it: single FAM and SSCA
estimates (`scd_fam`, `scd_ssca`) from the smallest to the largest sizes, the (f, alpha) map and the
cycle-frequency profile of an estimate, batches of uneven signals and streams of overlapping windows
(`BatchPlan`, `StreamPlan`).  The program keeps its output tensors, workspaces and plans between
passes, as a receive loop does; the inputs are digitally modulated signals in noise made on the GPU
from the seed.  The split-precision form is not among the cases: it is slower and less accurate than
the FP32 form on every size and is kept for precision studies.

A case is a dict of plain values.  `kind` is one of

  fam     one FAM estimate: Np, L, P, `extra` samples beyond the ones it consumes, `variant`
          ("auto", "cross": against a second signal, "conjugate", "power": normalised input)
  ssca    one SSCA estimate: Np, N, `variant`
  map     one estimate (`estimator`) and its (f, alpha) map and alpha profile, S kept to itself
  batch   `count` signals of lengths log-uniform in [2^lo, 2^hi) through one plan (`estimator`)
  stream  one group of `count` windows of `window` samples every `hop` samples, the new samples
          copied into the arena from the device, alpha profiles as output
"""
import math
import random

import torch

from paper_2506_18003_gb300 import binding

FAM, SSCA = "fam", "ssca"


def listed():
    return [
        # the smallest estimate in use: a short burst; two launches and little else
        {"name": "fam_280", "kind": "fam", "Np": 32, "L": 8, "P": 32, "extra": 0, "variant": "auto"},
        # the size the method's papers time (2048 samples, here with the 2240 it consumes)
        {"name": "fam_2240", "kind": "fam", "Np": 256, "L": 64, "P": 32, "extra": 0, "variant": "auto"},
        # a full-resolution FAM estimate of one capture
        {"name": "fam_65728", "kind": "fam", "Np": 256, "L": 64, "P": 1024, "extra": 0, "variant": "auto"},
        # two receive channels against each other (cross estimate: no symmetry to use)
        {"name": "fam_cross", "kind": "fam", "Np": 128, "L": 32, "P": 2048, "extra": 17, "variant": "cross"},
        # every block of a capture whose block count is not a power of two
        {"name": "fam_p1000", "kind": "fam", "Np": 256, "L": 64, "P": 1000, "extra": 0, "variant": "auto"},
        # an ordinary SSCA estimate
        {"name": "ssca_64k", "kind": "ssca", "Np": 256, "N": 1 << 16, "variant": "auto"},
        # the largest SSCA estimate: full resolution, 2.1 GB of output
        {"name": "ssca_1m", "kind": "ssca", "Np": 256, "N": 1 << 20, "variant": "auto"},
        # a capture of a length that is not a power of two, every sample used
        {"name": "ssca_n100000", "kind": "ssca", "Np": 128, "N": 100000, "variant": "auto"},
        # detection: the estimate is looked at through its map and its cycle-frequency profile
        {"name": "ssca_map", "kind": "map", "estimator": SSCA, "Np": 128, "L": 1, "P": 0, "N": 1 << 17},
        # a data set of uneven signals, FAM and SSCA
        {"name": "fam_batch", "kind": "batch", "estimator": FAM, "Np": 64, "L": 16, "count": 64, "lo": 12.0, "hi": 18.0,
         "lengths_seed": 4},
        {"name": "ssca_batch", "kind": "batch", "estimator": SSCA, "Np": 128, "L": 1, "count": 64, "lo": 12.0,
         "hi": 18.0, "lengths_seed": 4},
        # a live stream: overlapping windows, features (alpha profiles) instead of estimates
        {"name": "ssca_stream", "kind": "stream", "estimator": SSCA, "Np": 64, "L": 1, "window": 1 << 15,
         "hop": 1 << 14, "count": 16},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _hop(rng, Np):
    """The hop: mostly a quarter of the channels, as the method asks, else any up to half of them."""
    return Np // 4 if rng.random() < 0.6 else rng.randint(max(1, Np // 8), Np // 2)


def draw(rng):
    kind = rng.choice(["fam", "fam", "ssca", "ssca", "map", "batch", "stream"])
    Np = rng.choice([16, 32, 64, 64, 128, 128, 256, 256])
    if kind == "fam":
        top = min(8192, (1 << 26) // (Np * Np))
        P = int(_log(rng, 8, top + 1))
        if rng.random() < 0.7:
            P = 1 << (P.bit_length() - 1)
        else:
            P = min(P, 3000)
        return {"kind": kind, "Np": Np, "L": _hop(rng, Np), "P": P, "extra": rng.randint(0, 99),
                "variant": rng.choice(["auto", "auto", "auto", "cross", "conjugate", "power"])}
    if kind == "ssca":
        N = int(_log(rng, 4096, min(1 << 20, (1 << 27) // Np) + 1))
        if rng.random() < 0.7:
            N = 1 << (N.bit_length() - 1)
        else:
            N = min(N, 1 << 18)
        return {"kind": kind, "Np": Np, "N": N,
                "variant": rng.choice(["auto", "auto", "auto", "cross", "conjugate", "power"])}
    if kind == "map":
        if rng.random() < 0.5:
            P = 1 << int(_log(rng, 32, min(4096, (1 << 25) // (Np * Np)) + 1)).bit_length() - 1
            return {"kind": kind, "estimator": FAM, "Np": Np, "L": Np // 4, "P": P, "N": 0}
        N = 1 << int(_log(rng, 4096, (1 << 25) // Np + 1)).bit_length() - 1
        return {"kind": kind, "estimator": SSCA, "Np": Np, "L": 1, "P": 0, "N": min(N, 1 << 20)}
    if kind == "batch":
        Np = rng.choice([32, 64, 128])
        est = rng.choice([FAM, SSCA])
        lo = rng.uniform(12.0, 14.0)
        return {"kind": kind, "estimator": est, "Np": Np, "L": Np // 4 if est == FAM else 1,
                "count": int(_log(rng, 4, 49)), "lo": round(lo, 3), "hi": round(lo + rng.uniform(0.5, 4.0), 3),
                "lengths_seed": rng.randint(0, 9999)}
    window = 1 << rng.randint(12, 16)
    if rng.random() < 0.3:
        window += rng.randint(1, window - 1)
    return {"kind": "stream", "estimator": rng.choice([FAM, SSCA, SSCA]), "Np": rng.choice([32, 64, 128]), "L": 8,
            "window": window, "hop": max(64, int(window * rng.uniform(0.25, 1.0))), "count": rng.randint(4, 24)}


# ---------------------------------------------------------------------------------- inputs
def _signal(n, g):
    """n samples of QPSK with rectangular pulses of 8 samples on a carrier, 10 dB above white noise."""
    sym = torch.randint(0, 4, (n // 8 + 1,), generator=g, device="cuda")
    ph = (sym.double() * 0.5 + 0.25) * math.pi
    t = torch.arange(n, device="cuda", dtype=torch.float64)
    ph = ph.repeat_interleave(8)[:n] + 2.0 * math.pi * torch.remainder(0.0625 * 1.37 * t, 1.0)
    noise = torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(0.05)
    return torch.complex(torch.cos(ph) + noise[:, 0], torch.sin(ph) + noise[:, 1]).to(torch.complex64)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _lengths(case):
    r = random.Random(case["lengths_seed"])
    return [int(2.0 ** r.uniform(case["lo"], case["hi"])) for _ in range(case["count"])]


def _size(case, length):
    """Transform size of one signal of a batch or stream: SSCA N, FAM P."""
    if case["estimator"] == SSCA:
        return min(1 << 20, 1 << (length.bit_length() - 1))
    return min(8192, 1 << (((length - case["Np"]) // case["L"] + 1).bit_length() - 1))


def _kept(case):
    """Signals of a batch or stream: (start, length) in the arena."""
    if case["kind"] == "stream":
        return [(i * case["hop"], case["window"]) for i in range(case["count"])]
    out, at = [], 0
    for n in _lengths(case):
        out.append((at, n))
        at += n
    return out


def _inputs(case, seed):
    """The case's input tensors, a dict."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("batch", "stream"):
        start, length = _kept(case)[-1]
        d = {"x": _signal(start + length, g)}
        if kind == "stream":
            d["new"] = _signal(case["count"] * case["hop"], g)
            # the overlap kept from one group to the next: the same for every pass over this group
            keep = max(case["window"] - case["hop"], 0)
            if keep:
                d["x"][-keep:] = d["new"][-keep:]
        return d
    if kind == "fam":
        n = (case["P"] - 1) * case["L"] + case["Np"] + case["extra"]
    elif kind == "map" and case["estimator"] == FAM:
        n = (case["P"] - 1) * case["L"] + case["Np"]
    else:
        n = case["N"]
    d = {"x": _signal(n, g)}
    if case.get("variant") == "cross":
        d["y"] = _signal(n, g)
    return d


def _options(case):
    v = case.get("variant", "auto")
    return {"conjugate": v == "conjugate", "normalise": "power" if v == "power" else None}


def _bytes(nbytes):
    return torch.empty(max(1, nbytes), dtype=torch.uint8, device="cuda")


def _c64(*shape):
    return torch.empty(shape, dtype=torch.complex64, device="cuda")


def prepare(case, seed):
    lib = binding.load()
    s = dict(_inputs(case, seed), case=case)
    kind, Np = case["kind"], case["Np"]
    if kind in ("batch", "stream"):
        if kind == "batch":
            plan = binding.BatchPlan(case["estimator"], _lengths(case), Np, case["L"])
            s["out"] = _c64(plan.out_offsets[-1])
        else:
            plan = binding.StreamPlan(case["estimator"], case["window"], case["hop"], case["count"], Np, case["L"])
            plan.set_output("profile", 1)
            s["out"] = torch.empty(plan.out_offsets[-1], dtype=torch.float32, device="cuda")
        s["plan"], s["ws"] = plan, _bytes(plan.workspace_bytes)
        # a plan's runs replay a captured graph on a stream of the program's own
        s["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
        return s
    n = s["x"].numel()
    if kind == "fam" or case.get("estimator") == FAM:
        binding.scd_prepare("fam", n, Np, case["P"])
        s["out"] = _c64(Np, Np, case["P"])
        s["ws"] = _bytes(lib.scd_fam_workspace_bytes(n, Np, case["L"], case["P"], binding.SCD_FP32))
        if kind == "map":
            s["map"] = torch.empty((2 * Np, 2 * case["P"] * case["L"]), dtype=torch.float32, device="cuda")
            s["prof"] = torch.empty(2 * case["P"] * case["L"], dtype=torch.float32, device="cuda")
    else:
        binding.scd_prepare("ssca", n, Np)
        s["out"] = _c64(Np, n)
        s["ws"] = _bytes(lib.scd_ssca_workspace_bytes(n, Np, binding.SCD_FP32))
        if kind == "map":
            s["map"] = torch.empty((Np, 2 * n), dtype=torch.float32, device="cuda")
            s["prof"] = torch.empty(2 * n, dtype=torch.float32, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind, Np = case["kind"], case["Np"]
    if kind in ("batch", "stream"):
        # the library's work goes to the plan's stream, in order with the caller's
        st = s["stream"]
        here = torch.cuda.current_stream()
        st.wait_stream(here)
        if kind == "stream":
            s["plan"].advance(s["x"], s["new"], stream=st)
        s["plan"].run(s["x"], s["out"], s["ws"], stream=st)
        here.wait_stream(st)
        return s["out"]
    if kind == "fam":
        return binding.scd_fam(s["x"], Np, case["L"], case["P"], out=s["out"], workspace=s["ws"], y=s.get("y"),
                               **_options(case))
    if kind == "ssca":
        return binding.scd_ssca(s["x"], Np, out=s["out"], workspace=s["ws"], y=s.get("y"), **_options(case))
    if case["estimator"] == FAM:
        L, P = case["L"], case["P"]
        S = binding.scd_fam(s["x"], Np, L, P, out=s["out"], workspace=s["ws"])
        return {"map": binding.scd_fam_map(S, Np, L, P, map=s["map"]),
                "profile": binding.scd_fam_alpha_profile(S, Np, L, P, profile=s["prof"])}
    N = case["N"]
    S = binding.scd_ssca(s["x"], Np, out=s["out"], workspace=s["ws"])
    return {"map": binding.scd_ssca_map(S, N, Np, map=s["map"]),
            "profile": binding.scd_ssca_alpha_profile(S, N, Np, profile=s["prof"])}


# ---------------------------------------------------------------------------------- work
def _fft(m):
    return 5.0 * m * math.log2(m)


def _fam_flops(Np, P, pairs):
    return P * (2 * Np + _fft(Np)) + pairs * (6 * P + _fft(P))


def _ssca_flops(Np, N, auto):
    """Lag products, their N-point transforms (for the auto estimate one for each lag of one sign:
    the other sign's follow by conjugate symmetry) and an Np-point transform per frequency."""
    strips = Np // 2 + 1 if auto else Np
    return strips * (6 * N + _fft(N)) + N * (2 * Np + _fft(Np))


def work(case):
    kind, Np = case["kind"], case["Np"]
    if kind == "fam" or (kind == "map" and case["estimator"] == FAM):
        P, L = case["P"], case["L"]
        auto = case.get("variant", "auto") in ("auto", "power")
        used, out = (P - 1) * L + Np, 8 * Np * Np * P
        flops = _fam_flops(Np, P, Np * (Np + 1) // 2 if auto else Np * Np)
        if kind == "map":                       # S is the program's only intermediate: map and profile come out
            out = 4 * 2 * Np * 2 * P * L + 4 * 2 * P * L
        return {"bytes": 8 * used * (2 if case.get("variant") == "cross" else 1) + out, "flops": flops}
    if kind in ("ssca", "map"):
        N = case["N"]
        auto = case.get("variant", "auto") in ("auto", "power")
        out = 8 * Np * N if kind == "ssca" else 4 * Np * 2 * N + 4 * 2 * N
        return {"bytes": 8 * N * (2 if case.get("variant") == "cross" else 1) + out,
                "flops": _ssca_flops(Np, N, auto)}
    nbytes = flops = 0.0
    for _, length in _kept(case):
        sz = _size(case, length)
        if case["estimator"] == FAM:
            flops += _fam_flops(Np, sz, Np * (Np + 1) // 2)
            nbytes += 8 * Np * Np * sz if kind == "batch" else 8 * sz * case["L"]
            nbytes += 8 * ((sz - 1) * case["L"] + Np) if kind == "batch" else 0
        else:
            flops += _ssca_flops(Np, sz, True)
            nbytes += 8 * Np * sz + 8 * sz if kind == "batch" else 8 * sz
    if kind == "stream":                        # every sample of the group once, the new ones also copied in
        nbytes += 8 * (case["count"] - 1) * case["hop"] + 8 * case["window"] + 8 * case["count"] * case["hop"]
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------- 64-bit values
def _window(Np):
    n = torch.arange(Np, device="cuda", dtype=torch.float64)
    return (0.54 - 0.46 * torch.cos(2.0 * math.pi * n / (Np - 1))).to(torch.float32).double()


def _phase(idx, M):
    return torch.exp(-2j * math.pi * (torch.remainder(idx, M).double() / M))


def _fftshift(v):
    return torch.roll(v, v.shape[-1] // 2, dims=-1)


def _fam64(x, Np, L, P, y=None, conjugate=False):
    k = torch.arange(-Np // 2, Np // 2, device="cuda")
    p = torch.arange(P, device="cuda")

    def demodulates(v):
        blocks = v[: (P - 1) * L + Np].unfold(0, Np, L) * _window(Np)
        spec = torch.roll(torch.fft.fft(blocks, dim=-1), Np // 2, dims=-1)
        return (spec * _phase(p[:, None] * L * k[None, :], Np)).T.contiguous()

    X = demodulates(x)
    Y = X if y is None else demodulates(y)
    Y = Y if conjugate else Y.conj()
    out = torch.empty((Np, Np, P), dtype=torch.complex128, device="cuda")
    for i in range(0, Np, 16):
        out[i:i + 16] = _fftshift(torch.fft.fft(X[i:i + 16, None, :] * Y[None, :, :], dim=-1))
    return out


def _ssca64(x, Np, y=None, conjugate=False):
    N = x.numel()
    y = x if y is None else y
    y = y if conjugate else y.conj()
    k = torch.arange(-Np // 2, Np // 2, device="cuda")
    zero = torch.zeros(Np // 2, dtype=torch.complex128, device="cuda")
    frames = torch.cat([zero, x, zero])[: N + Np - 1].unfold(0, Np, 1)
    out = torch.empty((Np, N), dtype=torch.complex128, device="cuda")
    step = 1 << 16
    for n0 in range(0, N, step):
        n = torch.arange(n0, min(N, n0 + step), device="cuda")
        spec = torch.roll(torch.fft.fft(frames[n0:n0 + step] * _window(Np), dim=-1), Np // 2, dims=-1)
        spec = spec * _phase((n[:, None] - Np // 2) * k[None, :], Np)
        out[:, n0:n0 + step] = (spec * y[n0:n0 + step, None]).T
    for i in range(0, Np, 16):
        out[i:i + 16] = _fftshift(torch.fft.fft(out[i:i + 16], dim=-1))
    return out


def _fam_grid64(S, Np, L, P):
    PL, Q = P * L, P * L // Np
    k = torch.arange(-Np // 2, Np // 2, device="cuda")
    mag = S[:, :, P // 2 - Q:P // 2 + Q].abs()
    q = torch.arange(-Q, Q, device="cuda")
    fh = (k[:, None] + k[None, :] + Np)[:, :, None].expand(Np, Np, 2 * Q)
    ah = (k[:, None] - k[None, :])[:, :, None] * Q + q + PL
    grid = torch.zeros((2 * Np, 2 * PL), dtype=torch.float64, device="cuda")
    grid[fh, ah] = mag
    return grid


def _ssca_grid64(S, Np):
    N = S.shape[-1]
    k = torch.arange(-Np // 2, Np // 2, device="cuda")[:, None] * (N // Np)
    q = torch.arange(-N // 2, N // 2, device="cuda")[None, :]
    grid = torch.zeros((Np, 2 * N), dtype=torch.float64, device="cuda")
    grid[torch.div(k - q + N, 2 * (N // Np), rounding_mode="floor"), k + q + N] = S.abs()
    return grid


def exact(case, seed):
    d = _inputs(case, seed)
    kind, Np = case["kind"], case["Np"]
    x = d["x"].to(torch.complex128)
    if kind in ("batch", "stream"):
        if kind == "stream":
            # the advance keeps the samples behind the group's last hop and appends the new ones
            keep = max(case["window"] - case["hop"], 0)
            x = torch.cat([x[x.numel() - keep:], d["new"].to(torch.complex128)[: x.numel() - keep]])
        parts = []
        for start, length in _kept(case):
            sz = _size(case, length)
            v = x[start:start + length]
            S = _fam64(v, Np, case["L"], sz) if case["estimator"] == FAM else _ssca64(v[:sz], Np)
            if kind == "batch":
                parts.append(S.reshape(-1))
            else:
                grid = _fam_grid64(S, Np, case["L"], sz) if case["estimator"] == FAM else _ssca_grid64(S, Np)
                parts.append(grid.amax(dim=0))
        return torch.cat(parts)
    if kind == "map":
        if case["estimator"] == FAM:
            grid = _fam_grid64(_fam64(x, Np, case["L"], case["P"]), Np, case["L"], case["P"])
        else:
            grid = _ssca_grid64(_ssca64(x, Np), Np)
        return {"map": grid, "profile": grid.amax(dim=0)}
    y = d["y"].to(torch.complex128) if "y" in d else None
    conj = case["variant"] == "conjugate"
    if kind == "fam":
        S = _fam64(x, Np, case["L"], case["P"], y, conj)
        used = (case["P"] - 1) * case["L"] + Np
    else:
        S = _ssca64(x, Np, y, conj)
        used = case["N"]
    if case["variant"] == "power":
        S = S / x[:used].abs().square().mean()
    return S
