"""The work that users of this correlator have it do, as timed cases.

Each pass goes through the public entry points of paper_0909_0001_gb300.omni: a
plan accumulates a block of voltages and gives the visibilities of one
integration (with the radial profile where a case asks for it), or the F-engine
channelises a block of raw samples.

Visibilities are handed on as complex64, the type in which they are stored and
imaged (UVFITS and Measurement Set visibilities are pairs of 32-bit floats): the
transforms behind them run in FP32 or in split 16-bit products, and the
library's complex128 is the type of its time accumulator.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0909_0001_gb300 import omni, synth

SPEED_OF_LIGHT = 299_792_458.0


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one 16 x 16 array, one channel, a short snapshot; a
        # monitoring loop that waits for every result
        dict(name="grid16", kind="plan", levels="16x16", channels=1, samples=64, dtype="cf32",
             precision="fp32", profile=False),
        # the benchmark hierarchy (64 blocks of 16 x 16 antennas) in plain FP32, with
        # the radial profile of the baselines that a beam designer looks at
        dict(name="hier2_fp32", kind="plan", levels="16x16,8x8", channels=64, samples=1024, dtype="ci8",
             precision="fp32", profile=True),
        # the same in the mixed precision meant for production
        dict(name="hier2_mixed", kind="plan", levels="16x16,8x8", channels=64, samples=1024, dtype="ci8",
             precision="mixed", profile=False),
        # the same from host memory, as a station's receiver process feeds it
        dict(name="hier2_host", kind="host", levels="16x16,8x8", channels=16, samples=1024, dtype="ci8",
             precision="mixed", profile=False),
        # three levels, 262144 antennas, float voltages
        dict(name="hier3_fp32", kind="plan", levels="16x16,8x8,4x4", channels=8, samples=64, dtype="cf32",
             precision="fp32", profile=False),
        # the largest single grid, a million antennas, axes of 2048 points
        dict(name="grid1024", kind="plan", levels="1024x1024", channels=16, samples=64, dtype="cf32",
             precision="fp32", profile=False),
        # many independent arrays of uneven shapes in one plan
        dict(name="batch48", kind="batch", arrays=48, layout=9090004, channels=16, samples=512, dtype="ci8",
             precision="fp32"),
        # beam-space correlation (digital pointings of each block)
        dict(name="beams64", kind="beams", levels="16x16,8x8", channels=64, samples=1024, dtype="ci8"),
        # tiles at arbitrary places, correlated pairwise, in FP32
        dict(name="tiles64_fp32", kind="tiles", levels="16x16", tiles=64, channels=8, samples=1024, dtype="ci8",
             precision="fp32"),
        # tiles of a size that is no power of two, ragged sample count, float
        # voltages, mixed precision
        dict(name="tiles50_mixed", kind="tiles", levels="12x12", tiles=50, channels=16, samples=500, dtype="cf32",
             precision="mixed"),
        # the channeliser in front of the benchmark hierarchy: 64 channels, int8 out
        dict(name="fengine64", kind="fengine", antennas=16384, channels=64, taps=4, frames=1024, extra=0,
             dtype="ci8", gains=False, scale=20.0),
        # a fine channeliser for a smaller station: 1024 channels, calibrated floats out
        dict(name="fengine1024", kind="fengine", antennas=1000, channels=1024, taps=8, frames=200, extra=640,
             dtype="cf32", gains=True, scale=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels_samples(rng, antennas, padded, budget, most_channels=64):
    """Channels x samples, logarithmically spread, within a budget of padded lattice points."""
    points = max(1, int(budget // padded))
    samples = max(2, min(points, _log_int(rng, 4, 1024)))
    channels = max(1, min(points // samples, _log_int(rng, 1, most_channels)))
    return channels, samples


def draw(rng):
    """One more case of the listed kinds."""
    kind = rng.choice(["plan", "plan", "plan", "mixed", "mixed", "host", "batch", "beams", "tiles", "tiles",
                       "fengine", "fengine"])
    dtype = rng.choice(["cf32", "ci8"])
    if kind in ("plan", "mixed", "host", "beams"):
        precision = "fp32" if kind in ("plan", "beams") else rng.choice(["mixed", "mixed", "mixed_bf16"])
        side = lambda lo, hi: rng.choice([rng.randint(lo, hi), 1 << rng.randint(int(math.log2(lo)) + 1, int(math.log2(hi)))])
        if kind == "plan":
            depth = rng.choice([1, 1, 2, 2, 3])
            if depth == 1:
                shape = [(rng.choice([rng.randint(4, 48), 1 << rng.randint(2, 10)]), 1 << rng.randint(2, 9))]
                if rng.random() < 0.5:
                    shape[0] = shape[0][::-1]
            elif depth == 2:
                shape = [(side(3, 32), side(3, 32)), (side(2, 16), side(2, 16))]
            else:
                shape = [(side(3, 16), side(3, 16)), (side(2, 8), side(2, 8)), (side(1, 4), side(1, 4))]
        elif kind == "beams":
            s = 1 << rng.randint(1, 4)
            shape = [(s, rng.choice([s, 1 << rng.randint(1, 4)])), (side(2, 16), side(2, 16))]
        else:
            a = rng.choice([(16, 16), (16, 16), (8, 8), (4, 4), (2 * rng.randint(1, 10), rng.randint(1, 20))])
            shape = [a, (rng.randint(2, 8), rng.randint(1, 8))]
        antennas = math.prod(a * b for a, b in shape)
        padded = math.prod((2 * s if s > 1 else 1) for ab in shape for s in ab)
        # at most the padded points of the listed hierarchies (the mixed path pads level 1 alone)
        C, T = _channels_samples(rng, antennas, padded, 2.0 ** 32 if kind == "plan" else 2.0 ** 33)
        return dict(kind="host" if kind == "host" else "beams" if kind == "beams" else "plan",
                    levels=",".join("%dx%d" % s for s in shape), channels=C, samples=T, dtype=dtype,
                    **({} if kind == "beams" else dict(precision=precision, profile=rng.random() < 0.3)))
    if kind == "batch":
        n = _log_int(rng, 3, 48)
        return dict(kind="batch", arrays=n, layout=rng.randint(1, 10 ** 6), channels=_log_int(rng, 1, 16),
                    samples=_log_int(rng, 16, 512), dtype=dtype, precision="fp32")
    if kind == "tiles":
        precision = rng.choice(["fp32", "mixed", "mixed_bf16"])
        a = rng.choice([(16, 16), (8, 8), (4, 4), (2 * rng.randint(1, 8), rng.randint(2, 16))])
        n = _log_int(rng, 4, 64 if precision != "fp32" else 96)
        C, T = _channels_samples(rng, n * a[0] * a[1], n * 4 * a[0] * a[1] * max(1.0, n / 64), 2.0 ** 29, 16)
        return dict(kind="tiles", levels="%dx%d" % a, tiles=n, channels=C, samples=T, dtype=dtype, precision=precision)
    F = 1 << rng.randint(2, 12)
    N = _log_int(rng, 8, 4096)
    T = max(4, min(2048, int(2.0 ** 28 / (N * F) * rng.uniform(0.05, 1.0))))
    return dict(kind="fengine", antennas=N, channels=F, taps=rng.choice([1, 2, 4, 4, 8, 8, 12]), frames=T,
                extra=rng.choice([0, 0, 16, rng.randint(1, 2 * F - 1)]), dtype=dtype, gains=rng.random() < 0.5,
                scale=20.0 if dtype == "ci8" else 1.0)


# ------------------------------------------------------------------ inputs

def _shape(text):
    return [tuple(int(v) for v in ab.split("x")) for ab in text.split(",")]


def _levels(case):
    """Rotated and sheared levels, each block clear of its neighbours."""
    shape = _shape(case["levels"])
    theta = [0.0, math.radians(30.0), math.radians(75.0)]
    shear = [0.0, 0.2, -0.1]
    return synth.hierarchy(shape, theta[:len(shape)], shear[:len(shape)])


def _positions(levels):
    """r = sum_k A_k m_k of every antenna, float64 [N][2], first axis fastest."""
    r = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
    for lv in levels:
        A = torch.tensor(lv.A, dtype=torch.float64, device="cuda").reshape(2, 2)
        b, a = torch.meshgrid(torch.arange(lv.n2, dtype=torch.float64, device="cuda"),
                              torch.arange(lv.n1, dtype=torch.float64, device="cuda"), indexing="ij")
        block = torch.stack([a.reshape(-1), b.reshape(-1)], dim=1) @ A.T
        r = (block[:, None, :] + r[None, :, :]).reshape(-1, 2)
    return r


def _voltages(r, C, T, dtype, seed):
    """[C][T][N][2]: receiver noise and five point sources, 100-200 MHz."""
    N = r.shape[0]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sigma, source = (20.0, 10.0) if dtype == "ci8" else (1.0, 0.5)
    radius = torch.rand(5, generator=gen, device="cuda", dtype=torch.float64).sqrt()
    phi = torch.rand(5, generator=gen, device="cuda", dtype=torch.float64) * (2 * math.pi)
    phase = r @ torch.stack([radius * torch.cos(phi), radius * torch.sin(phi)])     # [N][5], metres
    out = torch.empty((C, T, N, 2), device="cuda", dtype=torch.int8 if dtype == "ci8" else torch.float32)
    for c in range(C):
        per_metre = 2 * math.pi * (1e8 + 1e8 * c / max(1, C - 1)) / SPEED_OF_LIGHT
        wave = torch.polar(torch.ones_like(phase), phase * per_metre).to(torch.complex64)
        amp = torch.randn((T, 5, 2), generator=gen, device="cuda") * source
        x = torch.randn((T, N, 2), generator=gen, device="cuda")
        x.mul_(sigma).add_(torch.view_as_real(torch.view_as_complex(amp) @ wave.T))
        if dtype == "ci8":
            x.round_().clamp_(-127, 127)
        out[c] = x
    return out


def _arrays(case):
    return synth.batch_arrays(case["arrays"], case["layout"])


def _offsets(case, seed):
    """Tile centres scattered over a field, no two tiles touching."""
    n1, n2 = _shape(case["levels"])[0]
    n = case["tiles"]
    g = int(math.ceil(math.sqrt(n)))
    rng = np.random.default_rng(seed)
    at = np.array([(i % g, i // g) for i in range(n)], dtype=np.float64) * (2.0 * max(n1, n2) + 4.0)
    return at + rng.uniform(0.0, 2.0, at.shape)


def _tile(case):
    n1, n2 = _shape(case["levels"])[0]
    return synth.Level(n1, n2)


def _window(case):
    """Hann x sinc prototype of the polyphase filter bank, [taps * 2F] float32."""
    P, M = case["taps"], 2 * case["channels"]
    w = np.hanning(P * M + 2)[1:-1] * np.sinc(np.linspace(-P / 2, P / 2, P * M))
    return w.astype(np.float32)


def _fengine_inputs(case, seed):
    N, F, P = case["antennas"], case["channels"], case["taps"]
    M = 2 * F
    S = (case["frames"] + P - 1) * M + case["extra"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    raw = torch.empty((N, S), device="cuda", dtype=torch.int8)
    tone = 12.0 * torch.cos(0.37 * math.pi * torch.arange(S, device="cuda", dtype=torch.float32))
    rows = max(1, (1 << 28) // S)
    for a in range(0, N, rows):
        x = torch.randn((min(rows, N - a), S), generator=gen, device="cuda")
        raw[a:a + rows] = x.mul_(20.0).add_(tone).round_().clamp_(-127, 127)
    w = _window(case)
    # unit gain for the noise: its channel voltages come out with the standard deviation scale
    scale = float(case["scale"] / (20.0 * math.sqrt(0.5 * float((w.astype(np.float64) ** 2).sum()))))
    gains = None
    if case["gains"]:
        gains = torch.polar(0.8 + 0.4 * torch.rand((F, N), generator=gen, device="cuda"),
                            2 * math.pi * torch.rand((F, N), generator=gen, device="cuda"))
    return raw, torch.from_numpy(w).cuda(), gains, scale


def _profile_bins(levels):
    """Width and number of the radial bins: about 300 out to the longest baseline."""
    r = sum(math.hypot(lv.A[0], lv.A[2]) * lv.n1 + math.hypot(lv.A[1], lv.A[3]) * lv.n2 for lv in levels)
    return r / 300.0, 301


def _inputs(case, seed):
    if case["kind"] == "batch":
        parts = [_voltages(_positions(lv), case["channels"], case["samples"], case["dtype"], seed + 101 * i)
                 for i, lv in enumerate(_arrays(case))]
        return parts
    if case["kind"] == "tiles":
        off = torch.from_numpy(_offsets(case, case["tiles"])).cuda()
        r = (off[:, None, :] + _positions([_tile(case)])[None, :, :]).reshape(-1, 2)
        return _voltages(r, case["channels"], case["samples"], case["dtype"], seed)
    return _voltages(_positions(_levels(case)), case["channels"], case["samples"], case["dtype"], seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        raw, window, gains, scale = _fengine_inputs(case, seed)
        N, F, T = case["antennas"], case["channels"], case["frames"] + case["extra"] // (2 * case["channels"])
        need = omni.load().omni_fengine_scratch_bytes(N, raw.shape[1], F, case["taps"])
        return dict(kind=kind, raw=raw, window=window, gains=gains, scale=scale, F=F, taps=case["taps"],
                    dtype=case["dtype"], scratch=torch.empty(max(1, need // 8), dtype=torch.float64, device="cuda"),
                    out=torch.empty((F, T, N, 2), device="cuda",
                                    dtype=torch.int8 if case["dtype"] == "ci8" else torch.float32))
    C, dtype = case["channels"], case["dtype"]
    x = _inputs(case, seed)
    state = dict(kind=kind)
    if kind == "batch":
        plan = omni.BatchPlan(_arrays(case), C, dtype=dtype, precision=case["precision"])
        x = plan.pack(x)
        shape = (C * plan.n_lags,)
    else:
        if kind == "beams":
            plan = omni.BeamPlan(_levels(case), C, dtype=dtype)
        elif kind == "tiles":
            plan = omni.TilePlan(_tile(case), _offsets(case, case["tiles"]), C, dtype=dtype,
                                 precision=case["precision"])
        else:
            plan = omni.Plan(_levels(case), C, dtype=dtype, precision=case["precision"])
        shape = (C, plan.n_lags)
    if kind == "host":
        x = torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
    if case.get("profile"):
        levels = _levels(case)
        width, n = _profile_bins(levels)
        state.update(bins=torch.from_numpy(omni.radial_bins(levels, width, n)[0]).cuda(), n_bins=n,
                     radial=torch.empty((C, n), dtype=torch.complex128, device="cuda"))
    state.update(plan=plan, x=x, vis=torch.empty(shape, dtype=torch.complex128, device="cuda"))
    return state


# ------------------------------------------------------------------ one pass

def run(state):
    if state["kind"] == "fengine":
        return omni.fengine(state["raw"], state["F"], state["taps"], window=state["window"], gains=state["gains"],
                            scale=state["scale"], dtype=state["dtype"], out=state["out"], scratch=state["scratch"])
    plan = state["plan"]
    if state["kind"] == "host":
        plan.correlate_host(state["x"])
    else:
        plan.correlate(state["x"])
    vis = plan.visibilities(reset=True, out=state["vis"])
    if "bins" in state:
        radial = omni.sum_groups(vis, state["bins"], state["n_bins"], out=state["radial"])
        return vis.to(torch.complex64), radial.to(torch.complex64)
    return vis.to(torch.complex64)


# ------------------------------------------------------------------ the work of a pass

def _fft_work(dims, lags=True, unpadded=0):
    """(flops per sample, padded points): the zero-padded transforms of a lattice,
    axis by axis, the lines that are all zero left out, and |F|^2 where `lags`."""
    flops, done = 0.0, 1.0
    for d, n in enumerate(dims):
        L = n if d < unpadded or n == 1 else 2 * n
        lines = done * math.prod(dims[d + 1:])
        flops += lines * 5.0 * L * math.log2(max(L, 2)) * (L > 1)
        done *= L
    return flops + (3.0 * done if lags else 0.0), done


def work(case):
    kind = case["kind"]
    eb = 2 if case["dtype"] == "ci8" else 8
    if kind == "fengine":
        N, F, P, T = case["antennas"], case["channels"], case["taps"], case["frames"]
        S = (T + P - 1) * 2 * F + case["extra"]
        flops = N * T * (2.0 * P * 2 * F + 2.5 * 2 * F * math.log2(2 * F) + 8.0 * F)
        return dict(bytes=float(N) * S + float(N) * T * F * eb + 4.0 * P * 2 * F + (8.0 * F * N if case["gains"] else 0),
                    flops=flops)
    C, T = case["channels"], case["samples"]
    if kind == "batch":
        total = dict(bytes=0.0, flops=0.0)
        for lv in _arrays(case):
            dims = [n for x in lv for n in (x.n1, x.n2)]
            total["bytes"] += C * (T * math.prod(dims) * eb + 16.0 * math.prod(2 * n - 1 for n in dims))
            total["flops"] += C * T * _fft_work(dims)[0]
        return total
    dims = [n for s in _shape(case["levels"]) for n in s]
    N, Q = math.prod(dims), math.prod(2 * n - 1 for n in dims)
    if kind == "tiles":
        n = case["tiles"]
        flops, K = _fft_work(dims, lags=False)
        # every pair once: S_ji is the conjugate of S_ij
        return dict(bytes=C * (T * n * N * eb + 16.0 * n * n * Q), flops=C * T * (n * flops + 8.0 * K * n * (n + 1) / 2))
    if kind == "beams":
        Q = dims[0] * dims[1] * math.prod(2 * n - 1 for n in dims[2:])
        return dict(bytes=C * (T * N * eb + 16.0 * Q), flops=C * T * _fft_work(dims, unpadded=2)[0])
    profile = 20.0 * Q if case.get("profile") else 0.0
    return dict(bytes=C * (T * N * eb + 16.0 * Q + profile), flops=C * T * _fft_work(dims)[0])


# ------------------------------------------------------------------ the same in 64 bits

def _complex(x):
    return torch.view_as_complex(x.to(torch.float64))


def _keep_lags(G, axes, dims):
    """Along each axis, lags -(n-1) .. n-1 of a padded transform."""
    for ax, n in zip(axes, dims):
        if n > 1:
            lag = torch.arange(-(n - 1), n, device=G.device)
            G = G.index_select(ax, lag % (2 * n))
    return G


def _correlate64(x, dims, unpadded=0):
    """[C][T][N][2] -> [C][lags] complex128 by padded FFTs; the first `unpadded`
    axes are transformed at their own length and not correlated over."""
    C, T = x.shape[:2]
    D = len(dims)
    pad = [n if d < unpadded or n == 1 else 2 * n for d, n in enumerate(dims)]
    axis = {d: D - d for d in range(D)}                      # the axis of dimension d in [t][n_{D-1}] .. [n_0]
    block = max(1, int(2 ** 27 // math.prod(pad)))
    out = []
    for c in range(C):
        P = torch.zeros([1] + pad[::-1], dtype=torch.float64, device=x.device)
        for t0 in range(0, T, block):
            F = _complex(x[c, t0:t0 + block]).reshape([-1] + list(dims[::-1]))
            for d in range(D):
                if pad[d] > 1:
                    F = torch.fft.fft(F, n=pad[d], dim=axis[d])
            P += (F.real.square() + F.imag.square()).sum(dim=0, keepdim=True)
        G = P.to(torch.complex128)
        for d in range(unpadded, D):
            if pad[d] > 1:
                G = torch.fft.ifft(G, dim=axis[d])
        G = _keep_lags(G, [axis[d] for d in range(unpadded, D)], dims[unpadded:])
        out.append(G.reshape(1, -1))
    return torch.cat(out)


def _tiles64(x, dims, n):
    """Every ordered tile pair's cross-correlation, [C][n * n * lags] complex128."""
    n1, n2 = dims
    C, T = x.shape[:2]
    L1, L2 = (2 * n1 if n1 > 1 else 1), (2 * n2 if n2 > 1 else 1)
    out = []
    for c in range(C):
        S = torch.zeros((L1 * L2, n, n), dtype=torch.complex128, device=x.device)
        block = max(1, int(2 ** 26 // (n * L1 * L2)))
        for t0 in range(0, T, block):
            Y = torch.fft.fft2(_complex(x[c, t0:t0 + block]).reshape(-1, n, n2, n1), s=(L2, L1))
            Y = Y.reshape(-1, n, L1 * L2).permute(2, 1, 0)   # [k][tile][t]
            S += Y @ Y.conj().transpose(1, 2)
        G = torch.fft.ifft2(S.permute(1, 2, 0).reshape(n, n, L2, L1))
        out.append(_keep_lags(G, [3, 2], dims).reshape(1, -1))
    return torch.cat(out)


def _fengine64(case, seed):
    if case["dtype"] == "ci8":
        return None                                           # rounded codes: no 64-bit value
    raw, window, gains, scale = _fengine_inputs(case, seed)
    N, F, P = case["antennas"], case["channels"], case["taps"]
    M = 2 * F
    T = (raw.shape[1] - (P - 1) * M) // M
    w = window.to(torch.float64).reshape(P, M)
    out = torch.empty((F, T, N, 2), dtype=torch.float64, device="cuda")
    rows = max(1, int(2 ** 26 // (T * M)))
    for a in range(0, N, rows):
        r = raw[a:a + rows, :(T + P - 1) * M].to(torch.float64).reshape(-1, T + P - 1, M)
        u = sum(w[p] * r[:, p:p + T] for p in range(P))
        X = torch.fft.rfft(u, dim=2)[:, :, :F].permute(2, 1, 0) * scale
        if gains is not None:
            X = X * gains[:, a:a + rows].to(torch.complex128)[:, None, :]
        out[:, :, a:a + rows] = torch.view_as_real(X)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        return _fengine64(case, seed)
    x = _inputs(case, seed)
    if kind == "batch":
        return torch.cat([_correlate64(v, [n for l in lv for n in (l.n1, l.n2)]).reshape(-1)
                          for v, lv in zip(x, _arrays(case))])
    dims = [n for s in _shape(case["levels"]) for n in s]
    if kind == "tiles":
        return _tiles64(x, dims, case["tiles"])
    vis = _correlate64(x, dims, unpadded=2 if kind == "beams" else 0)
    if not case.get("profile"):
        return vis
    # the sums of the lags at floor(|dr| / width), as a plain histogram
    levels = _levels(case)
    dr = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
    for lv in levels:
        A = torch.tensor(lv.A, dtype=torch.float64, device="cuda").reshape(2, 2)
        b, a = torch.meshgrid(torch.arange(1 - lv.n2, lv.n2, dtype=torch.float64, device="cuda"),
                              torch.arange(1 - lv.n1, lv.n1, dtype=torch.float64, device="cuda"), indexing="ij")
        dr = ((torch.stack([a.reshape(-1), b.reshape(-1)], dim=1) @ A.T)[:, None, :] + dr[None, :, :]).reshape(-1, 2)
    width, n = _profile_bins(levels)
    b = torch.floor(torch.hypot(dr[:, 0], dr[:, 1]) / width).to(torch.int64)
    keep = b < n
    radial = torch.zeros((vis.shape[0], n), dtype=torch.complex128, device="cuda")
    radial.index_add_(1, b[keep], vis[:, keep])
    return vis, radial
