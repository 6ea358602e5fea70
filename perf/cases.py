"""Performance cases: what programs that use this library have it do.

A case is one pass through the public entry points of
``paper_1101_0086_gb300.mpa`` on seeded synthetic WDM fields and the
benchmark's dispersion-managed fiber maps.  ``listed()`` gives the named
cases, ``draw(rng)`` further ones of the same ranges, ``prepare`` what a
program holds before the call (field, plan or batch, workspace), ``run`` the
pass itself, ``work`` the bytes and operations a pass cannot do without, and
``exact`` the result in 64-bit torch arithmetic.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1101_0086_gb300 import mpa
from paper_1101_0086_gb300.workloads import FiberMap, Segment, batch_links, dm_map

DEVICE = "cuda"
SPACING_GHZ = {16: 50.0, 8: 50.0, 4: 50.0, 2: 50.0, 64: 25.0}
FWHM_PS, SLOT_PS = 30.0, 100.0


# ------------------------------------------------------------------ cases
def listed():
    return [
        # The spectrum of a short field, as a program looks at it between
        # propagations: a call of a few microseconds.
        {"name": "fft_n12", "kind": "fft", "prec": "fp32", "log2n": 12, "sign": 1},
        # One span of the shortest link of a batch study, propagated by itself
        # in a loop over links or powers.
        {"name": "link_n12", "kind": "link", "prec": "fp32", "log2n": 12, "spp": 256, "channels": 8, "peak_mw": 2.0,
         "ook": False, "z0": 0.0, "L": 5.0, "M": 142, "n_iter": 3, "intervals": 10, "tune": False},
        # The 4-channel OOK link over its whole 200 km (four intervals of a span).
        {"name": "link_n14_ook_200km", "kind": "link", "prec": "fp32", "log2n": 14, "spp": 128, "channels": 4,
         "peak_mw": 1.0, "ook": True, "z0": 0.0, "L": 50.0, "M": 800, "n_iter": 3, "intervals": 4, "tune": False},
        # One span of a mid-size link of a batch study on a tuned plan.
        {"name": "link_n16", "kind": "link", "prec": "fp32", "log2n": 16, "spp": 256, "channels": 16, "peak_mw": 2.0,
         "ook": False, "z0": 0.0, "L": 5.0, "M": 142, "n_iter": 3, "intervals": 10, "tune": True},
        # The 16-channel QPSK link of the benchmark, one of its 40 spans.
        {"name": "link_n20_span", "kind": "link", "prec": "fp32", "log2n": 20, "spp": 1024, "channels": 16,
         "peak_mw": 2.0, "ook": False, "z0": 0.0, "L": 5.0, "M": 125, "n_iter": 2, "intervals": 10, "tune": True},
        # The 64-channel link, the interval behind its dispersion jump.
        {"name": "link_n24", "kind": "link", "prec": "fp32", "log2n": 24, "spp": 8192, "channels": 64, "peak_mw": 2.0,
         "ook": False, "z0": 45.0, "L": 5.0, "M": 142, "n_iter": 4, "intervals": 1, "tune": True},
        # The FP64 run that an FP32 result is checked against.
        {"name": "link_n18_fp64", "kind": "link", "prec": "fp64", "log2n": 18, "spp": 1024, "channels": 16,
         "peak_mw": 2.0, "ook": False, "z0": 40.0, "L": 5.0, "M": 125, "n_iter": 2, "intervals": 2, "tune": False},
        # Independent links of different sizes, powers and lengths in one call.
        {"name": "batch_24", "kind": "batch", "links": 24, "log2n_min": 12, "log2n_max": 16, "spans_max": 2, "mix": 3,
         "L": 5.0, "M": 142, "n_iter": 3},
        # One step of fitting a link's input and coefficients: forward, loss and
        # gradients over 10 km that hold the dispersion jump and an amplifier.
        {"name": "grad_n20", "kind": "grad", "log2n": 20, "spp": 2048, "channels": 16, "peak_mw": 2.0, "z0": 40.0,
         "L": 5.0, "M": 142, "n_iter": 2, "intervals": 2},
        # The split-step of the 4-channel OOK link, a tenth of a span.
        {"name": "ss_n14", "kind": "ss", "prec": "fp32", "log2n": 14, "spp": 128, "channels": 4, "peak_mw": 1.0,
         "ook": True, "z0": 0.0, "dz": 0.1, "steps": 50},
        # The FP64 split-step reference of the 16-channel link, 5 km across the jump.
        {"name": "ss_n20_fp64", "kind": "ss", "prec": "fp64", "log2n": 20, "spp": 1024, "channels": 16,
         "peak_mw": 2.0, "ook": False, "z0": 42.5, "dz": 0.05, "steps": 100},
        # Gradients through the FP32 split-step across the jump.
        {"name": "ss_grad_n20", "kind": "ss_grad", "log2n": 20, "spp": 2048, "channels": 16, "peak_mw": 2.0,
         "z0": 44.25, "dz": 0.05, "steps": 30},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: every kind in turn of chance, sizes over the listed
    ranges (field lengths are powers of two; node, step, interval and link
    counts are any number)."""
    kind = rng.choice(["fft", "link", "link", "link", "link64", "batch", "grad", "ss", "ss", "ss_grad"])
    if kind == "fft":
        return {"kind": "fft", "prec": rng.choice(["fp32", "fp64"]), "log2n": rng.randint(9, 22),
                "sign": rng.choice([1, -1])}
    spp = rng.choice([128, 256, 512, 1024])
    peak = round(rng.uniform(0.5, 4.0), 3)
    if kind in ("link", "link64"):
        f64 = kind == "link64"
        log2n = rng.randint(12, 19 if f64 else 22)
        channels = rng.choice([2, 4, 8, 16])
        L = rng.choice([2.5, 5.0, 5.0, 10.0])
        if channels <= 4 and peak <= 1.5:
            L = rng.choice([10.0, 25.0, 50.0])
        M = max(8, int(round(L / math.exp(rng.uniform(math.log(0.03), math.log(0.08))))))
        n_iter = rng.randint(2, 4)
        # node spectra of a pass: at most the largest listed case's, a tenth of it in FP64
        most = (2.0 ** 24 * 143 * 4) / (10.0 if f64 else 1.0)
        cap = max(1, int(0.8 * most / (2.0 ** log2n * (M + 1) * n_iter)))
        intervals = min(cap, _log_int(rng, 1, 20), int(100.0 / L))
        while intervals > 1 and 2.0 ** log2n * (M + 1) * n_iter * intervals > 0.8 * most:
            intervals -= 1
        z0 = L * rng.randint(0, int(100.0 / L) - intervals)
        return {"kind": "link", "prec": "fp64" if f64 else "fp32", "log2n": log2n, "spp": spp, "channels": channels,
                "peak_mw": peak, "ook": rng.random() < 0.25, "z0": z0, "L": L, "M": M, "n_iter": n_iter,
                "intervals": intervals, "tune": rng.random() < 0.5}
    if kind == "batch":
        lo = rng.randint(11, 14)
        return {"kind": "batch", "links": rng.randint(3, 40), "log2n_min": lo, "log2n_max": rng.randint(lo, 16),
                "spans_max": rng.randint(1, 2), "mix": rng.randint(0, 10 ** 6), "L": 5.0, "M": rng.randint(90, 160),
                "n_iter": rng.randint(2, 3)}
    if kind == "grad":
        log2n = rng.randint(13, 20)
        M = rng.randint(60, 160)
        intervals = rng.randint(1, 2) if log2n > 18 else rng.randint(1, 3)
        return {"kind": "grad", "log2n": log2n, "spp": rng.choice([256, 1024, 2048]), "channels": rng.choice([4, 8, 16]),
                "peak_mw": peak, "z0": 50.0 - 5.0 * intervals, "L": 5.0, "M": M, "n_iter": rng.randint(2, 3),
                "intervals": intervals}
    if kind == "ss":
        f64 = rng.random() < 0.5
        steps = _log_int(rng, 20, 400) if f64 else _log_int(rng, 15, 60)
        log2n = rng.randint(12, 20 if f64 else 22)
        return {"kind": "ss", "prec": "fp64" if f64 else "fp32", "log2n": log2n, "spp": spp,
                "channels": rng.choice([2, 4, 8, 16]), "peak_mw": peak, "ook": rng.random() < 0.25, "z0": 40.0,
                "dz": 0.05, "steps": steps}
    return {"kind": "ss_grad", "log2n": rng.randint(13, 20), "spp": rng.choice([256, 1024, 2048]),
            "channels": rng.choice([4, 8, 16]), "peak_mw": peak, "z0": 44.25, "dz": 0.05, "steps": _log_int(rng, 8, 30)}


# ----------------------------------------------------------------- inputs
def _wdm(log2n, spp, channels, peak_mw, ook, seed):
    """A WDM pulse train (complex128, on the GPU): per channel one Gaussian RZ
    pulse of 30 ps FWHM per 100-ps slot, OOK bits or QPSK symbols."""
    N = 1 << log2n
    slots = N // spp
    T = SLOT_PS * slots
    rng = np.random.Generator(np.random.PCG64(seed))
    t0 = FWHM_PS / (2.0 * math.sqrt(math.log(2.0)))
    x = torch.arange(spp, dtype=torch.float64, device=DEVICE) * (SLOT_PS / spp) - 0.5 * SLOT_PS
    reach = range(-2, 3)  # pulse tails beyond two slots are below 1e-15
    shapes = torch.stack([torch.exp(-((x + d * SLOT_PS) ** 2) / (2.0 * t0 * t0)) for d in reach]).to(torch.complex128)
    n = torch.arange(N, dtype=torch.int64, device=DEVICE)
    field = torch.zeros(N, dtype=torch.complex128, device=DEVICE)
    spacing = SPACING_GHZ[channels] * 1e-3
    for c in range(channels):
        sym = rng.integers(0, 2, slots).astype(np.complex128) if ook else np.exp(0.5j * np.pi * rng.integers(0, 4, slots))
        taps = np.stack([np.roll(sym, d) for d in reach], axis=1)
        train = (torch.from_numpy(taps).to(DEVICE) @ shapes).reshape(N)
        cycles = int(round((c - 0.5 * (channels - 1)) * spacing * T))  # whole cycles of the window
        turn = ((n * cycles) % N).to(torch.float64) * (-2.0 * math.pi / N)
        field += train * torch.polar(torch.ones_like(turn), turn)
    return field * math.sqrt(peak_mw * 1e-3), T


def _dtype(prec):
    return torch.complex64 if prec == "fp32" else torch.complex128


def _fiber(case):
    return dm_map(4, beta3=0.08 if case.get("channels") == 64 else 0.1)


def _links(case):
    return batch_links(case["links"], seed=case["mix"], log2_n=(case["log2n_min"], case["log2n_max"]),
                       spans=(1, case["spans_max"]))


def _field(case, seed):
    return _wdm(case["log2n"], case["spp"], case["channels"], case["peak_mw"], case.get("ook", False), seed)


def _link_fields(case, seed):
    return [_wdm(k.N.bit_length() - 1, 256, k.n_channels, k.peak_mW, False, 1000 * seed + i)[0].to(torch.complex64)
            for i, k in enumerate(_links(case))]


def _linear(field, fib, T, z0, z1):
    """The field carried by the exact linear flow from z0 to z1 (complex128)."""
    phase, gain = _flow(fib, T, field.numel(), z0, z1)
    return _ifft(_fft(field.to(torch.complex128)) * torch.polar(torch.full_like(phase, gain), phase))


def _float32_fiber():
    """The benchmark's span with coefficients that 32-bit tensors hold."""
    f = dm_map(1)
    return FiberMap(tuple(Segment(s.length_km, float(np.float32(s.beta2_ps2_per_km)), s.beta3_ps3_per_km,
                                  float(np.float32(s.sigma_per_W_km))) for s in f.segments),
                    f.gamma_per_km, f.z_a_km, f.n_periods)


# -------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        N = 1 << case["log2n"]
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        data = torch.randn(N, dtype=_dtype(case["prec"]), device=DEVICE, generator=g)
        ws = torch.empty(mpa.ss_workspace_bytes(N, case["prec"]), dtype=torch.uint8, device=DEVICE)
        return {"kind": kind, "data": data, "sign": case["sign"], "ws": ws}
    if kind == "batch":
        fields = _link_fields(case, seed)
        buffers = [f.clone() for f in fields]
        b = mpa.Batch([(k.fiber, k.T_ps, k.length_km, f) for k, f in zip(_links(case), buffers)], case["L"], case["M"],
                      case["n_iter"])
        b.autotune()
        return {"kind": kind, "fields": fields, "buffers": buffers, "batch": b}
    if kind == "link":
        field, T = _field(case, seed)
        plan = mpa.Plan(_fiber(case), field.numel(), T, case["L"], case["M"], case["n_iter"], precision=case["prec"])
        if case["tune"]:
            plan.autotune()
        return {"kind": kind, "field": field.to(_dtype(case["prec"])), "plan": plan, "z0": case["z0"],
                "z1": case["z0"] + case["L"] * case["intervals"]}
    if kind == "grad":
        fib = _float32_fiber()
        field, T = _field(case, seed)
        z0, z1 = case["z0"], case["z0"] + case["L"] * case["intervals"]
        field = field.to(torch.complex64)
        plan = mpa.Plan(fib, field.numel(), T, case["L"], case["M"], case["n_iter"])
        sig, b2 = plan.segment_coefficients()
        return {"kind": kind, "field": field, "plan": plan, "z0": z0, "z1": z1,
                "sigma": torch.tensor(sig, dtype=torch.float32), "beta2": torch.tensor(b2, dtype=torch.float32),
                "target": _linear(field, fib, T, z0, z1).to(torch.complex64)}
    field, T = _field(case, seed)
    fib = _fiber(case) if kind == "ss" else _float32_fiber()
    z0, z1 = case["z0"], case["z0"] + case["dz"] * case["steps"]
    dtype = _dtype(case.get("prec", "fp32"))
    state = {"kind": kind, "field": field.to(dtype), "fiber": fib, "T": T, "dz": case["dz"], "z0": z0, "z1": z1}
    if kind == "ss":
        state["ws"] = torch.empty(mpa.ss_workspace_bytes(field.numel(), dtype), dtype=torch.uint8, device=DEVICE)
    else:
        # the loss Im <B, A_out> with B the field carried by the linear flow: the nonlinear phase
        state["grad_out"] = (1j * _linear(state["field"], fib, T, z0, z1)).to(dtype)
    return state


def run(state):
    kind = state["kind"]
    if kind == "fft":
        return mpa.fft(state["data"].clone(), state["sign"], workspace=state["ws"])
    if kind == "batch":
        torch._foreach_copy_(state["buffers"], state["fields"])  # the links' new inputs, in the batch's buffers
        state["batch"].propagate()
        return state["buffers"]
    if kind == "link":
        return state["plan"].propagate(state["field"].clone(), state["z0"], state["z1"])
    if kind == "ss":
        return mpa.ss_propagate(state["field"].clone(), state["fiber"], state["T"], state["dz"], state["z0"],
                                state["z1"], workspace=state["ws"])
    if kind == "grad":
        field = state["field"].clone().requires_grad_(True)
        sigma = state["sigma"].clone().requires_grad_(True)
        beta2 = state["beta2"].clone().requires_grad_(True)
        out = mpa.MPAFunction.apply(field, sigma, beta2, state["plan"], state["z0"], state["z1"])
        loss = (out - state["target"]).abs().square().sum()
        loss.backward()
        return {"out": out.detach(), "field": field.grad, "sigma": sigma.grad, "beta2": beta2.grad}
    gi, gs, gb = mpa.ss_adjoint(state["field"], state["grad_out"], state["fiber"], state["T"], state["dz"],
                                state["z0"], state["z1"])
    # the coefficients of a 32-bit fit are updated in 32 bits
    return {"field": gi, "sigma": torch.from_numpy(gs).to(torch.float32), "beta2": torch.from_numpy(gb).to(torch.float32)}


# ------------------------------------------------------------------- work
def work(case):
    """Fields in and out once; 5 N log2 N operations a transform and the
    pointwise steps (two phase products, the Kerr term and the sums of a node,
    a phase product and a Kerr rotation of a split step)."""
    if case["kind"] == "batch":
        b = f = 0.0
        for k in _links(case):
            lg = k.N.bit_length() - 1
            nodes = k.length_km / case["L"] * (case["M"] + 1) * case["n_iter"]
            b += 2.0 * 8 * k.N
            f += nodes * k.N * (10.0 * lg + 30.0)
        return {"bytes": b, "flops": f}
    lg, N = case["log2n"], float(1 << case["log2n"])
    size = 16 if case.get("prec") == "fp64" else 8
    if case["kind"] == "fft":
        return {"bytes": 2 * size * N, "flops": 5.0 * N * lg}
    if case["kind"] == "link":
        nodes = case["intervals"] * (case["M"] + 1) * case["n_iter"]
        return {"bytes": 2 * size * N, "flops": nodes * N * (10.0 * lg + 30.0)}
    if case["kind"] == "grad":  # field, target in; output, gradient out; a forward and a reverse transform pair a node
        nodes = case["intervals"] * (case["M"] + 1) * case["n_iter"]
        return {"bytes": 4 * size * N, "flops": nodes * N * (20.0 * lg + 80.0)}
    if case["kind"] == "ss":
        return {"bytes": 2 * size * N, "flops": case["steps"] * N * (10.0 * lg + 20.0)}
    return {"bytes": 3 * size * N, "flops": case["steps"] * N * (20.0 * lg + 60.0)}


# ------------------------------------------------------- 64-bit reference
def _fft(a):
    """F[x]_k = sum_n x_n exp(+2 pi i k n / N)."""
    return torch.fft.ifft(a, norm="forward")


def _ifft(a):
    return torch.fft.fft(a, norm="forward")


def _omega(N, T):
    return torch.fft.fftfreq(N, d=T / N, dtype=torch.float64, device=DEVICE) * (2.0 * math.pi)


def _overlap(fib, za, zb):
    """Length of [za, zb] within each segment kind of the period."""
    out = np.zeros(len(fib.segments))
    for p in range(int(za // fib.period_km), int(zb // fib.period_km) + 1):
        a = p * fib.period_km
        for i, s in enumerate(fib.segments):
            out[i] += max(0.0, min(zb, a + s.length_km) - max(za, a))
            a += s.length_km
    return out


def _amplifiers(fib, za, zb):
    return math.floor(zb / fib.z_a_km + 1e-9) - math.floor(za / fib.z_a_km + 1e-9)


def _flow(fib, T, N, za, zb):
    """Phase and real factor of the exact linear flow from za to zb."""
    w = _omega(N, T)
    ov = _overlap(fib, za, zb)
    i2 = float(sum(o * s.beta2_ps2_per_km for o, s in zip(ov, fib.segments)))
    i3 = float(sum(o * s.beta3_ps3_per_km for o, s in zip(ov, fib.segments)))
    g = math.exp(fib.gamma_per_km * (_amplifiers(fib, za, zb) * fib.z_a_km - (zb - za)))
    return w * w * (0.5 * i2) + w * w * w * (i3 / 6.0), g


def _tables(fib, z0, L, M):
    """Overlaps from z0 to each node (M+1, segments), beta3 integrals, losses
    and the share of each segment's sigma at each node."""
    z = [z0 + L * j / M for j in range(M + 1)]
    ov = np.stack([_overlap(fib, z0, zj) for zj in z])
    i3 = ov @ np.array([s.beta3_ps3_per_km for s in fib.segments])
    loss = np.exp(-fib.gamma_per_km * (np.array(z) - z0))
    eps = 1e-7
    share = np.zeros_like(ov)
    for j, zj in enumerate(z):
        left = _overlap(fib, zj - eps, zj) / eps if j else None
        right = _overlap(fib, zj, zj + eps) / eps if j < M else None
        share[j] = right if left is None else left if right is None else 0.5 * (left + right)
    return [torch.from_numpy(np.ascontiguousarray(a)).to(DEVICE) for a in (ov, i3, loss, np.round(2 * share) / 2)]


def _interval(psi0, fib, T, z0, L, M, n_iter, sigma, beta2):
    """psi after n_iter Picard iterations at the last node, then the step to
    A_hat(z0 + L).  sigma, beta2: 64-bit tensors per segment."""
    N = psi0.numel()
    w = _omega(N, T)
    ov, i3, loss, share = _tables(fib, z0, L, M)
    weight = (share @ sigma) * (L / M)
    i2 = ov @ beta2
    grad = beta2.requires_grad or psi0.requires_grad
    block = M + 1 if grad else max(1, min(M + 1, (1 << 27) // N))

    def phase(a, b):
        p = (w * w)[None] * (0.5 * i2[a:b, None]) + (w * w * w)[None] * (i3[a:b, None] / 6.0)
        return torch.polar(torch.ones_like(p), p)

    psi = None
    for it in range(n_iter):
        r = torch.zeros_like(psi0)
        new = []
        for a in range(0, M + 1, block):
            b = min(M + 1, a + block)
            ph = phase(a, b)
            cur = psi0[None].expand(b - a, N) if psi is None else psi[a:b]
            A = _ifft(cur * ph * loss[a:b, None])
            A = A * (A.real.square() + A.imag.square())
            V = _fft(A) * ph.conj() * (weight[a:b] / loss[a:b])[:, None]
            del A, ph
            if a == 0:  # the first node enters with half its weight
                first = torch.ones(b - a, 1, dtype=torch.float64, device=DEVICE)
                first[0] = 0.5
                V = V * first
            s = torch.cumsum(V, 0) + r[None]
            r = s[-1]
            half = V * 0.5
            if a == 0:
                half = half * (first * 2.0 - 1.0)  # node 0: nothing summed, psi_0 stays
                half = half + torch.cat([V[:1], torch.zeros_like(V[1:])])
            out = psi0[None] + 1j * (s - half)
            if it == n_iter - 1:
                new = [out[-1:]]
            elif grad:
                new.append(out)
            elif psi is None and not new:
                new = [torch.empty(M + 1, N, dtype=psi0.dtype, device=DEVICE)]
                new[0][a:b] = out
            elif psi is None:
                new[0][a:b] = out
            else:
                psi[a:b] = out
            del s, half, V, out
        if it == n_iter - 1 or grad:
            psi = torch.cat(new) if it < n_iter - 1 else new[0]
        elif psi is None:
            psi = new[0]
    g = loss[M] * math.exp(_amplifiers(fib, z0, z0 + L) * fib.z_a_km * fib.gamma_per_km)
    return psi[-1] * phase(M, M + 1)[0] * g


def _coefficients(fib):
    return (torch.tensor([s.sigma_per_W_km for s in fib.segments], dtype=torch.float64, device=DEVICE),
            torch.tensor([s.beta2_ps2_per_km for s in fib.segments], dtype=torch.float64, device=DEVICE))


def _mpa64(A, fib, T, z0, L, M, n_iter, intervals, sigma, beta2):
    a = _fft(A)
    for q in range(intervals):
        args = (a, fib, T, z0 + L * q, L, M, n_iter, sigma, beta2)
        a = checkpoint(_interval, *args, use_reentrant=False) if A.requires_grad else _interval(*args)
    return _ifft(a)


def _ss64(A, fib, T, z0, dz, steps, sigma, beta2):
    w = _omega(A.numel(), T)

    def linear(a, za, zb):
        ov = torch.from_numpy(_overlap(fib, za, zb)).to(DEVICE)
        i3 = float(sum(o * s.beta3_ps3_per_km for o, s in zip(_overlap(fib, za, zb), fib.segments)))
        g = math.exp(fib.gamma_per_km * (_amplifiers(fib, za, zb) * fib.z_a_km - (zb - za)))
        p = w * w * (0.5 * (ov @ beta2)) + w * w * w * (i3 / 6.0)
        return a * torch.polar(torch.ones_like(p), p) * g

    a = linear(_fft(A), z0, z0 + 0.5 * dz)
    for k in range(steps):
        zk = z0 + dz * k
        x = _ifft(a)
        s = torch.from_numpy(_overlap(fib, zk, zk + dz)).to(DEVICE) @ sigma
        p = (x.real.square() + x.imag.square()) * s
        x = x * torch.polar(torch.ones_like(p), p)
        end = z0 + dz * steps if k == steps - 1 else zk + 1.5 * dz
        a = linear(_fft(x), zk + 0.5 * dz, end)
    return _ifft(a)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        x = prepare(case, seed)["data"].to(torch.complex128)
        return _fft(x) if case["sign"] > 0 else _ifft(x)
    if kind == "batch":
        out = []
        for k, f in zip(_links(case), _link_fields(case, seed)):
            fib = k.fiber
            out.append(_mpa64(f.to(torch.complex128), fib, k.T_ps, 0.0, case["L"], case["M"], case["n_iter"],
                              int(round(k.length_km / case["L"])), *_coefficients(fib)))
        return out
    field, T = _field(case, seed)
    if kind == "link":
        if case["intervals"] * case["n_iter"] * (case["M"] + 1) * field.numel() > 2 ** 33.5:
            return None
        fib = _fiber(case)
        x = field.to(_dtype(case["prec"])).to(torch.complex128)
        return _mpa64(x, fib, T, case["z0"], case["L"], case["M"], case["n_iter"], case["intervals"],
                      *_coefficients(fib))
    if kind == "ss":
        fib = _fiber(case)
        x = field.to(_dtype(case["prec"])).to(torch.complex128)
        return _ss64(x, fib, T, case["z0"], case["dz"], case["steps"], *_coefficients(fib))
    # gradients by automatic differentiation of the same method
    fib = _float32_fiber()
    N = field.numel()
    if kind == "grad" and N * (case["M"] + 1) * case["n_iter"] > 2 ** 28.7 or kind == "ss_grad" and N * case["steps"] > 2 ** 27.5:
        return None
    field = field.to(torch.complex64)
    x = field.to(torch.complex128).requires_grad_(True)
    sigma, beta2 = (c.requires_grad_(True) for c in _coefficients(fib))
    if kind == "grad":
        z1 = case["z0"] + case["L"] * case["intervals"]
        target = _linear(field, fib, T, case["z0"], z1).to(torch.complex64).to(torch.complex128)
        out = _mpa64(x, fib, T, case["z0"], case["L"], case["M"], case["n_iter"], case["intervals"], sigma, beta2)
        (out - target).abs().square().sum().backward()
        return {"out": out.detach(), "field": x.grad, "sigma": sigma.grad, "beta2": beta2.grad}
    z1 = case["z0"] + case["dz"] * case["steps"]
    out = _ss64(x, fib, T, case["z0"], case["dz"], case["steps"], sigma, beta2)
    out.backward((1j * _linear(field, fib, T, case["z0"], z1)).to(torch.complex64).to(torch.complex128))
    return {"field": x.grad, "sigma": sigma.grad, "beta2": beta2.grad}
