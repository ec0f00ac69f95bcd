"""Measured cases: the calls a program makes to search spectra, over the sizes and options in use.

``listed`` names them, ``draw`` gives further ones of the same ranges, ``prepare`` makes what the
program holds before the call, ``run`` is one call through the package's public entry points, ``work``
is what one call cannot do without, and ``exact`` is its result in 64 bits by torch alone.

Spectra are unit-power complex Gaussian noise with a few drifting tones of eight harmonics a little
above the 6-sigma thresholds, as a survey's spectra are. Every search returns the F-A plane, the
candidates of every harmonic plane (power; column; row, plane), their counts and the loudest points.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1806_01556_gb300 as fdas

F = 2048  # overlap-save segment length
FORMS = {"fp32": 0, "bf16x3": 1, "fp16s": 2}


def _case(name, call, n, **kw):
    base = dict(name=name, call=call, n=n, n_temp=85, n_tap=421, n_harm=8, form="fp32", index="fundamental")
    base.update(kw)
    return base


def listed():
    return [
        # The shortest spectra: one call's latency and launches are all of its time.
        _case("search_n4099", "search", 4099),
        # A short observation (the small test workload's length).
        _case("search_n65536", "search", 65536),
        # The survey's own spectrum: 2^21 bins, 85 templates, 8 harmonic planes.
        _case("search_n2097152", "search", 2097152),
        # The request loop's parameter set (16 harmonic planes) on a spectrum of odd length.
        _case("search_16planes_n1000003", "search", 1000003, n_harm=16),
        # The precision forms of the convolution: the survey's length, and a short odd one.
        _case("search_bf16x3_n2097152", "search", 2097152, form="bf16x3"),
        _case("search_fp16s_n200003", "search", 200003, form="fp16s"),
        # Harmonic planes indexed by the highest harmonic, up to 8 and up to 16 planes.
        _case("search_highest8_n1048576", "search", 1048576, index="highest"),
        _case("search_highest16_n262147", "search", 262147, index="highest", n_harm=16),
        # The first stage on its own, with the shorter templates, on the longest spectrum.
        _case("convolve_tap257_n4194303", "convolve", 4194303, n_tap=257),
        # The second stage on its own, on a plane the caller holds.
        _case("harmonic_n2097152", "harmonic", 2097152),
        # Dedispersion trials of uneven length (floor(2^U), U in 18..22) in one replayed batch.
        _case("batch8", "batch", 0,
              lengths="294763,3811091,561133,1746508,262147,2389120,1048576,848001"),
        # End to end from pinned host memory, results back on the host.
        _case("host_n524288", "host", 524288),
    ]


def _length(rng, lo, hi):
    n = int(2.0 ** rng.uniform(lo, hi))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search16", "form", "highest", "highest16", "convolve",
                       "harmonic", "batch", "host"])
    shape = dict(n_temp=rng.choice([85, 85, 85, 43, 127]), n_tap=rng.choice([421, 421, 257, 129]),
                 n_harm=rng.choice([8, 8, 8, 4, 5]))
    if kind == "search16":
        c = _case("", "search", _length(rng, 12, 21), **{**shape, "n_harm": rng.choice([16, 16, 12])})
    elif kind == "form":
        c = _case("", "search", _length(rng, 12, 21), **shape, form=rng.choice(["bf16x3", "fp16s"]))
    elif kind == "highest":
        c = _case("", "search", _length(rng, 12, 20), **{**shape, "n_temp": rng.choice([85, 43])}, index="highest")
    elif kind == "highest16":
        c = _case("", "search", _length(rng, 12, 18), **{**shape, "n_temp": rng.choice([85, 43]),
                                                         "n_harm": rng.choice([16, 16, 12])}, index="highest")
    elif kind == "batch":
        lengths = [_length(rng, 18, 21.25) for _ in range(rng.randint(2, 4))]
        c = _case("", "batch", 0, **{**shape, "n_temp": 85}, lengths=",".join(map(str, lengths)))
    elif kind == "convolve":
        c = _case("", "convolve", _length(rng, 12, 21.5), **shape)
    else:
        c = _case("", kind, _length(rng, 12, 21), **shape)
    del c["name"]
    return c


def _lengths(case):
    return [int(x) for x in case["lengths"].split(",")] if case["call"] == "batch" else [case["n"]]


def _params(case):
    c = (case["n_temp"] - 1) // 2
    return fdas.Params(n_temp=case["n_temp"], z_min=-c, n_tap=case["n_tap"], n_harm=case["n_harm"],
                       harm_mask=(1 << case["n_harm"]) - 1, precision=FORMS[case["form"]],
                       harm_index=int(case["index"] == "highest"))


def _generator(seed, b=0):
    return torch.Generator(device="cuda").manual_seed(1009 * int(seed) + b)


def _spectrum(n, seed, b):
    """complex64[n] on the GPU: noise of unit power, and two tones of eight harmonics (three on long spectra)."""
    g = _generator(seed, b)
    x = torch.view_as_complex(torch.randn(n, 2, generator=g, device="cuda") * math.sqrt(0.5)).to(torch.complex128)
    u = torch.rand(3, 3, generator=g, device="cuda").tolist()
    tau = torch.arange(n, dtype=torch.float64, device="cuda") / n
    t = torch.zeros(n, dtype=torch.complex128, device="cuda")
    for mean, drift, loud in u[: 3 if n > 1 << 20 else 2]:
        mean, z, amp = n / 64 + mean * (n / 9 - n / 64), round(40 * (2 * drift - 1)), 7 + 5 * loud
        for k in range(1, 9):
            cycles = k * ((mean - 0.5 * z) * tau + 0.5 * z * tau * tau)
            t += torch.polar(torch.full_like(tau, amp / k), 2 * math.pi * (cycles - cycles.floor()))
    return (x + torch.fft.fft(t) / n).to(torch.complex64)


def _plane(case, seed):
    """float32[n_temp][n]: powers of unit-mean noise, as the first stage leaves them."""
    return torch.empty(case["n_temp"], case["n"], device="cuda").exponential_(generator=_generator(seed))


def _views(p, cands, counts, peaks):
    """The candidate records (power, j, then i and k in one word) as tensors of their fields."""
    rec, top = cands.view(torch.int32).view(p.n_harm, p.cand_cap, 3), peaks.view(torch.int32).view(p.n_harm, 3)
    return dict(power=cands.view(torch.float32).view(p.n_harm, p.cand_cap, 3)[:, :, 0], place=rec[:, :, 1:],
                counts=counts, peak_power=peaks.view(torch.float32).view(p.n_harm, 3)[:, 0], peak_place=top[:, 1:])


def prepare(case, seed):
    p = _params(case)
    if case["call"] == "batch":
        b = fdas.Batch(p, _lengths(case))
        for k, n in enumerate(b.lengths):
            b.specs[k].copy_(_spectrum(n, seed, k))
            b.cands[k].zero_()
        out = [dict(plane=b.planes[k][:, :n], **_views(p, b.cands[k], b.counts[k], b.peaks[k]))
               for k, n in enumerate(b.lengths)]
        return dict(call="batch", plan=b.plan(), batch=b, out=out)
    n = case["n"]
    s = fdas.Searcher(p, n)
    s.cands.zero_()
    state = dict(call=case["call"], p=p, n=n, s=s)
    if case["call"] == "harmonic":
        s.plane[:, :n] = _plane(case, seed)
        state["out"] = _views(p, s.cands, s.counts, s.peaks)
        return state
    spec = _spectrum(n, seed, 0)
    state["out"] = dict(plane=s.plane[:, :n])
    if case["call"] == "host":
        state["spec"] = torch.empty(n, dtype=torch.complex64, pin_memory=True).copy_(spec)
        state["out"].update(_views(p, s.h_cands, s.h_counts, s.h_peaks))
    else:
        state["spec"] = spec
        if case["call"] == "search":
            state["out"].update(_views(p, s.cands, s.counts, s.peaks))
    return state


def run(state):
    call = state["call"]
    if call == "search":
        state["s"].search(state["spec"])
    elif call == "host":
        state["s"].search_host(state["spec"])
    elif call == "batch":
        state["plan"].launch()
    elif call == "convolve":
        s = state["s"]
        fdas.fdas_convolve(state["p"], state["spec"], state["n"], s.tmpl, s.plane, s.ld)
    else:
        s = state["s"]
        fdas.fdas_harmonic_sum(state["p"], s.plane, state["n"], s.ld, s.thresh, s.cands, s.counts, s.peaks, s.ws,
                               s.ws_bytes)
    return state["out"]


def work(case):
    """Bytes: spectrum (or plane), template bank and thresholds read once, plane and candidates written once.
    Flops: overlap-save with segments of F points (5 F log2 F per transform), and the harmonic additions."""
    t, k = case["n_temp"], case["n_harm"]
    c = (t - 1) // 2
    total = {"bytes": 0.0, "flops": 0.0}
    for n in _lengths(case):
        if case["call"] != "harmonic":
            seg = -(-n // (F - case["n_tap"] + 1))
            total["bytes"] += 8 * n + 8 * F * (t + 1) + 4 * t * n
            total["flops"] += seg * (5 * F * math.log2(F) * (1 + t) + 6 * F * t) + 3 * t * n
        else:
            total["bytes"] += 4 * t * n
        if case["call"] != "convolve":
            total["bytes"] += 12 * k * 201 + 4 * k * t
            if case["index"] == "highest":
                total["flops"] += t * n * k * (k - 1) / 2
            else:
                total["flops"] += sum((2 * (c // l) + 1) * ((n - 1) // l + 1) for l in range(2, k + 1))
    return total


# ---- the same results in 64 bits ------------------------------------------------------------------


def _taps(case):
    """a_z(q) = integral over tau in [0, 1] of exp(2 pi i (-(q + z/2) tau + z tau^2/2)), complex128[n_temp][n_tap]."""
    c, h = (case["n_temp"] - 1) // 2, (case["n_tap"] - 1) // 2
    z = torch.arange(-c, c + 1, dtype=torch.float64, device="cuda")
    q = torch.arange(-h, h + 1, dtype=torch.float64, device="cuda")
    node, weight = np.polynomial.legendre.leggauss(16)
    panels = h + c + 8  # under a cycle of the integrand each
    out = torch.zeros(len(z), len(q), dtype=torch.complex128, device="cuda")
    left = torch.arange(panels, dtype=torch.float64, device="cuda") / panels
    for x, w in zip(node.tolist(), weight.tolist()):
        tau = left + (x + 1) / 2 / panels
        quad = 0.5 * z[:, None] * (tau * tau - tau)  # [z][panel]
        lin = q[:, None] * tau  # [q][panel]
        ez = torch.polar(torch.ones_like(quad), 2 * math.pi * (quad - quad.floor()))
        eq = torch.polar(torch.ones_like(lin), -2 * math.pi * (lin - lin.floor()))
        out += (w / 2 / panels) * (ez @ eq.T)
    return out


def _exact_plane(case, spec):
    """|sum_q X[j+q] conj(a_t[q])|^2 by overlap-save with long segments, float64[n_temp][n]."""
    n, h, size = spec.numel(), (case["n_tap"] - 1) // 2, 16384
    keep = size - 2 * h
    seg = -(-n // keep)
    x = torch.zeros(seg * keep + 2 * h, dtype=torch.complex128, device="cuda")
    x[h: h + n] = spec
    x = torch.fft.fft(x.unfold(0, size, keep), dim=1)
    out = torch.empty(case["n_temp"], n, dtype=torch.float64, device="cuda")
    for t, a in enumerate(_taps(case)):
        filt = torch.fft.fft(a, n=size).conj()  # correlation: output m of a segment starts at its point m
        y = torch.fft.ifft(x * filt, dim=1)[:, :keep].reshape(-1)[:n]
        out[t] = y.real.square() + y.imag.square()
    return out


def _threshold(k, sigma=6.0):
    """The x with P(Gamma(k, 1) > x) = the Gaussian tail at sigma, rounded to float32."""
    tail, lo, hi = 0.5 * math.erfc(sigma / math.sqrt(2)), 0.0, 200.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        term = total = 1.0
        for m in range(1, k):
            term *= mid / m
            total += term
        lo, hi = (mid, hi) if math.exp(-mid) * total > tail else (lo, mid)
    return float(np.float32(0.5 * (lo + hi)))


def _round_div(a, b):
    """a / b to the nearest integer, halves away from zero (int64 tensors)."""
    return torch.sign(a) * torch.div(2 * a.abs() + b, 2 * b, rounding_mode="floor")


def _exact_lists(case, plane):
    t, n = plane.shape
    c = (t - 1) // 2
    cap = fdas.Params().cand_cap
    power = torch.zeros(case["n_harm"], cap, dtype=torch.float64, device="cuda")
    peak = torch.zeros(case["n_harm"], dtype=torch.float64, device="cuda")
    i, j = torch.arange(-c, c + 1, device="cuda"), torch.arange(n, device="cuda")
    hp, m = plane, c
    for k in range(1, case["n_harm"] + 1):
        if case["index"] == "highest":
            hp = torch.zeros_like(plane)
            for l in range(1, k + 1):
                hp += plane[c + _round_div(l * i, k)][:, _round_div(l * j, k)]
        elif k > 1:
            mk, cols = c // k, (n - 1) // k + 1
            hp = hp[m - mk: m + mk + 1, :cols] + plane[c - k * mk: c + k * mk + 1: k][:, ::k]
            m = mk
        over = hp[hp > _threshold(k)].sort(descending=True).values[:cap]
        power[k - 1, : len(over)] = over
        peak[k - 1] = hp.max()
    return dict(power=power, place=None, counts=None, peak_power=peak, peak_place=None)


def exact(case, seed):
    if case["call"] == "harmonic":
        return _exact_lists(case, _plane(case, seed).double())
    out = []
    for b, n in enumerate(_lengths(case)):
        plane = _exact_plane(case, _spectrum(n, seed, b).to(torch.complex128))
        out.append(dict(plane=plane, **(_exact_lists(case, plane) if case["call"] != "convolve" else {})))
    return out if case["call"] == "batch" else out[0]
