"""Workloads on which this library's speed is measured, as a program that uses it runs them.

A case is one call (or one pass of calls) through the public entry points of
``paper_2607_23763_gb300``: ``SosFilter.run`` and ``SosFilter.run_host``, ``BatchPlan.launch`` and
``run_batch``.  Signals are N(0,1) samples; the filters are Butterworth low-pass designs, a bank of
narrow resonators and random stable sections.  ``exact`` gives the outputs in float64 through the
cascade's frequency response (no recurrence), on the device.

Cases by ``kind``:
    run    one signal on the device, optionally with an initial and a final state, at any offset
           into its buffers (a signal that starts inside a larger recording)
    host   one signal in pinned host memory, copied in, filtered and copied out by the library
    plan   a prepared batch of signals of uneven length and order, launched again and again
    batch  chunks of many streams, each continuing from its stream's state, planned per call
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_23763_gb300 import BatchPlan, SosFilter, run_batch

SOLVER_TC = 4  # sos_tuning.solver: PH factorization on the tensor cores


def listed():
    return [
        # one block of a live stream (a receive loop that filters every block as it arrives and carries
        # the state on the device): the smallest call, all latency
        dict(name="live_block", kind="run", family="butter", order=4, cutoff=0.2, n=4096, state=True, offset=0, tc=False),
        # a second or so of a radio channel: order 2 at 0.2 Nyquist, the paper's smallest benchmark filter
        dict(name="signal_1m_order2", kind="run", family="butter", order=2, cutoff=0.2, n=1 << 20, state=False,
             offset=0, tc=False),
        # a piece of a recording that starts at an odd sample and has an odd length, state in and out
        dict(name="piece_3m_order8_odd", kind="run", family="butter", order=8, cutoff=0.1, n=3000017, state=True,
             offset=1, tc=False),
        # a 12-band equaliser over a few minutes of audio: more sections than one pass takes
        dict(name="signal_16m_order24", kind="run", family="butter", order=24, cutoff=0.1, n=1 << 24, state=False,
             offset=0, tc=False),
        # a long recording with the library's defaults
        dict(name="signal_64m_order16", kind="run", family="butter", order=16, cutoff=0.05, n=1 << 26, state=True,
             offset=0, tc=False),
        # narrow resonators (poles at radius 0.999, a memory of many thousand samples)
        dict(name="resonators_64m_tc", kind="run", family="resonator", order=16, cutoff=0.0, n=1 << 26, state=False,
             offset=0, tc=True),
        # a ragged long recording of middle order on the tensor cores
        dict(name="signal_70m_order8_tc", kind="run", family="butter", order=8, cutoff=0.1, n=70000003, state=True,
             offset=0, tc=True),
        # the two ends of the paper's order sweep on a signal far larger than the caches
        dict(name="signal_256m_order2_tc", kind="run", family="butter", order=2, cutoff=0.2, n=1 << 28, state=False,
             offset=0, tc=True),
        dict(name="signal_256m_order16_tc", kind="run", family="butter", order=16, cutoff=0.05, n=1 << 28,
             state=False, offset=0, tc=True),
        # a signal that lives in host memory
        dict(name="host_32m_order16", kind="host", family="butter", order=16, cutoff=0.05, n=1 << 25, state=True),
        # many signals of uneven length and order in one prepared launch
        dict(name="mix_plan_192", kind="plan", signals=192, log2_lo=10.0, log2_hi=22.0, mix=1000, state=False),
        # what a serving loop runs: one chunk of each of many streams, planned on every call
        dict(name="stream_chunks_512", kind="batch", signals=512, lo=4096, hi=65536, mix=500000, state=True),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.70:
        family = rng.choice(["butter", "butter", "random", "resonator"])
        order = rng.choice([2, 4, 6, 8, 12, 16, 16, 20, 24])
        if family == "resonator":
            order = min(order, 16)
        n = int(round(2.0 ** rng.uniform(12.0, 27.0)))
        if rng.random() < 0.3:
            n = 1 << int(round(math.log2(n)))
        return dict(kind="run", family=family, order=order, cutoff=round(rng.uniform(0.04, 0.6), 3), n=n,
                    state=rng.random() < 0.5, offset=rng.choice([0, 0, 0, 1, 3]), tc=rng.random() < 0.5,
                    mix=rng.randrange(1 << 20))
    if u < 0.78:
        return dict(kind="host", family="butter", order=rng.choice([2, 4, 8, 16]), cutoff=0.1,
                    n=int(round(2.0 ** rng.uniform(18.0, 25.0))), state=rng.random() < 0.5)
    if u < 0.90:
        hi = rng.uniform(17.0, 22.0)
        return dict(kind="plan", signals=rng.randrange(8, 193), log2_lo=10.0, log2_hi=round(hi, 2),
                    mix=rng.randrange(1 << 20), state=rng.random() < 0.5)
    lo = int(round(2.0 ** rng.uniform(8.0, 13.0)))
    return dict(kind="batch", signals=rng.randrange(16, 513), lo=lo, hi=lo * rng.randrange(2, 17),
                mix=rng.randrange(1 << 20), state=rng.random() < 0.7)


# ---------------------------------------------------------------------------
# filters: [K][5] rows of b0, b1, b2, a1, a2

def _butter(order, cutoff):
    """Butterworth low-pass through the bilinear transform, sections by ascending pole radius, each
    with unit gain at zero frequency."""
    wc = 2.0 * math.tan(math.pi * cutoff / 2.0)
    poles = []
    for k in range(order // 2):
        t = math.pi * (2 * k + order + 1) / (2 * order)
        p = wc * complex(math.cos(t), math.sin(t))
        poles.append((2.0 + p) / (2.0 - p))
    poles.sort(key=abs)
    rows = []
    for z in poles:
        a1, a2 = -2.0 * z.real, abs(z) ** 2
        g = (1.0 + a1 + a2) / 4.0
        rows.append([g, 2.0 * g, g, a1, a2])
    return np.array(rows)


def _gain(row, w):
    e = np.exp(-1j * np.asarray(w))
    return np.abs((row[0] + row[1] * e + row[2] * e * e) / (1.0 + row[3] * e + row[4] * e * e))


def _resonators(sections, radius=0.999, lo=0.30, hi=0.34):
    rows = []
    for k in range(sections):
        t = math.pi * (lo + (hi - lo) * (k / (sections - 1) if sections > 1 else 0.0))
        row = np.array([1.0, 0.0, -1.0, -2.0 * radius * math.cos(t), radius * radius])
        row[:3] /= _gain(row, t)
        rows.append(row)
    return np.array(rows)


_GRID = np.linspace(0.0, math.pi, 2048)


def _random(sections, rng):
    """Stable sections: pole radius 0.6 .. 0.995, any angle but the very ends, zeros on the unit circle,
    unit peak gain."""
    rows = []
    for _ in range(sections):
        r, t, z = rng.uniform(0.6, 0.995), math.pi * rng.uniform(0.05, 0.95), math.pi * rng.uniform(0.0, 1.0)
        row = np.array([1.0, -2.0 * math.cos(z), 1.0, -2.0 * r * math.cos(t), r * r])
        row[:3] /= max(float(_gain(row, _GRID).max()), float(_gain(row, t)))
        rows.append(row)
    return np.array(rows)


def _design(case):
    if case["family"] == "butter":
        return _butter(case["order"], case["cutoff"])
    if case["family"] == "resonator":
        return _resonators(case["order"] // 2)
    return _random(case["order"] // 2, np.random.default_rng(case["mix"]))


def _mix(case):
    """(filters, lengths) of a plan or batch case: orders 2, 4, 8 and 16, every signal its own filter."""
    rng = np.random.default_rng(case["mix"])
    filters, lengths = [], []
    for _ in range(case["signals"]):
        if case["kind"] == "plan":
            sections = int(rng.choice([1, 2, 4, 8]))
            lengths.append(int(round(2.0 ** rng.uniform(case["log2_lo"], case["log2_hi"]))))
        else:
            sections = int(rng.choice([1, 2, 4, 8], p=[0.4, 0.3, 0.2, 0.1]))
            lengths.append(int(rng.integers(case["lo"], case["hi"] + 1)))
        filters.append(_random(sections, rng))
    return filters, lengths


# ---------------------------------------------------------------------------
# inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _arena(lengths, dtype=torch.float32):
    """One buffer for many signals, as a program that owns its device memory lays them out: every signal
    starts on a 256-byte boundary, what lies between them stays zero."""
    starts, total = [], 0
    for n in lengths:
        starts.append(total)
        total += (n + 63) // 64 * 64
    flat = torch.zeros(total, device="cuda", dtype=dtype)
    return flat, [flat[s:s + n] for s, n in zip(starts, lengths)]


def _state_arena(filters, dtype=torch.float32):
    flat = torch.zeros(sum(len(s) for s in filters), 2, device="cuda", dtype=dtype)
    return flat, list(flat.split([len(s) for s in filters]))


def _signals(case, seed):
    """Input samples and initial states (or None), as the call takes them."""
    g = _generator(seed)
    if case["kind"] in ("run", "host"):
        off = case.get("offset", 0)
        x = torch.randn(case["n"] + off, device="cuda", generator=g)[off:]
        zi = 0.01 * torch.randn(case["order"] // 2, 2, device="cuda", generator=g) if case["state"] else None
        return x, zi
    filters, lengths = _mix(case)
    xs = [v.normal_(generator=g) for v in _arena(lengths)[1]]
    zis = None
    if case["state"]:
        flat, zis = _state_arena(filters)
        flat.copy_(0.01 * torch.randn(flat.shape, device="cuda", generator=g))
    return xs, zis


def prepare(case, seed):
    x, zi = _signals(case, seed)
    if case["kind"] == "run":
        f = SosFilter(_design(case), tuning={"solver": SOLVER_TC} if case["tc"] else None)
        y = torch.empty(case["n"] + case["offset"], device="cuda")[case["offset"]:]
        zf = torch.empty_like(zi) if case["state"] else None
        return dict(kind="run", f=f, x=x, y=y, zi=zi, zf=zf)
    if case["kind"] == "host":
        f = SosFilter(_design(case))
        xh = torch.empty(case["n"], pin_memory=True).copy_(x)
        yh = torch.empty(case["n"], pin_memory=True)
        return dict(kind="host", f=f, x=xh, y=yh, zi=zi.cpu().numpy() if case["state"] else None)
    designs, lengths = _mix(case)
    filters = [SosFilter(s) for s in designs]
    y, ys = _arena(lengths)
    zf, zfs = _state_arena(designs) if case["state"] else (None, None)
    state = dict(kind=case["kind"], f=filters, x=x, ys=ys, zi=zi, zfs=zfs, out=[y] if zf is None else [y, zf])
    if case["kind"] == "plan":
        state["plan"] = BatchPlan(filters, x, ys, zi, zfs)
    return state


def run(state):
    if state["kind"] == "run":
        state["f"].run(state["x"], state["y"], zi=state["zi"], zf=state["zf"])
        return [state["y"]] if state["zf"] is None else [state["y"], state["zf"]]
    if state["kind"] == "host":
        if state["zi"] is None:
            return [state["f"].run_host(state["x"], state["y"])]
        return list(state["f"].run_host(state["x"], state["y"], zi=state["zi"], return_state=True))
    if state["kind"] == "plan":
        state["plan"].launch()
    else:
        run_batch(state["f"], state["x"], state["ys"], state["zi"], state["zfs"])
    return state["out"]


def work(case):
    """Every sample read once and written once (float32) with the states; nine operations per section
    and sample (five products, four sums)."""
    if case["kind"] in ("run", "host"):
        n, k = case["n"], case["order"] // 2
        return {"bytes": 8.0 * n + (16.0 * k if case["state"] else 0.0), "flops": 9.0 * k * n}
    filters, lengths = _mix(case)
    b = f = 0.0
    for s, n in zip(filters, lengths):
        b += 8.0 * n + (16.0 * len(s) if case["state"] else 0.0)
        f += 9.0 * len(s) * n
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the outputs in float64: a section driven from the state (z1, z2) of its transposed direct form II is
# y = (B x + z1 + z2 z^-1) / A, so the cascade's output is its frequency response times the input's
# spectrum plus that of the state; overlap-save over blocks much longer than the impulse response

def _spectra(sos, m):
    e = torch.exp(-2j * math.pi * torch.arange(m // 2 + 1, device="cuda", dtype=torch.float64) / m)
    sec = []
    for b0, b1, b2, a1, a2 in np.asarray(sos, dtype=np.float64).tolist():
        a = 1.0 + a1 * e + a2 * e * e
        sec.append(((b0 + b1 * e + b2 * e * e) / a, 1.0 / a))
    return e, sec


def _exact_signal(sos, x, zi):
    """(y, final state) of one signal in float64."""
    sos = np.asarray(sos, dtype=np.float64)
    n, k = x.numel(), len(sos)
    radius = max(math.sqrt(abs(row[4])) if row[3] ** 2 < 4 * row[4] else
                 (abs(row[3]) + math.sqrt(row[3] ** 2 - 4 * row[4])) / 2 for row in sos)
    memory = 1 << max(10, math.ceil(math.log2(min(65536.0, 8192.0 + 60.0 / max(1e-6, 1.0 - radius)))))
    m = 1 << math.ceil(math.log2(min(max(n, 16) + memory, 4 * memory)))
    hop = m - memory
    e, sec = _spectra(sos, m)
    whole = torch.ones_like(e)
    for h, _ in sec:
        whole = whole * h
    y = torch.empty(n, device="cuda", dtype=torch.float64)
    blocks = (n + hop - 1) // hop
    step = max(1, (1 << 24) // m)
    for first in range(0, blocks, step):
        count = min(step, blocks - first)
        buf = torch.zeros((count - 1) * hop + m, device="cuda", dtype=torch.float64)
        a, b = first * hop - memory, min(n, (first + count) * hop)
        lo = max(a, 0)
        buf[lo - a:b - a] = x[lo:b].double()
        out = torch.fft.irfft(torch.fft.rfft(buf.unfold(0, m, hop)) * whole, m)[:, memory:].reshape(-1)
        y[first * hop:b] = out[:b - first * hop]
    # the last samples again, section by section: the final state is made of every section's last two
    # inputs and outputs; a signal within one block also carries the initial state here
    z = None if zi is None else zi.double().tolist()
    last = min(n, m - memory)
    spec = torch.zeros(m, device="cuda", dtype=torch.float64)
    pre = min(n - last, memory)
    spec[:last + pre] = x[n - last - pre:].double()
    spec = torch.fft.rfft(spec)
    carried = torch.zeros_like(e)  # the initial state's share of the output so far
    within = n == last
    ends = [[float(x[n - 2]) if n > 1 else 0.0, float(x[n - 1])]]
    for i, (h, inv) in enumerate(sec):
        spec, carried = spec * h, carried * h
        if z is not None:
            carried = carried + (z[i][0] + z[i][1] * e) * inv
        t = torch.fft.irfft(spec + carried if within else spec, m)[:last + pre]
        ends.append([float(t[-2]), float(t[-1])])
    if z is not None:
        c = torch.fft.irfft(carried, m)
        s = min(n, memory)
        y[:s] += c[:s]
    zf = torch.empty(k, 2, device="cuda", dtype=torch.float64)
    for i, row in enumerate(sos):
        (x1, x0), (y1, y0) = ends[i], ends[i + 1]
        zf[i, 0] = row[1] * x0 - row[3] * y0 + row[2] * x1 - row[4] * y1
        zf[i, 1] = row[2] * x0 - row[4] * y0
    return y, zf


def exact(case, seed):
    x, zi = _signals(case, seed)
    if case["kind"] in ("run", "host"):
        y, zf = _exact_signal(_design(case), x, zi)
        if case["kind"] == "host":
            y, zf = y.cpu(), zf.cpu().numpy()
        return [y, zf] if case["state"] else [y]
    designs, lengths = _mix(case)
    y, ys = _arena(lengths, torch.float64)
    zf, zfs = _state_arena(designs, torch.float64)
    for i, (s, v) in enumerate(zip(designs, x)):
        one, last = _exact_signal(s, v, None if zi is None else zi[i])
        ys[i].copy_(one)
        zfs[i].copy_(last)
    return [y, zf] if case["state"] else [y]
