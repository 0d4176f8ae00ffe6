"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or, for the served stream, one burst of requests) through the public entry
points of ``paper_1507_07733_gb300.binding``: ``ar_unfold`` on device buffers in its output modes,
``ar_unfold_host``, ``ar_unfold_tc``, ``ar_reconstruct``, a batch plan and a server. Sizes are those
of the repository's workloads (3-124 stations, 1024/2048/4096 samples, 1-256 directions) and odd
ones between them. ``exact`` restates the path in plain 64-bit PyTorch and NumPy.
"""
import math
import random

import numpy as np
import torch

from paper_1507_07733_gb300 import binding, synth

C_M_PER_NS = 0.299792458
SAMPLES = (1024, 2048, 4096)
RATES = (200e6, 200e6, 200e6, 204.8e6, 220e6, 240e6)

#: entry point -> what it stands for
KINDS = ("unfold", "mixed", "host", "tc", "reconstruct", "batch", "server")


def _case(name, kind, stations, samples, dirs, *, traces=True, fine=False, snr=False, fs=200e6, terms=0, events=0,
          sizes=0):
    c = dict(kind=kind, stations=stations, samples=samples, dirs=dirs, traces=traces, fine=fine, snr=snr, fs=fs,
             terms=terms, events=events, sizes=sizes)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small event with one candidate direction, as an online monitor unfolds each trigger
        _case("single_event", "unfold", 10, 2048, 1),
        # a few stations and directions, peaks only: the inner call of a direction search
        _case("small_peaks_1024", "unfold", 7, 1024, 19, traces=False),
        # the full array scanned over a direction grid with every trace kept
        _case("scan_2048", "unfold", 124, 2048, 64),
        # the same with long traces and odd counts, at another digitiser rate
        _case("scan_4096", "unfold", 67, 4096, 51, fs=220e6),
        # the same with short traces
        _case("scan_1024", "unfold", 101, 1024, 97),
        # a fine direction search that keeps only the peaks
        _case("peaks_2048", "unfold", 113, 2048, 251, traces=False),
        # sub-sample peak times and SNR weights, the timing analysis
        _case("timing_2048", "unfold", 89, 2048, 77, fine=True, snr=True),
        # an array of three antenna types
        _case("mixed_antennas", "mixed", 124, 2048, 64),
        # the tensor-core precision variant at its FP32-level split
        _case("tc_4096", "tc", 43, 4096, 29, terms=6),
        # the iterative reconstruction of one event
        _case("reconstruct", "reconstruct", 124, 2048, 1),
        # uneven events in one graph launch, every trace kept
        _case("batch_uneven", "batch", 0, 0, 0, events=12, sizes=1),
        # a burst of uneven requests to the server, host buffers in, peaks out
        _case("served_burst", "server", 0, 0, 0, traces=False, events=10, sizes=2),
    ]


def draw(rng):
    """One more case: any entry point, sizes spread over their logarithm, any rate and output mode."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        case = _draw(rng)
        if work(case)["flops"] <= most:
            return case


def _draw(rng):
    kind = rng.choice(("unfold", "unfold", "unfold", "unfold", "unfold", "mixed", "host", "tc", "reconstruct",
                       "batch", "server"))
    log_int = lambda lo, hi: min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))
    s, n, d = log_int(3, 124), rng.choice(SAMPLES), log_int(1, 256)
    fs = rng.choice(RATES)
    traces, fine, snr = rng.random() < 0.6, rng.random() < 0.2, rng.random() < 0.2
    if kind in ("batch", "server"):
        return _case(None, kind, 0, 0, 0, traces=traces and kind == "batch", events=rng.randint(2, 10),
                     sizes=rng.randint(2, 10 ** 6))
    if kind == "reconstruct":
        return _case(None, kind, max(s, 5), n, 1, fs=fs)
    if kind == "tc":
        return _case(None, kind, s, n, min(d, 48), traces=traces, fs=fs, terms=rng.choice((3, 6)))
    if kind == "host":
        return _case(None, kind, s, n, min(d, 64), traces=traces, fs=fs)
    if kind == "mixed":
        return _case(None, kind, s, n, d, traces=traces, fs=fs)
    return _case(None, kind, s, n, d, traces=traces, fine=fine, snr=snr, fs=fs)


# ---- inputs -----------------------------------------------------------------------------

def _key(seed):
    return int(seed) % (1 << 31)


def _sizes(case):
    """(stations, samples, directions) of each event of the case."""
    if not case["events"]:
        return [(case["stations"], case["samples"], case["dirs"])]
    r = random.Random(case["sizes"])
    return [(r.randint(3, 124), r.choice(SAMPLES), r.randint(16, 256)) for _ in range(case["events"])]


def _patterns(case, seed):
    k = _key(seed)
    if case["kind"] != "mixed":
        return [synth.make_pattern(seed_key=k)]
    return [synth.make_pattern(seed_key=k), synth.make_pattern(seed_key=k + 1),
            synth.make_pattern(seed_key=k + 2, grid=synth.LARGE_PATTERN_GRID)]


def _events(case, seed):
    k = _key(seed)
    out = []
    for i, (s, n, d) in enumerate(_sizes(case)):
        rng = np.random.default_rng([k, i])
        dirs = synth.random_directions(d, rng)
        out.append(synth.make_event(s, n, dirs, seed_key=k + 97 * i, plane_wave=True, fs_hz=case["fs"]))
    return out


def _types(case, seed):
    return synth.station_antenna_types(case["stations"], seed_key=_key(seed), sort=False)


_FLAT = (("efield", torch.float32), ("envelope", torch.float32), ("peak_idx", torch.int32),
         ("peak_amp", torch.float32), ("peak_time_ns", torch.float64), ("residual_ns", torch.float64),
         ("t0_ns", torch.float64), ("chi2", torch.float64), ("status", torch.int32))


def _flat_sizes(s, n, d, traces):
    t = 1 if traces else 0
    return dict(efield=t * d * s * 2 * n, envelope=t * d * s * n, peak_idx=d * s, peak_amp=d * s, peak_time_ns=d * s,
                residual_ns=d * s, t0_ns=d, chi2=d, status=d * s)


def _flat_outputs(sizes, traces, host):
    """One buffer per output for all events of a launch, and each event's part of it."""
    per = [_flat_sizes(*x, traces) for x in sizes]
    flat = {}
    for k, dt in _FLAT:
        total = sum(p[k] for p in per)
        if total:
            flat[k] = torch.zeros(total, dtype=dt, pin_memory=True) if host else torch.zeros(total, dtype=dt, device="cuda")
    parts, at = [], dict.fromkeys(flat, 0)
    for p in per:
        parts.append({k: flat[k][at[k]:at[k] + p[k]] for k in flat})
        for k in flat:
            at[k] += p[k]
    return flat, parts


def prepare(case, seed):
    kind = case["kind"]
    host = kind in ("host", "server")
    put = (lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()) if host else \
        (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda())
    ctx = binding.Context(0, state_budget_bytes=1 << 28)
    pids = [ctx.load_pattern(p) for p in _patterns(case, seed)]
    evs = _events(case, seed)
    for e in evs:
        ctx.prepare(e.n_samples, e.fs_hz, pids[0], e.n_stations)
    state = dict(kind=kind, ctx=ctx, pid=pids[0], case=case)
    ins = [[put(a) for a in (e.traces, e.pos_m, e.t_start_ns, e.dirs_rad)] for e in evs]
    types = put(np.asarray(pids, np.int32)[_types(case, seed)]) if kind == "mixed" else None
    if kind in ("batch", "server"):
        sizes = _sizes(case)
        state["out"], parts = _flat_outputs(sizes, case["traces"], host)
        state["events"] = [binding.make_event(pids[0], *x, e.fs_hz) for x, e in zip(ins, evs)]
        state["outs"] = [binding.outputs_struct(p) for p in parts]
        if kind == "batch":
            state["plan"] = ctx.batch(len(sizes), sum(s for s, _, _ in sizes), sum(d for _, _, d in sizes))
        else:
            state["server"] = binding.Server(ctx, max_batch_events=8)
        return state
    e, (s, n, d) = evs[0], _sizes(case)[0]
    if kind == "reconstruct":
        state["args"] = (pids[0], *ins[0][:3], e.fs_hz)
        return state
    out, _ = binding.alloc_outputs(d, s, n, device="cpu" if host else "cuda", traces=case["traces"], pin_memory=host,
                                   fine=case["fine"], snr=case["snr"])
    state["out"] = out
    state["event"] = binding.make_event(pids[0], *ins[0], e.fs_hz, station_pattern=types)
    state["outs"] = binding.outputs_struct(out)
    return state


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind in ("unfold", "mixed"):
        binding.ar_unfold(ctx.h, state["event"], state["outs"], stream)
    elif kind == "host":
        binding.ar_unfold_host(ctx.h, state["event"], state["outs"], stream)
    elif kind == "tc":
        binding.ar_unfold_tc(ctx.h, state["event"], state["outs"], state["case"]["terms"], stream)
    elif kind == "batch":
        state["plan"].run(state["events"], state["outs"])
    elif kind == "server":
        sv = state["server"]
        tickets = [sv.submit(e, o) for e, o in zip(state["events"], state["outs"])]
        for t in tickets:
            if sv.wait(t) != binding.AR_OK:
                raise RuntimeError("a request failed")
            sv.release(t)
    else:
        res = ctx.reconstruct(*state["args"], sync=False)
        return dict(direction=res["direction"], t0_ns=res["t0_ns"], chi2=res["chi2"], iterations=res["iterations"],
                    history=res["history"], last=res["last"])
    return state["out"]


# ---- what a pass cannot do without ---------------------------------------------------------

def work(case):
    nbytes = flops = 0.0
    for s, n, d in _sizes(case):
        m, pairs = n // 4, s * d
        types = 3 if case["kind"] == "mixed" else 1
        # traces, positions, window starts, directions; the four corner slabs of a direction's cell
        nbytes += 8.0 * n * s + 32.0 * s + 16.0 * d + min(types * d * 4 * 51 * 32.0, types * 19 * 72 * 51 * 32.0)
        # peaks, times, residuals, status; t0, chi2; the traces
        nbytes += pairs * (28.0 + 8.0 * case["fine"] + 4.0 * case["snr"]) + 16.0 * d
        nbytes += pairs * 12.0 * n if case["traces"] else 0.0
        # two real transforms per station; the 2x2 inverse per direction and bin; per pair the solve, the band's
        # two one-sided transforms (four M-point ones each), the envelope and the peak
        flops += s * 5.0 * n * math.log2(n) + types * d * m * 60.0
        flops += pairs * (28.0 * m + 8 * 5.0 * m * math.log2(m) + 6.0 * n)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error against ``exact``: FP32 transforms 2.8e-7 to 4.8e-7 (2-norm; single samples
    near zero 1.4e-5 of the rms), the tensor-core splits 5.3e-6 (x3) and 2.7e-6 (x6; single samples 1.2e-4).
    Peaks may move where two samples tie at FP32 resolution."""
    if case["kind"] == "tc":
        return {"rel": 2.2e-5 if case["terms"] == 3 else 1.1e-5, "max": 5e-4, "differ": 2e-3}
    return {"rel": 2e-6, "max": 6e-5, "differ": 2e-3}


# ---- the same in 64 bits -----------------------------------------------------------------

def _response(pattern, dirs, n, fs, dev):
    """H [D][N/2+1][c][p] by trilinear interpolation, and the band's bins."""
    f = np.arange(n // 2 + 1) * fs / n
    band = np.flatnonzero((f >= 30e6) & (f <= 80e6))
    tab = torch.from_numpy(pattern.table).to(dev).to(torch.complex128)

    def cell(u, count):
        i = np.minimum(np.floor(u).astype(np.int64), count - 2)
        return i, u - i

    iz, tz = cell(np.clip((dirs[:, 0] - pattern.zen0_rad) / pattern.dzen_rad, 0, pattern.n_zen - 1), pattern.n_zen)
    ua = np.mod((dirs[:, 1] - pattern.az0_rad) / pattern.daz_rad, pattern.n_az)
    ia = np.floor(ua).astype(np.int64)
    ta, ia = ua - ia, ia % pattern.n_az
    jf, tf = cell(np.clip((f[band] - pattern.f0_hz) / pattern.df_hz, 0, pattern.n_freq - 1), pattern.n_freq)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    h = 0
    for a in (0, 1):
        for b in (0, 1):
            w = (tz if a else 1 - tz) * (ta if b else 1 - ta)
            g = tab[t(iz + a), t((ia + b) % pattern.n_az)]                      # [D][f][c][p]
            tff = t(tf)[None, :, None, None]
            h = h + t(w)[:, None, None, None] * (g[:, t(jf)] * (1 - tff) + g[:, t(jf + 1)] * tff)
    return h, band


def _unfold64(patterns, types, ev, dirs, fine=False, snr=False, traces=True):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    s, n, d = ev.n_stations, ev.n_samples, len(dirs)
    dt = 1e9 / ev.fs_hz
    spec = torch.fft.rfft(torch.from_numpy(ev.traces).to(dev).double(), dim=2)     # [S][2][N/2+1]
    o = dict(efield=torch.empty((d, s, 2, n), dtype=torch.float64, device=dev) if traces else None,
             envelope=torch.empty((d, s, n), dtype=torch.float64, device=dev) if traces else None)
    idx = torch.empty((d, s), dtype=torch.int64, device=dev)
    amp = torch.empty((d, s), dtype=torch.float64, device=dev)
    off, ratio = torch.zeros_like(amp), torch.zeros_like(amp)
    types = np.zeros(s, np.int64) if types is None else np.asarray(types, np.int64)
    hs = [_response(p, dirs, n, ev.fs_hz, dev) for p in patterns]
    for i in range(d):
        z = torch.zeros((s, 2, n), dtype=torch.complex128, device=dev)
        for p, (h, band) in enumerate(hs):
            st = torch.from_numpy(np.flatnonzero(types == p)).to(dev)
            if not len(st):
                continue
            b = torch.from_numpy(band).to(dev)
            v = spec[st][:, :, b]
            hh = h[i]
            det = hh[:, 0, 0] * hh[:, 1, 1] - hh[:, 0, 1] * hh[:, 1, 0]
            zz = torch.zeros((len(st), 2, n), dtype=torch.complex128, device=dev)
            zz[:, 0, b] = 2 * (hh[:, 1, 1] * v[:, 0] - hh[:, 0, 1] * v[:, 1]) / det
            zz[:, 1, b] = 2 * (hh[:, 0, 0] * v[:, 1] - hh[:, 1, 0] * v[:, 0]) / det
            z[st] = torch.fft.ifft(zz, dim=2)
        env = torch.sqrt((z.real ** 2 + z.imag ** 2).sum(1))
        if traces:
            o["efield"][i], o["envelope"][i] = z.real, env
        amp[i], k = env.max(1)
        idx[i] = k
        if fine:
            at = lambda j: env.gather(1, j.clamp(0, n - 1)[:, None])[:, 0]
            a, b0, c = at(k - 1), at(k), at(k + 1)
            second = a - 2 * b0 + c
            ok = (k > 0) & (k < n - 1) & (second < 0)
            off[i] = torch.where(ok, (0.5 * (a - c) / second).clamp(-0.5, 0.5), torch.zeros_like(a))
        if snr:
            far = (torch.arange(n, device=dev)[None] - k[:, None]).abs() > n // 16
            ratio[i] = amp[i] ** 2 / ((env ** 2 * far).sum(1) / far.sum(1))
    idx, amp, off, ratio = (x.cpu().numpy() for x in (idx, amp, off, ratio))
    t = ev.t_start_ns[None] + idx * dt
    tt = ev.t_start_ns[None] + (idx + off) * dt if fine else t
    zen, az = dirs[:, 0], dirs[:, 1]
    u = np.stack([np.sin(zen) * np.cos(az), np.sin(zen) * np.sin(az), np.cos(zen)], 1)
    ds = tt + (u @ ev.pos_m.T) / C_M_PER_NS
    w = ratio if snr else np.ones_like(ds)
    t0 = (w * ds).sum(1) / w.sum(1)
    res = ds - t0[:, None]
    o.update(peak_idx=None, peak_amp=amp, peak_time_ns=t, residual_ns=res, t0_ns=t0, chi2=(w * res ** 2).sum(1),
             status=None)
    if fine:
        o["peak_time_fine_ns"] = tt
    if snr:
        o["snr"] = ratio
    return o, idx


def _fit64(pos, times):
    """Least-squares plane wave, linear in (t0, nx, ny) for a fixed nz, four times from nz = 1."""
    k, nz = 1.0 / C_M_PER_NS, 1.0
    a = np.stack([np.ones(len(pos)), pos[:, 0], pos[:, 1]], 1)
    for _ in range(4):
        x = np.linalg.solve(a.T @ a, a.T @ (times + k * nz * pos[:, 2]))
        nx, ny = -x[1] / k, -x[2] / k
        h = math.hypot(nx, ny)
        if h > 1:
            nx, ny = nx / h, ny / h
        nz = math.sqrt(max(0.0, 1 - (nx * nx + ny * ny)))
    zen, az = math.atan2(math.hypot(nx, ny), nz), math.atan2(ny, nx) % (2 * math.pi)
    u = np.array([math.sin(zen) * math.cos(az), math.sin(zen) * math.sin(az), math.cos(zen)])
    ds = times + pos @ u * k
    return zen, az, x[0], ((ds - ds.mean()) ** 2).sum(), u


def _reconstruct64(pattern, ev, max_iter=8, tol=1e-6):
    dt = 1e9 / ev.fs_hz
    idx = (ev.traces.astype(np.float64) ** 2).sum(1).argmax(1)
    hist = np.full((max_iter + 1, 2), np.nan)
    zen, az, t0, chi2, u = _fit64(ev.pos_m, ev.t_start_ns + idx * dt)
    hist[0] = zen, az
    for it in range(1, max_iter + 1):
        last, new = _unfold64([pattern], None, ev, np.array([[zen, az]]))
        zen, az, t0, chi2, v = _fit64(ev.pos_m, last["peak_time_ns"][0])
        hist[it] = zen, az
        done = np.array_equal(new[0], idx) or math.acos(max(-1.0, min(1.0, float(u @ v)))) < tol
        idx, u = new[0], v
        if done:
            break
    return dict(direction=np.array([zen, az]), t0_ns=np.array([t0]), chi2=np.array([chi2]), iterations=None,
                history=hist, last=last)


def exact(case, seed):
    pats, evs = _patterns(case, seed), _events(case, seed)
    if case["kind"] == "reconstruct":
        return _reconstruct64(pats[0], evs[0])
    if case["kind"] not in ("batch", "server"):
        types = _types(case, seed) if case["kind"] == "mixed" else None
        return _unfold64(pats, types, evs[0], evs[0].dirs_rad, case["fine"], case["snr"], case["traces"])[0]
    flat = {k: [] for k, _ in _FLAT}
    for e in evs:
        one = _unfold64(pats, None, e, e.dirs_rad, traces=case["traces"])[0]
        for k, v in one.items():
            if v is not None:
                flat[k].append(torch.as_tensor(v).cpu().reshape(-1))
    return {k: torch.cat(v) if v else None for k, v in flat.items()}
