"""Measured cases: the excision work that a program has this library do, through its public calls.

A case is a dict of plain values. `form` says which call it makes:

  plan    Plan.excise: the batched (or per-stream) excision into separate output buffers
  mom     the same with the Median of MAD setting the thresholds (mom_windows >= 2)
  copies  CopiesPlan.excise: eight (k, replacement) variants of one input in one pass
  float   Plan.excise with the samples written as fp16 or bf16
  power   Plan.excise with power metering, and the per-window powers
  host    Plan.excise_host: pinned host buffers, copies included
  serve   Server: a chunk pushed to every stream, a backfill request, drained; zero-copy views

Stream lengths and windows follow from `streams`, `len_lo` .. `len_hi` (log-uniform where they
differ), `win_lo` .. `win_hi`, `wins` (how windows are chosen) and `spread` (the generator of
those choices). Samples are receiver noise with impulsive bursts, as the benchmark's feeds have
them: Gaussian noise of sigma 16 (int8) or 120 (12-bit, on a slow drift), bursts of up to 64
(256) samples at a rate per sample between 1e-4 and 1e-2 (5e-3), 5-15 (4-30) sigma high.
"""
import math

import numpy as np
import torch

import paper_1710_08576_gb300 as rfi

ZERO, CONST, CLIP, NOISE = 0, 1, 2, 3
SEED = 7          # digital-noise key of every case
ALIGN = 256       # streams start on a multiple of this many elements, as separate allocations do
FLAGS = {"graph": rfi.RFI_PLAN_GRAPH, "autotune": rfi.RFI_PLAN_AUTOTUNE, "noise_pass": rfi.RFI_PLAN_NOISE_PASS,
         "per_stream": rfi.RFI_PLAN_PER_STREAM}
# windows of a whole number of microseconds or nanoseconds at 800 Msps and of round sample counts
DECIMAL = [800, 1000, 1600, 2000, 4000, 5000, 8000, 10000, 12500, 16000, 20000, 25000, 32000, 40000, 50000, 64000]
VARIANTS = [(k, m, 1 if m == CONST else 0, SEED) for k in (3.0, 5.0) for m in (ZERO, CONST, CLIP, NOISE)]


def listed():
    base = {"bits": 8, "streams": 60, "wins": "pow2", "spread": 2, "k": 3.0, "mode": NOISE, "flags": "graph", "form": "plan"}

    def case(name, n, w, **more):
        return {**base, "name": name, "len_lo": n[0], "len_hi": n[-1], "win_lo": w[0], "win_hi": w[-1], **more}

    return [
        # one antenna's short record, blanked: the smallest call, where launch and latency count
        case("single", [1 << 20], [4096], streams=1, spread=1, mode=ZERO),
        # a real-time block: all 60 inputs of the backend, 0.66 ms of sky at 800 Msps
        case("block60", [1 << 19], [16384]),
        # records of any length cut into windows of round decimal lengths, held at the threshold,
        # by a program that neither captures nor tunes
        case("ragged24", [1 << 18, 1 << 22], [1000, 40000], streams=24, wins="decimal", spread=6, k=4.0, mode=CLIP,
             flags=""),
        # the backend's full batch (84 ms of all inputs), blanked and with digital noise
        case("gwb60_zero", [1 << 26], [16384], mode=ZERO, flags="graph autotune"),
        case("gwb60_noise", [1 << 26], [16384], flags="graph autotune noise_pass"),
        # streams of very different lengths and windows in one call
        case("uneven60", [1 << 22, 1 << 27], [1024, 65536], spread=3, flags="graph autotune noise_pass"),
        # 12-bit samples, dense interference on a drifting baseline
        case("twelve60", [1 << 25], [8192], bits=12, spread=4, k=3.5, flags="graph autotune"),
        # thresholds from the median of 4096 windows' MADs
        case("mom60", [1 << 24], [4096], form="mom", flags="graph noise_pass"),
        # one input filtered with several thresholds and replacements for comparison
        case("copies60", [1 << 22], [16384], form="copies"),
        # fp16 samples for a channeliser that follows
        case("f16_60", [1 << 24], [16384], form="float", mode=CLIP),
        # recorded data in host memory
        case("host60", [1 << 22], [16384], form="host", mode=NOISE),
        # live chunks of 30 inputs with an archive request in the mix
        case("serve30", [1 << 18, 1 << 24], [16384], form="serve", streams=30, spread=5,
             request=(1 << 26) + 1000),
    ]


def draw(rng):
    """One more case: sizes from a few windows of one stream to a quarter of the full batch, any
    window choice, width, replacement and form of call that the listed cases stand for."""
    form = rng.choices(["plan", "mom", "copies", "float", "power", "host", "serve"], [10, 2, 2, 2, 1, 1, 1])[0]
    bits = 12 if form != "copies" and rng.random() < 0.3 else 8
    most = {"plan": 29.5, "mom": 29.5, "copies": 27.5, "float": 29.5, "power": 29.5, "host": 27.5, "serve": 28.0}[form]
    streams = min(60, max(1, int(2 ** rng.uniform(0.0, 6.0))))
    if form == "serve":
        streams = min(30, streams)
    total = 2 ** rng.uniform(17.0, most)
    length = max(2048, int(total / streams))
    wins = rng.choice(["pow2", "pow2", "decimal", "any"])
    if form == "serve":
        wins = "pow2"
    lo = int(2 ** rng.uniform(9.0, 14.5))
    hi = min(65536, lo * rng.choice([1, 1, 4, 16]))
    case = {"form": form, "bits": bits, "streams": streams, "wins": wins, "spread": rng.randrange(1 << 20),
            "len_lo": length, "len_hi": length if rng.random() < 0.5 else int(length * rng.uniform(1.1, 4.0)),
            "win_lo": lo, "win_hi": hi, "k": rng.choice([3.0, 3.5, 4.0, 5.0]),
            "mode": rng.choice([ZERO, CONST, CLIP, NOISE, NOISE]), "flags": rng.choice(["", "graph", "graph"])}
    if form in ("plan", "mom") and case["mode"] == NOISE and rng.random() < 0.5:
        case["flags"] = (case["flags"] + " noise_pass").strip()
    if form == "plan" and rng.random() < 0.15:
        case["flags"] = "per_stream"
    if form == "float":
        case["bf16"] = bits == 8 and rng.random() < 0.3
    if form == "serve":
        case["request"] = int(2 ** rng.uniform(20.0, 26.0))
    return case


# ---------------------------------------------------------------------------- shapes and buffers
def _shape(case):
    """(stream lengths, window lengths, bursts per sample) of a case."""
    r = np.random.default_rng(case["spread"])
    S = case["streams"]
    a, b = math.log2(case["len_lo"]), math.log2(case["len_hi"])
    lens = [case["len_lo"]] * S if case["len_lo"] == case["len_hi"] else [int(2.0 ** u) for u in r.uniform(a, b, size=S)]
    lo, hi = case["win_lo"], case["win_hi"]
    if case["wins"] == "pow2":
        e0, e1 = int(math.log2(lo)), int(math.log2(hi))
        W = [1 << int(e) for e in r.integers(e0, e1 + 1, size=S)]
    elif case["wins"] == "decimal":
        some = [v for v in DECIMAL if lo <= v <= hi] or [min(DECIMAL, key=lambda v: abs(v - lo))]
        W = [some[int(i)] for i in r.integers(0, len(some), size=S)]
    else:
        W = [int(2.0 ** u) for u in r.uniform(math.log2(lo), math.log2(hi), size=S)]
    if case["form"] == "serve":  # chunks of whole windows that never straddle the ring's end
        lens = [max(w, 1 << int(math.log2(n))) for n, w in zip(lens, W)]
    rates = [5e-3] * S if case["bits"] == 12 else [float(10.0 ** (-4.0 + 2.0 * u))
                                                  for u in np.random.default_rng(case["spread"]).uniform(size=60)][:S]
    return lens, W, rates


def _mom_windows(case):
    return 4096 if case["form"] == "mom" else 0


def _offsets(sizes):
    off, at = [], 0
    for n in sizes:
        off.append(at)
        at += -(-n // ALIGN) * ALIGN
    return off, at


def _parts(t, sizes):
    off, _ = _offsets(sizes)
    return [t[o:o + n] for o, n in zip(off, sizes)]


def _windows(n, W):
    return -(-n // W)


def _fill(x, bits, rate, g):
    """Samples of one stream into x. Noise and bursts add in 1/256 LSB, so that the sum does not
    depend on the order of additions."""
    n, dev = x.numel(), x.device
    sigma, lmax, alo, ahi = (16.0, 64, 5.0, 15.0) if bits == 8 else (120.0, 256, 4.0, 30.0)
    acc = torch.randn(n, device=dev, generator=g).mul_(sigma * 256.0).round_().to(torch.int32)
    if bits == 12:
        ph = torch.rand(1, device=dev, generator=g, dtype=torch.float64)
        t = torch.arange(n, device=dev, dtype=torch.float64).mul_(2.0 ** -20).add_(ph).mul_(2.0 * math.pi)
        acc += t.sin_().mul_(50.0 * 256.0).round_().to(torch.int32)
        del t
    nb = max(1, int(rate * n))
    at = torch.randint(0, n, (nb,), device=dev, generator=g)
    ln = torch.randint(1, lmax + 1, (nb,), device=dev, generator=g)
    amp = torch.rand(nb, device=dev, generator=g).mul_(ahi - alo).add_(alo).mul_(sigma * 256.0).to(torch.int32)
    amp = torch.where(torch.rand(nb, device=dev, generator=g) < 0.5, -amp, amp)
    last = torch.cumsum(ln, 0)
    pos = torch.arange(int(last[-1]), device=dev) + torch.repeat_interleave(at - (last - ln), ln)
    val = torch.repeat_interleave(amp, ln)
    ok = pos < n
    acc.index_add_(0, pos[ok], val[ok])
    lo, hi = (-128, 127) if bits == 8 else (-2048, 2047)
    x.copy_(acc.add_(128).bitwise_right_shift_(8).clamp_(lo, hi))


def _inputs(case, seed, sizes, rates):
    g = torch.Generator(device="cuda").manual_seed(seed)
    _, total = _offsets(sizes)
    x = torch.zeros(total, dtype=torch.int8 if case["bits"] == 8 else torch.int16, device="cuda")
    for part, rate in zip(_parts(x, sizes), rates):
        _fill(part, case["bits"], rate, g)
    return x


class _Memory:
    """Device memory of a server's rings, as torch takes it in; it keeps the server alive."""

    def __init__(self, server, ptr, n, kind):
        self.server = server
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (n,), "typestr": kind, "version": 3}


def _flag_bits(case):
    return sum(FLAGS[f] for f in case["flags"].split())


def _const(case):
    return 1 if case["mode"] == CONST else 0


def prepare(case, seed):
    lens, W, rates = _shape(case)
    S, bits, form = case["streams"], case["bits"], case["form"]
    nwin = [_windows(n, w) for n, w in zip(lens, W)]
    words = [nw * ((w + 31) // 32) for nw, w in zip(nwin, W)]
    x = _inputs(case, seed, lens, rates)
    st = {"case": case, "x": x}
    if form == "serve":
        n = case["request"]
        q = torch.zeros(n, dtype=x.dtype, device="cuda")
        _fill(q, bits, rates[0], torch.Generator(device="cuda").manual_seed(seed + (1 << 40)))
        nq, mw = _windows(n, W[0]), (W[0] + 31) // 32
        ring = 2 * max(lens)
        budget = sum(2 * (ring + w) * x.element_size() + (ring // w + 1) * ((w + 31) // 32 + 3) * 4 + 4096 for w in W) + (64 << 20)
        st["server"] = rfi.Server(bits, W, ring, case["k"], case["mode"], _const(case), SEED, memory_budget=budget)
        st.update(ins=_parts(x, lens), lens=lens, q=q, W0=W[0], qz=torch.zeros_like(q),
                  qmask=torch.zeros(nq * mw, dtype=torch.int32, device="cuda"),
                  qcounts=torch.zeros(nq, dtype=torch.int32, device="cuda"), at=[0] * S, words=[(w + 31) // 32 for w in W],
                  W=W)
        torch.cuda.synchronize()  # the server copies on its own streams
        return st
    zt = x.dtype if form != "float" else (torch.bfloat16 if case.get("bf16") else torch.float16)
    nv = len(VARIANTS) if form == "copies" else 1
    z = [torch.zeros(_offsets(lens)[1], dtype=zt, device="cuda") for _ in range(nv)]
    mask = [torch.zeros(_offsets(words)[1], dtype=torch.int32, device="cuda") for _ in range(nv)]
    counts = [torch.zeros(_offsets(nwin)[1], dtype=torch.int32, device="cuda") for _ in range(nv)]
    flags = _flag_bits(case)
    if form == "copies":
        st["plan"] = rfi.CopiesPlan(bits, lens, W, VARIANTS, flags)
    else:
        if form == "power":
            flags |= rfi.RFI_PLAN_POWER
            st["power"] = torch.zeros(2 * _offsets(nwin)[1], dtype=torch.int64, device="cuda")
            st["powers"] = _parts(st["power"], [2 * n for n in nwin])
        st["plan"] = rfi.Plan(bits, lens, W, case["k"], case["mode"], _const(case), SEED, flags, mom_windows=_mom_windows(case),
                              out_format=0 if form != "float" else (rfi.RFI_OUT_BF16 if case.get("bf16") else rfi.RFI_OUT_F16))
    if form == "host":
        x, z, mask, counts = x.cpu().pin_memory(), [z[0].cpu().pin_memory()], [mask[0].cpu().pin_memory()], [counts[0].cpu().pin_memory()]
        st["x"] = x
    st.update(z=z, mask=mask, counts=counts, ins=_parts(x, lens), outs=[_parts(t, lens) for t in z],
              masks=[_parts(t, words) for t in mask], cnts=[_parts(t, nwin) for t in counts])
    return st


def _serve(st):
    sv, at, res = st["server"], st["at"], {"chunks": [], "masks": []}
    for s, c in enumerate(st["ins"]):
        rfi.check(sv.push(s, c)[0], "rfi_server_push")
    rfi.check(sv.submit(st["q"], st["qz"], st["W0"], stream_id=1000, mask=st["qmask"], counts=st["qcounts"])[0],
              "rfi_server_submit")
    sv.drain()
    kind = "|i1" if sv.bits == 8 else "<i2"
    for s, n in enumerate(st["lens"]):
        status, out, mask, there = sv.view(s, at[s])
        rfi.check(status, "rfi_server_view")
        if there < n:
            raise RuntimeError("stream %d: %d of %d samples are there" % (s, there, n))
        res["chunks"].append(torch.as_tensor(_Memory(sv, out, n, kind), device="cuda"))
        res["masks"].append(torch.as_tensor(_Memory(sv, mask, n // st["W"][s] * st["words"][s], "<i4"), device="cuda"))
        at[s] += n
        rfi.check(sv.release(s, at[s]), "rfi_server_release")
    return {**res, "request": st["qz"], "request_mask": st["qmask"], "request_counts": st["qcounts"]}


def run(state):
    form = state["case"]["form"]
    if form == "serve":
        return _serve(state)
    plan = state["plan"]
    if form == "copies":
        plan.excise(state["ins"], state["outs"], state["masks"], state["cnts"])
    elif form == "host":
        plan.excise_host(state["ins"], state["outs"][0], state["masks"][0], state["cnts"][0])
    else:
        plan.excise(state["ins"], state["outs"][0], state["masks"][0], state["cnts"][0])
    res = {"out": state["z"], "mask": state["mask"], "counts": state["counts"]}
    if form == "power":
        plan.stats_power(state["powers"])
        res["power"] = state["power"]
    return res


def work(case):
    """Every sample read once; every output sample, mask word and count written once."""
    lens, W, _ = _shape(case)
    bps = 1 if case["bits"] == 8 else 2
    obps = 2 if case["form"] == "float" else bps
    nv = len(VARIANTS) if case["form"] == "copies" else 1
    if case["form"] == "serve":
        lens, W = lens + [case["request"]], W + [W[0]]
    total = 0
    for n, w in zip(lens, W):
        nw = _windows(n, w)
        total += n * bps + nv * (n * obps + nw * (4 * ((w + 31) // 32) + 4))
        if case["form"] == "power":
            total += 16 * nw
    return {"bytes": total, "flops": 0}


# ---------------------------------------------------------------------------- in 64-bit integers
def _noise(M, D, idx, stream, bits):
    """M plus the digital noise of sample idx: Philox4x32-10 (Salmon et al., SC'11) keyed by the
    seed, the eight 16-bit halves summed and scaled by 1.4826 D, rounded half away from zero."""
    m32 = 0xFFFFFFFF
    c = [idx & m32, idx >> 32, torch.full_like(idx, stream), torch.zeros_like(idx)]
    k0, k1 = SEED & m32, SEED >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        h0, h1 = (p0 >> 32) & m32, (p1 >> 32) & m32
        c = [h1 ^ c[1] ^ k0, p1 & m32, h0 ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    s = sum((v & 0xFFFF) + (v >> 16) for v in c)
    s2 = 2 * s - 8 * 65535
    den = 107020 * 65536
    q = (s2.abs() * 97164 * D + den // 2) // den
    lo, hi = (-128, 127) if bits == 8 else (-2048, 2047)
    return (M + torch.where(s2 < 0, -q, q)).clamp(lo, hi)


def _pack(fl, W):
    """Flags [windows, W] to mask words, sample j of a window at bit j % 32 of its word j / 32."""
    mw = (W + 31) // 32
    fl = torch.nn.functional.pad(fl, (0, 32 * mw - W)).view(-1, mw, 32).to(torch.int64)
    v = (fl << torch.arange(32, device=fl.device)).sum(-1)
    return torch.where(v >= 1 << 31, v - (1 << 32), v).to(torch.int32).reshape(-1)


def _median_mad(x, W):
    """Lower median and lower median absolute deviation of every window."""
    M, D, n = [], [], x.numel()
    full = n // W
    for part in ([x[:full * W].view(full, W)] if full else []) + ([x[full * W:].view(1, -1)] if n % W else []):
        for rows in part.split(max(1, (1 << 24) // part.shape[1])):
            m = rows.to(torch.int16).median(dim=1).values
            M.append(m)
            D.append((rows.to(torch.int16) - m[:, None]).abs().median(dim=1).values)
    return torch.cat(M).to(torch.int64), torch.cat(D).to(torch.int64)


def _sliding_median(D, k):
    """Lower median of D[max(0, j - k + 1) .. j] for every j."""
    res, top = [], int(D.max()) + 1
    c = torch.zeros(D.numel() + 1, top, dtype=torch.int32, device=D.device)
    c[1:] = torch.nn.functional.one_hot(D, top).to(torch.int32).cumsum(0)
    j = torch.arange(D.numel(), device=D.device)
    for rows in j.split(1 << 16):
        cnt = torch.clamp(rows + 1, max=k)
        h = (c[rows + 1] - c[torch.clamp(rows + 1 - k, min=0)]).cumsum(1)
        res.append((h < ((cnt + 1) // 2)[:, None]).sum(1))
    return torch.cat(res)


def _excised(x, W, M, D, k, mode, const, stream, bits):
    """(samples, mask, counts) of one stream."""
    kq = math.floor(k * 1.4826 * 65536 + 0.5)
    t, c = (kq * D + 65535) >> 16, (kq * D) >> 16
    lo, hi = (-128, 127) if bits == 8 else (-2048, 2047)
    n, nwin = x.numel(), M.numel()
    z, mask, counts = torch.empty_like(x), [], []
    step = max(1, (1 << 24) // W)
    for w0 in range(0, nwin, step):
        w1 = min(nwin, w0 + step)
        xs = x[w0 * W:min(n, w1 * W)].to(torch.int64)
        pad = (w1 - w0) * W - xs.numel()
        xs = torch.nn.functional.pad(xs, (0, pad)).view(w1 - w0, W)
        m, d, tt, cc = (v[w0:w1, None] for v in (M, D, t, c))
        fl = ((xs - m).abs() >= tt) & (d > 0)
        if pad:
            fl[-1, W - pad:] = False
        if mode == NOISE:
            r, col = torch.nonzero(fl, as_tuple=True)
            zs = xs.clone()
            zs[r, col] = _noise(M[w0 + r], D[w0 + r], (w0 + r) * W + col, stream, bits)
        else:
            rep = torch.where(xs > m, m + cc, m - cc).clamp(lo, hi) if mode == CLIP else torch.full_like(xs, const if mode == CONST else 0)
            zs = torch.where(fl, rep, xs)
        z[w0 * W:min(n, w1 * W)] = zs.view(-1)[:zs.numel() - pad].to(x.dtype)
        mask.append(_pack(fl, W))
        counts.append(fl.sum(1).to(torch.int32))
    return z, torch.cat(mask), torch.cat(counts)


def exact(case, seed):
    lens, W, rates = _shape(case)
    bits, form = case["bits"], case["form"]
    nwin = [_windows(n, w) for n, w in zip(lens, W)]
    words = [nw * ((w + 31) // 32) for nw, w in zip(nwin, W)]
    x = _inputs(case, seed, lens, rates)
    xs = _parts(x, lens)
    if form == "serve":
        res = {"chunks": [], "masks": []}
        for s, p in enumerate(xs):
            z, m, _ = _excised(p, W[s], *_median_mad(p, W[s]), case["k"], case["mode"], _const(case), s, bits)
            res["chunks"].append(z)
            res["masks"].append(m)
        q = torch.zeros(case["request"], dtype=x.dtype, device="cuda")
        _fill(q, bits, rates[0], torch.Generator(device="cuda").manual_seed(seed + (1 << 40)))
        z, m, c = _excised(q, W[0], *_median_mad(q, W[0]), case["k"], case["mode"], _const(case), 1000, bits)
        return {**res, "request": z, "request_mask": m, "request_counts": c}
    variants = VARIANTS if form == "copies" else [(case["k"], case["mode"], _const(case), SEED)]
    zt = x.dtype if form != "float" else (torch.bfloat16 if case.get("bf16") else torch.float16)
    z = [torch.zeros(_offsets(lens)[1], dtype=zt, device="cuda") for _ in variants]
    mask = [torch.zeros(_offsets(words)[1], dtype=torch.int32, device="cuda") for _ in variants]
    counts = [torch.zeros(_offsets(nwin)[1], dtype=torch.int32, device="cuda") for _ in variants]
    power = torch.zeros(2 * _offsets(nwin)[1], dtype=torch.int64, device="cuda")
    for s, p in enumerate(xs):
        M, D = _median_mad(p, W[s])
        if form == "mom":
            D = _sliding_median(D, _mom_windows(case))
        for v, (k, mode, const, _) in enumerate(variants):
            a, b, c = _excised(p, W[s], M, D, k, mode, const, s, bits)
            _parts(z[v], lens)[s].copy_(a)
            _parts(mask[v], words)[s].copy_(b)
            _parts(counts[v], nwin)[s].copy_(c)
            if form == "power":
                for j, t in enumerate((p, a)):
                    sq = torch.nn.functional.pad(t.to(torch.int64) ** 2, (0, nwin[s] * W[s] - lens[s]))
                    _parts(power, [2 * n for n in nwin])[s][j::2] = sq.view(nwin[s], W[s]).sum(1)
    res = {"out": z, "mask": mask, "counts": counts}
    if form == "power":
        res["power"] = power
    return res
