"""Timed cases of the library's public calls: what a Read Until program has it do.

Every case is one call (or one burst of serving calls) of
paper_2211_07340_gb300.Context on seeded synthetic nanopore data: a random
genome read through a random 6-mer pore model, half of the reads from that
genome and half from an unrelated one, levels skipped with probability 0.1
and otherwise emitted one to three times with 2 pA noise (raw-signal reads:
an adaptor, then levels held for about ten noisy ADC samples each).
"""
import math

import numpy as np
import torch

import paper_2211_07340_gb300 as haru

PRECISION = {"int16": haru.HARU_INT16, "fp32": haru.HARU_FP32, "acc32": haru.HARU_INT16_ACC32}
SARS_BASES = 29_903     # SARS-CoV-2: 59,796 reference columns
RFC1_BASES = 128_915    # RFC1: 257,820 columns
LONG_BASES = 5_000_000  # 9,999,990 columns
K = 6
# The launch shape haru_autotune keeps for large batches; other cases run the default one.
TUNED = {"warps_per_cta": 12, "tile_cols": 16384}


def _case(name, call, nq, lo, hi, bases=SARS_BASES, form="int16", tuned=False, scale=6):
    c = {"call": call, "nq": nq, "lo": lo, "hi": hi, "bases": bases, "form": form, "tuned": tuned, "scale": scale}
    return dict(c, name=name) if name else c


def listed():
    return [
        # One read's decision through the host call: the latency of a single Read Until request.
        _case("host_1x250_int16", "host", 1, 250, 250),
        # A handful of reads in the plain form, results left on the device.
        _case("device_32x250_fp32", "device", 32, 250, 250, form="fp32"),
        # What one loop turn of a busy flow cell gathers: a mid-sized batch of full and cut prefixes.
        _case("device_100_uneven_int16", "device", 100, 120, 250),
        # The serving loop: 96 channels deliver their prefix at once, every decision is collected.
        _case("serve_96x250_int16", "serve", 96, 250, 250),
        # Mapping accepted reads: start and end columns, uneven lengths.
        _case("span_512_uneven_fp32", "span", 512, 100, 500, form="fp32"),
        # The exact-integer form at the size of the precision study, through the host call.
        _case("host_4096x250_acc32", "host", 4096, 250, 250, form="acc32"),
        # Offline throughput: thousands of reads of uneven length, in both main forms.
        _case("device_8192_uneven_int16", "device", 8192, 100, 500, tuned=True),
        _case("device_8192_uneven_fp32", "device", 8192, 100, 500, form="fp32", tuned=True),
        # A gene-sized target, and a bacterial-genome-sized one.
        _case("device_512x250_rfc1_int16", "device", 512, 250, 250, bases=RFC1_BASES),
        _case("device_512x250_long_int16", "device", 512, 250, 250, bases=LONG_BASES, tuned=True),
        # From raw ADC samples: events detected on the device, then aligned; and detection alone.
        _case("signal_1000_int16", "signal", 1000, 250, 250),
        _case("detect_8192_uneven", "detect", 8192, 100, 500),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    call = rng.choice(["device"] * 5 + ["host"] * 3 + ["span"] * 2 + ["signal", "detect", "serve"])
    forms = {"span": ["fp32", "acc32"], "serve": ["int16", "fp32"], "detect": ["int16"]}
    form = rng.choice(forms.get(call, ["int16", "int16", "fp32", "acc32"]))
    lo = rng.randint(30, 400) if call in ("device", "host", "span") else rng.randint(100, 300)
    hi = rng.randint(lo, 500)
    if call == "serve":  # the loop decides on one prefix length
        lo = hi = rng.randint(100, 300)
    bases = log(200_000, LONG_BASES) if rng.random() < 0.1 else log(3_000, 150_000)
    nq = log(1, 300 if call == "serve" else 8192)
    # at most what the largest listed case costs, each form at its own speed
    most = {"int16": 5e11, "fp32": 3e11, "acc32": 3e11}[form] * (0.4 if call == "span" else 1.0)
    nq = max(1, min(nq, int(most / (2 * bases * hi))))
    return _case(None, call, nq, lo, hi, bases=bases, form=form,
                 tuned=nq > 2000 and rng.random() < 0.5, scale=rng.choice([5, 6, 6, 7]))


# ------------------------------------------------------------------ inputs --
def _codes(bases):
    n = bases.shape[0] - K + 1
    code = torch.zeros(n, dtype=torch.int64, device=bases.device)
    for u in range(K):
        code = code * 4 + bases[u:u + n].long()
    return code


def _strands(bases, model):
    """Levels along the forward strand, then along the reverse complement."""
    b = torch.from_numpy(bases).cuda()
    return torch.cat([model[_codes(b)], model[_codes((3 - b).flip(0))]])


def _inputs(case, seed):
    """Genome and pore model (host), levels of both genomes, and a seeded generator."""
    rng = np.random.default_rng(seed)
    genome = rng.integers(0, 4, case["bases"], dtype=np.uint8)
    other = rng.integers(0, 4, min(case["bases"], RFC1_BASES), dtype=np.uint8)
    model = rng.normal(90.0, 12.0, 4 ** K).astype(np.float32)
    dm = torch.from_numpy(model).cuda()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lengths = torch.randint(case["lo"], case["hi"] + 1, (case["nq"],), generator=gen, device="cuda")
    return genome, model, _strands(genome, dm), _strands(other, dm), lengths, gen


def _walk(on, off, span, nq, gen):
    """[nq, span] consecutive levels from a random place and strand: even reads on target, odd ones off."""
    out = []
    for levels in (on, off):
        half = levels.shape[0] // 2
        start = (torch.rand(nq, generator=gen, device="cuda") * max(1, half - span)).long()
        start += half * torch.randint(0, 2, (nq,), generator=gen, device="cuda")
        at = start[:, None] + torch.arange(span, device="cuda")
        out.append(levels[at.clamp_(max=levels.shape[0] - 1)])
    return torch.where((torch.arange(nq, device="cuda") % 2 == 0)[:, None], out[0], out[1])


def _offsets(lengths):
    off = torch.zeros(lengths.shape[0] + 1, dtype=torch.int64, device="cuda")
    off[1:] = lengths.cumsum(0)
    return off


def _events(on, off, lengths, gen):
    """Raw event currents in CSR form: (events float32, offsets int64)."""
    nq, m = lengths.shape[0], int(lengths.max())
    span = m + 64  # levels emit 1.4 events each on average
    walk = _walk(on, off, span, nq, gen)
    u = torch.rand(nq, span, generator=gen, device="cuda")
    dwell = torch.where(u < 0.1, 0, torch.where(u < 0.614, 1, torch.where(u < 0.871, 2, 3)))
    e = torch.arange(m, device="cuda").expand(nq, m).contiguous()
    src = torch.searchsorted(dwell.cumsum(1), e, right=True).clamp_(max=span - 1)
    ev = walk.gather(1, src) + 2.0 * torch.randn(nq, m, generator=gen, device="cuda")
    return ev[e < lengths[:, None]].contiguous(), _offsets(lengths)


def _signal(on, off, lengths, gen):
    """Raw ADC samples in CSR form: 50 adaptor levels, then the levels of about `lengths` events."""
    nq = lengths.shape[0]
    span = int(lengths.max()) * 5 // 4 + 16
    walk = torch.cat([75.0 + 8.0 * torch.randn(nq, 50, generator=gen, device="cuda"), _walk(on, off, span, nq, gen)], 1)
    u = torch.rand(nq, 50 + span, generator=gen, device="cuda").clamp_(min=1e-6)
    dwell = 4 + (u.log() / math.log(6.0 / 7.0)).long()
    skip = torch.rand(nq, 50 + span, generator=gen, device="cuda") < 0.1
    skip[:, :50] = False
    level = torch.arange(50 + span, device="cuda") - 50
    dwell = dwell.masked_fill(skip | (level >= (lengths * 5 // 4 + 16)[:, None]), 0)
    pa = torch.repeat_interleave(walk.reshape(-1), dwell.reshape(-1))
    pa = pa + 2.5 * torch.randn(pa.shape[0], generator=gen, device="cuda")
    return ((pa * (8192 / 1402.1)).round() - 10).to(torch.int16), _offsets(dwell.sum(1))


def _data(case, seed):
    genome, model, on, off, lengths, gen = _inputs(case, seed)
    make = _signal if case["call"] in ("signal", "detect") else _events
    x, offsets = make(on, off, lengths, gen)
    return genome, model, on, x, offsets


_stream = []


def _program_stream():
    """The one stream the program queues its device calls on."""
    if not _stream:
        _stream.append(torch.cuda.Stream())
    return _stream[0].cuda_stream


def prepare(case, seed):
    genome, model, _, x, off = _data(case, seed)
    nq, call = case["nq"], case["call"]
    cfg = dict(TUNED) if case["tuned"] else {}
    if call == "serve":
        cfg.update(serve_precision=PRECISION[case["form"]], serve_prefix=case["hi"], threshold=80.0)
    ctx = haru.Context(0, **cfg)
    ctx.ref_build(genome, model, K, scale_log2=case["scale"])
    s = {"case": case, "ctx": ctx, "form": PRECISION[case["form"]]}
    if call in ("host", "serve"):
        s["x"], s["off"] = x.cpu().numpy(), off.cpu().numpy().astype(np.uint32)
        s["next_id"] = 0
    else:
        s["x"], s["off"] = x, off.to(torch.int32)  # same bits as uint32
        s["cost"] = torch.empty(nq, dtype=torch.float32, device="cuda")
        s["col"] = torch.empty(nq, dtype=torch.int64, device="cuda")
        s["start"] = torch.empty(nq, dtype=torch.int64, device="cuda")
        s["count"] = torch.empty(nq, dtype=torch.int32, device="cuda")
        s["events"] = torch.zeros(nq * 250 if call == "detect" else 1, dtype=torch.float32, device="cuda")
        s["event_off"] = torch.empty(nq + 1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    return s


def _serve(s):
    ctx, x, off, nq = s["ctx"], s["x"], s["off"], s["case"]["nq"]
    first, s["next_id"] = s["next_id"], s["next_id"] + nq
    for q in range(nq):
        haru.check(ctx.stream_submit(first + q, q, x[off[q]:off[q + 1]], 0, True))
    cost, col, accept = np.empty(nq, np.float32), np.empty(nq, np.int64), np.empty(nq, np.int32)
    left = nq
    while left:
        got = ctx.stream_poll(nq, 2_000_000)
        if not got:
            raise RuntimeError("no decision within two seconds")
        for r in got:
            haru.check(r.status)
            q = r.read_id - first
            cost[q], col[q], accept[q] = r.cost, r.end_col, r.decision
            left -= 1
    return {"cost": cost, "col": col, "accept": accept}


def run(s):
    ctx, call = s["ctx"], s["case"]["call"]
    if call == "host":
        cost, col = ctx.sdtw_batch(s["form"], s["x"], s["off"])
        return {"cost": cost, "col": col}
    if call == "serve":
        return _serve(s)
    st = _program_stream()
    if call == "device":
        ctx.sdtw_batch_device(s["form"], s["x"], s["off"], s["cost"], s["col"], stream=st, asynchronous=True)
        return {"cost": s["cost"], "col": s["col"]}
    if call == "span":
        ctx.sdtw_batch_span_device(s["form"], s["x"], s["off"], s["cost"], s["col"], s["start"], stream=st,
                                   asynchronous=True)
        return {"cost": s["cost"], "col": s["col"], "start": s["start"]}
    if call == "signal":
        ctx.sdtw_batch_signal_device(s["form"], s["x"], s["off"], s["cost"], s["col"], s["count"], stream=st,
                                     asynchronous=True)
        return {"cost": s["cost"], "col": s["col"], "count": s["count"]}
    ctx.detect_events_device(s["x"], s["off"], s["events"], s["event_off"], stream=st, asynchronous=True)
    return {"events": s["events"], "event_off": s["event_off"]}


def work(case):
    """Bytes: events or samples, the reference once in the form the sweep reads it, and the results.
    Operations: five per cell (subtract, magnitude, a minimum of three, add); ten per sample for detection."""
    nq, m, n = case["nq"], (case["lo"] + case["hi"]) / 2, 2 * (case["bases"] - K + 1)
    samples = nq * (50 + 0.9 * (1.25 * m + 16)) * 10
    if case["call"] == "detect":
        return {"bytes": 2 * samples + 4 * nq * min(m, 250) + 8 * nq, "flops": 10 * samples}
    if case["call"] == "signal":
        m = min(m, 250)
        return {"bytes": 2 * samples + 4 * n + 20 * nq, "flops": 10 * samples + 5 * nq * m * n}
    return {"bytes": 4 * nq * m + 4 * n + (24 if case["call"] == "span" else 16) * nq, "flops": 5 * nq * m * n}


# ------------------------------------------------------------------- exact --
def _exact_events(x, off):
    """Events of every read: [nq, 250] means in 64 bits and their counts. Windows of 3 and 6 samples,
    thresholds 1.40 and 9.00; a peak is above its threshold, above the w statistics before it and not below
    the w after it; short-window peaks count where no long-window peak is within 3; the first 50 events go."""
    nq, n = off.shape[0] - 1, off[1:] - off[:-1]
    out = torch.zeros(nq, 250, dtype=torch.float64, device="cuda")
    count = torch.zeros(nq, dtype=torch.int64, device="cuda")
    for lo in range(0, nq, 512):
        hi = min(nq, lo + 512)
        nn, w = n[lo:hi, None], int(n[lo:hi].max())
        at = torch.arange(w, device="cuda")
        v = torch.where(at < nn, x[(off[lo:hi, None] + at).clamp_(max=x.shape[0] - 1)].double(), 0.0)
        zero = torch.zeros(hi - lo, 1, dtype=torch.float64, device="cuda")
        s1, s2 = torch.cat([zero, v.cumsum(1)], 1), torch.cat([zero, (v * v).cumsum(1)], 1)

        def peaks(win, centi):
            t = torch.full((hi - lo, w), -1.0, dtype=torch.float64, device="cuda")
            p = at[win:w - win + 1] if w >= 2 * win else at[:0]
            a, b = s1[:, p] - s1[:, p - win], s1[:, p + win] - s1[:, p]
            qq = s2[:, p + win] - s2[:, p - win]
            num, den = win * (b - a) ** 2, (win * qq - a * a - b * b).clamp_(min=1.0)
            t[:, p] = num / den
            t.masked_fill_(at > nn - win, -1.0)
            ok = torch.zeros_like(t, dtype=torch.bool)
            ok[:, p] = 1e4 * num > centi * centi * den  # whole numbers: t above the threshold, exactly
            ok &= t >= 0
            for k in range(1, win + 1):
                ok[:, k:] &= t[:, k:] > t[:, :-k]
                ok[:, :-k] &= t[:, :-k] >= t[:, k:]
            return ok

        long_, short = peaks(6, 900), peaks(3, 140)
        near = torch.nn.functional.max_pool1d(long_.float()[:, None], 7, 1, 3)[:, 0] > 0
        bound = (long_ | (short & ~near)) & (at >= 1) & (at <= nn - 1)
        event = bound.long().cumsum(1) - 50  # the event each sample belongs to, after the trim
        keep = (at < nn) & (event >= 0) & (event < 250)
        idx = event.clamp(0, 249)
        total, length = torch.zeros_like(out[lo:hi]), torch.zeros_like(out[lo:hi])
        total.scatter_add_(1, idx, torch.where(keep, v, 0.0))
        length.scatter_add_(1, idx, keep.double())
        out[lo:hi] = total / length.clamp(min=1.0)
        count[lo:hi] = (length > 0).sum(1)
    return out, count


def _exact_cost(case, q, m, levels):
    """Smallest last-row value per query of Eq. 1 in 64 bits. q: [nq, H] raw events, right-aligned; m: lengths.
    The cells of one step lie on an oblique column: row i at reference column t - i. Rows above a query are
    free-start rows (distance 0)."""
    nq, h = q.shape
    real = (torch.arange(h, device="cuda") >= h - m[:, None]).double()
    mean = (q * real).sum(1, keepdim=True) / m[:, None]
    sd = (((q - mean) * real).square().sum(1, keepdim=True) / m[:, None]).sqrt()
    z, ref = (q - mean) / sd, levels.double()
    ref = (ref - ref.mean()) / ref.std(unbiased=False)
    if case["form"] != "fp32":
        scale = float(1 << case["scale"])
        z, ref = ((v.float() * scale).round().clamp(-2047, 2047).double() for v in (z, ref))
    n = ref.shape[0]
    far = torch.full((h,), 1e30, dtype=torch.float64, device="cuda")
    back = torch.cat([far, ref, far]).flip(0)  # reversed, so that row i at step t sits i to the right
    z = z * real
    g = [torch.full((nq, h + 1), 1e30, dtype=torch.float64, device="cuda") for _ in range(3)]
    for x in g:
        x[:, 0] = 0.0
        x[:, 1:] *= real
    best = torch.full((nq,), 1e30, dtype=torch.float64, device="cuda")
    d = torch.empty(nq, h, dtype=torch.float64, device="cuda")
    for t in range(n + h - 1):
        a = n + h - 1 - t
        new, one, two = g[t % 3], g[(t + 2) % 3], g[(t + 1) % 3]
        torch.addcmul(z, real, back[a:a + h], value=-1.0, out=d)
        torch.minimum(one[:, :-1], two[:, :-1], out=new[:, 1:])
        torch.minimum(new[:, 1:], one[:, 1:], out=new[:, 1:])
        new[:, 1:].add_(d.abs_())
        if t >= h - 1:
            torch.minimum(best, new[:, -1], out=best)
    if case["form"] != "fp32":
        best = (best.clamp(max=28673) if case["form"] == "int16" else best) / scale
    return best


def exact(case, seed):
    nq, h, n = case["nq"], case["hi"], 2 * (case["bases"] - K + 1)
    if case["call"] in ("signal", "detect"):
        _, _, levels, x, off = _data(case, seed)
        ev, count = _exact_events(x, off)
        if case["call"] == "detect":
            flat = torch.zeros(nq * 250, dtype=torch.float64, device="cuda")
            got = ev[torch.arange(250, device="cuda") < count[:, None]]
            flat[:got.shape[0]] = got
            return {"events": flat, "event_off": None}
        h = 250
    if n * max(5e-5, nq * h * 4e-11) > 12.0:  # seconds, about
        return None
    if case["call"] == "signal":
        at = torch.arange(250, device="cuda") - (250 - count[:, None])
        q = torch.where(at >= 0, ev.float().double().gather(1, at.clamp(min=0)), 0.0)
        return {"cost": _exact_cost(case, q, count, levels), "col": None, "count": None}
    _, _, levels, x, off = _data(case, seed)
    m = off[1:] - off[:-1]
    at = torch.arange(h, device="cuda") - (h - m[:, None])
    q = torch.where(at >= 0, x[(off[:-1, None] + at.clamp(min=0)).clamp_(max=x.shape[0] - 1)].double(), 0.0)
    out = {"cost": _exact_cost(case, q, m, levels), "col": None}
    if case["call"] == "span":
        out["start"] = None
    if case["call"] == "serve":
        out["accept"] = None
    return out
