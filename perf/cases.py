"""What the period search is used for, as cases that can be timed.

Each case is one call (or the two or three calls that belong together) of the
public binding: whole searches over short and long series, batches of
dedispersion trials, and the steps of a search through their own entry points
(folding one base period, scoring a set of profiles, dereddening a series).
"""
import math

import numpy as np
import torch

from paper_1703_05581_gb300 import ffa

SURVEY_TSAMP = 64e-6     # the survey's sampling interval (s)
PLAIN_TSAMP = 2.048e-3   # the plain workload's
BATCH_TSAMP = 512e-6     # dedispersion trials


def listed():
    return [
        # The plain workload: one short series, 256 base periods of 256..511
        # bins, and its best 64 candidates.  The smallest whole search: launch
        # and host latency count.
        dict(name="plain_search", kind="search", n=65536, tsamp=PLAIN_TSAMP, pmin=256 * PLAIN_TSAMP,
             pmax=512 * PLAIN_TSAMP, duty=0.0, d0=1, u8=False, i8=False, clip=0.0, top_k=64, pulse=0.8),
        # A survey beam as the paper searches it (2^26 8-bit samples, D0 = 64,
        # 1-30 s): short profiles, many rows, several octaves, then candidates.
        dict(name="beam_u8_d64", kind="search", n=1 << 26, tsamp=SURVEY_TSAMP, pmin=1.0, pmax=30.0,
             duty=0.1, d0=64, u8=True, i8=False, clip=0.0, top_k=256, pulse=7.3),
        # The survey at full time resolution over one band of periods (a known
        # source, or one process's share): base periods of 19 532..20 000
        # bins, 4096 rows, FP32.
        dict(name="band_20k_f32", kind="search", n=1 << 26, tsamp=SURVEY_TSAMP, pmin=1.25, pmax=1.28,
             duty=0.1, d0=1, u8=False, i8=False, clip=0.0, top_k=0, pulse=1.266),
        # The same at the survey's longest profiles (29 375..29 687 bins) in
        # the int8 code: the largest case.
        dict(name="band_30k_i8", kind="search", n=1 << 26, tsamp=SURVEY_TSAMP, pmin=1.88, pmax=1.90,
             duty=0.1, d0=1, u8=False, i8=True, clip=0.0, top_k=0, pulse=1.889),
        # Dedispersion trials of uneven length searched together, 0.5-20 s.
        dict(name="batch_f32", kind="batch", series=12, lo=1 << 19, hi=1 << 20, i8=False),
        # Fewer and longer ones in the int8 code.
        dict(name="batch_i8", kind="batch", series=4, lo=1 << 20, hi=1 << 21, i8=True),
        # One base period folded on its own: the survey's shape (long rows,
        # an odd pitch), every trial's profile written.
        dict(name="fold_f32_long", kind="fold", p0=19977, m_data=3359, i8=False),
        # A dedispersion trial's shape: short odd rows, many of them, int8.
        dict(name="fold_i8_short", kind="fold", p0=1489, m_data=5632, i8=True),
        # Algorithm 1 on ready profiles: short ones, FP32, widths to 20 % duty.
        dict(name="score_f32_short", kind="score", p0=1489, count=8192, i32=False, alg=1),
        # Long integer profiles (an int8 fold's).
        dict(name="score_i32_long", kind="score", p0=12011, count=2048, i32=True, alg=1),
        # Algorithm 2 on profiles of ordinary length.
        dict(name="score_alg2", kind="score", p0=4201, count=4096, i32=False, alg=2),
        # Dereddening and normalising a long series with the survey's window.
        dict(name="deredden", kind="prep", n=1 << 24, window=62501, i8=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "band", "batch", "fold", "fold", "score", "score", "alg2", "prep"])
    if kind == "search":
        # a short series, or a long one downsampled to a short one
        d0 = rng.choice([1, 1, 2, 4, 16, 64])
        n0 = _log(rng, 1 << 15, 1 << 19)
        p0 = _log(rng, 64, 1200)
        ts = rng.choice([PLAIN_TSAMP, BATCH_TSAMP])
        span = rng.uniform(1.2, 6.0)
        return dict(kind="search", n=n0 * d0 + rng.randrange(d0), tsamp=ts, pmin=p0 * ts * d0,
                    pmax=p0 * ts * d0 * span, duty=rng.choice([0.0, 0.1, 0.2]), d0=d0, u8=rng.random() < 0.4,
                    i8=rng.random() < 0.4, clip=rng.choice([0.0, 0.0, 4.0]), top_k=rng.choice([0, 16, 64]),
                    pulse=p0 * ts * d0 * rng.uniform(1.05, 1.2))
    if kind == "band":
        # a band of base periods at full resolution
        n = _log(rng, 1 << 24, 1 << 26)
        p0 = _log(rng, 4000, 30000)
        bands = max(8, int(160 * (1 << 26) / n * 20000 / p0 / 4))
        pmin = p0 * SURVEY_TSAMP
        return dict(kind="search", n=n, tsamp=SURVEY_TSAMP, pmin=pmin, pmax=(p0 + bands) * SURVEY_TSAMP,
                    duty=rng.choice([0.1, 0.2]), d0=1, u8=rng.random() < 0.3, i8=rng.random() < 0.4, clip=0.0,
                    top_k=0, pulse=(p0 + bands / 2) * SURVEY_TSAMP)
    if kind == "batch":
        lo = _log(rng, 1 << 18, 1 << 20)
        return dict(kind="batch", series=rng.randrange(2, 9), lo=lo, hi=int(lo * rng.uniform(1.1, 2.0)),
                    i8=rng.random() < 0.5)
    if kind == "fold":
        p0 = _log(rng, 200, 31000)
        return dict(kind="fold", p0=p0, m_data=min(_log(rng, 40, 8000), 100_000_000 // p0), i8=rng.random() < 0.4)
    if kind == "prep":
        return dict(kind="prep", n=_log(rng, 1 << 18, 1 << 24), window=_log(rng, 900, 62501) | 1, i8=rng.random() < 0.4)
    p0 = _log(rng, 200, 31000)
    return dict(kind="score", p0=p0, count=max(1, min(_log(rng, 100, 8192), 80_000_000 // p0)),
                i32=rng.random() < 0.4, alg=2 if kind == "alg2" else 1)


# ---- inputs -------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _red(g, rows, n, coef, std):
    """Stationary AR(1) rows (std in units of the white noise's)."""
    r = torch.randn((rows, n), generator=g, device="cuda") * (std * math.sqrt(1 - coef * coef))
    s = 1
    while s < n and coef ** s > 1e-4:
        r[:, s:] += coef ** s * r[:, :-s].clone()
        s *= 2
    return r


def _series(n, seed, pulse=0.0, snr=15.0):
    """White noise, AR(1) red noise and a train of Gaussian pulses of period
    `pulse` samples: a dedispersed series."""
    g = _gen(seed)
    x = torch.randn(n, generator=g, device="cuda") + _red(g, 1, n, 0.999, 0.3)[0]
    if pulse > 0:
        c = 0.03 * pulse / 2.3548
        ph = float(torch.rand(1, generator=g, device="cuda"))
        d = torch.remainder(torch.arange(n, device="cuda", dtype=torch.float64) - ph * pulse, pulse)
        s = torch.exp(-0.5 * (torch.minimum(d, pulse - d) / c) ** 2)
        x += (s * (snr / float(s.square().sum().sqrt()))).float()
    return x


def _input(case, seed):
    x = _series(case["n"], seed, case["pulse"] / case["tsamp"])
    return (x * 16 + 128).round_().clamp_(0, 255).to(torch.uint8) if case["u8"] else x


def _codes(z):
    return (z * 16).round_().clamp_(-127, 127).to(torch.int8)


def _fold_input(case, seed):
    n = case["p0"] * case["m_data"]
    z = _series(n, seed, case["p0"] + 0.3)
    z = (z - z.mean()) / z.std()
    return _codes(z) if case["i8"] else z


def _plain_fold(z, p0, m_data, m_rows):
    """The FFA of the rows of z by its recursion, in z's type (or int32)."""
    a = torch.zeros((m_rows, p0), dtype=z.dtype, device=z.device)
    a[:m_data] = z[: m_data * p0].view(m_data, p0)
    col = torch.arange(p0, device=z.device)
    s = 1
    while s < m_rows:
        a = a.view(-1, 2, s, p0)
        k = torch.arange(2 * s, device=z.device)
        idx = (col[None, :] + ((k + 1) // 2)[:, None]) % p0
        out = torch.empty((a.shape[0], 2 * s, p0), dtype=a.dtype, device=a.device)
        per = max(1, (1 << 26) // (2 * s * p0))
        for i in range(0, a.shape[0], per):
            b = a[i:i + per]
            tail = b[:, 1].repeat_interleave(2, dim=1)
            out[i:i + per] = b[:, 0].repeat_interleave(2, dim=1) + tail.gather(2, idx.expand(b.shape[0], -1, -1))
        a = out
        s *= 2
    return a.view(m_rows, p0)


def _rows(m):
    r = 1
    while r < m:
        r *= 2
    return r


def _widths(p0, duty):
    w = [1]
    while w[-1] <= duty * p0 and len(w) < 16:
        w.append(2 * w[-1])
    return w


def _profiles(case, seed):
    """The profiles a fold leaves: all trials of a base period (`count` of them)."""
    p0, count = case["p0"], case["count"]
    m = min(count, 2048)
    z = _series(p0 * m, seed, p0 + 0.3)
    z = (z - z.mean()) / z.std()
    z = _codes(z).to(torch.int32) if case["i32"] else z
    a = _plain_fold(z, p0, m, _rows(m))
    # more trials than the fold has rows: the later ones at other phases
    parts = [a.roll(37 * i, 1) for i in range(-(-count // a.shape[0]))]
    return torch.cat(parts)[:count].contiguous()


def _config(case):
    duty = case["duty"]
    return ffa.Config(tsamp=case["tsamp"], period_min=case["pmin"], period_max=case["pmax"],
                      duty=duty if duty > 0 else 0.2, downsample0=case["d0"],
                      in_type=ffa.IN_U8 if case["u8"] else ffa.IN_F32,
                      precision=ffa.FOLD_I8 if case["i8"] else ffa.FOLD_F32,
                      widths=() if duty > 0 else (1, 2, 4, 8, 16), clip_sigma=case["clip"])


def _batch(case, seed):
    """Lengths of the batch's series (from the sizes alone: a plan is made for a length)."""
    n, lo, hi = case["series"], case["lo"], case["hi"]
    return [lo + (hi - lo) * i // max(1, n - 1) + (7 * i) % 13 for i in range(n)]


def _batch_config(case):
    return ffa.Config(tsamp=BATCH_TSAMP, period_min=0.5, period_max=20.0, duty=0.2,
                      precision=ffa.FOLD_I8 if case["i8"] else ffa.FOLD_F32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        x = _input(case, seed)
        plan = ffa.Plan(_config(case), case["n"])
        return dict(kind=kind, x=x, plan=plan, ws=plan.workspace(), rec=plan.records(), status=ffa.status_word(),
                    top_k=case["top_k"])
    if kind == "batch":
        ns = _batch(case, seed)
        xs = [_series(n, seed * 1009 + i, 3.1 / BATCH_TSAMP if i % 4 == 0 else 0.0) for i, n in enumerate(ns)]
        plans = [ffa.Plan(_batch_config(case), n) for n in ns]
        ws = torch.empty(ffa.batch_workspace_bytes(plans), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, xs=xs, plans=plans, ws=ws, recs=[p.records() for p in plans], status=ffa.status_word())
    if kind == "fold":
        return dict(kind=kind, z=_fold_input(case, seed), p0=case["p0"], m_data=case["m_data"],
                    m_rows=_rows(case["m_data"]))
    if kind == "score":
        return dict(kind=kind, prof=_profiles(case, seed), widths=_widths(case["p0"], 0.2), alg=case["alg"],
                    status=ffa.status_word())
    return dict(kind=kind, x=_series(case["n"], seed).double(), window=case["window"], status=ffa.status_word(),
                precision=ffa.FOLD_I8 if case["i8"] else ffa.FOLD_F32)


# ---- the calls ----------------------------------------------------------------

def _records(rec, n):
    """A record's fields: the S/N, and the width, phase and flags."""
    return dict(snr=rec[:n, 0].view(torch.float32), best=rec[:n, 1:])


def run(state):
    kind = state["kind"]
    if kind == "search":
        plan = state["plan"]
        rec = ffa.search(plan, state["x"], state["ws"], state["rec"], state["status"])
        out = _records(rec, plan.n_trials)
        if state["top_k"]:
            cands, best = ffa.candidates(plan, rec, state["ws"], snr_min=3.0, top_k=state["top_k"],
                                         status=state["status"])
            out.update(top=cands["trial"], top_snr=cands["snr"], top_period=cands["period_s"], best_trial=best)
        return out
    if kind == "batch":
        recs = ffa.search_batch(state["plans"], state["xs"], state["ws"], state["recs"], state["status"])
        return [_records(r, p.n_trials) for r, p in zip(recs, state["plans"])]
    if kind == "fold":
        return ffa.fold(state["z"], state["p0"], state["m_data"], state["m_rows"])
    if kind == "score":
        prof = state["prof"]
        if state["alg"] == 2:
            rec = ffa.score_alg2(prof, state["widths"])
        else:
            rec = ffa.score(prof, state["widths"], status=state["status"])
        return _records(rec, prof.shape[0])
    resid = ffa.detrend(state["x"], state["window"], status=state["status"])
    z, stats = ffa.normalise(resid, state["precision"])
    return dict(resid=resid, z=z, stats=stats[:2])


# ---- what a pass cannot do without -------------------------------------------------

def _search_work(plan, in_bytes, i8):
    e = plan.entries
    m, md, p0 = (e[k].astype(np.float64) for k in ("m_rows", "m_data", "p0"))
    octs = {int(o): int(n) for o, n in zip(e["octave"], e["n_octave"])}
    flops = float((m * p0 * (np.log2(m) + 3 + 2 * e["n_widths"])).sum())
    flops += sum(12.0 * n for n in octs.values())  # downsample, median, normalise
    # the input once and the records once: every fold is of that same series
    return dict(bytes=float(in_bytes + 16 * m.sum()), flops=flops)


def work(case):
    kind = case["kind"]
    if kind == "search":
        return _search_work(ffa.Plan(_config(case), case["n"]), case["n"] * (1 if case["u8"] else 4), case["i8"])
    if kind == "batch":
        ws = [_search_work(ffa.Plan(_batch_config(case), n), 4 * n, case["i8"]) for n in _batch(case, 0)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "fold":
        p0, md, m = case["p0"], case["m_data"], _rows(case["m_data"])
        return dict(bytes=float((1 if case["i8"] else 4) * p0 * md + 4 * p0 * m), flops=float(p0 * m * math.log2(m)))
    if kind == "score":
        bins = case["p0"] * case["count"]
        return dict(bytes=float(4 * bins + 16 * case["count"]), flops=float(bins * (3 + 2 * len(_widths(case["p0"], 0.2)))))
    n = case["n"]
    return dict(bytes=float(8 * n + 8 * n + (1 if case["i8"] else 4) * n), flops=12.0 * n)


# ---- the same in 64 bits -------------------------------------------------------------

def _exact_score1(prof, widths):
    """Algorithm 1's S/N of each row."""
    p0 = prof.shape[1]
    out = []
    per = max(1, (1 << 25) // p0)
    for i in range(0, prof.shape[0], per):
        x = prof[i:i + per].double()

        def mid(a):
            a = a.sort(dim=1).values
            return (a[:, (p0 - 1) // 2] + a[:, p0 // 2]) / 2

        med = mid(x)
        mad = mid((x - med[:, None]).abs())
        ext = torch.cat([x, x.repeat(1, -(-widths[-1] // p0))[:, : widths[-1]]], dim=1)
        c = torch.cat([torch.zeros_like(x[:, :1]), ext.cumsum(1)], dim=1)
        best = torch.full_like(med, -math.inf)
        for w in widths:
            b = (c[:, w:w + p0] - c[:, :p0]).amax(1)
            best = torch.maximum(best, (b - w * med) / (1.4826 * mad * math.sqrt(w)))
        out.append(torch.where(mad > 0, best, torch.zeros_like(best)))
    return torch.cat(out)


def _exact_score2(prof, widths, frac=0.2):
    """Algorithm 2's S/N of each row (statistics outside the window around each width's best box)."""
    p0 = prof.shape[1]
    h = int(math.floor(np.float32(frac) * np.float32(p0) / np.float32(2)))
    n_off = p0 - min(p0, 2 * h + 1)
    out = []
    per = max(1, (1 << 25) // p0)
    for i in range(0, prof.shape[0], per):
        x = prof[i:i + per].double()
        x = x - x.mean(1, keepdim=True)
        shift = prof[i:i + per].double().mean(1)
        cat = torch.cat([x, x, x], dim=1)
        zero = torch.zeros_like(x[:, :1])
        c1 = torch.cat([zero, cat.cumsum(1)], dim=1)
        c2 = torch.cat([zero, cat.square().cumsum(1)], dim=1)
        best = torch.full_like(shift, -math.inf)
        for w in widths:
            box, j = (c1[:, w:w + p0] - c1[:, :p0]).max(1)
            lo = (j + w // 2) % p0 + p0 - h

            def win(c):
                return (c.gather(1, (lo + 2 * h + 1)[:, None]) - c.gather(1, lo[:, None]))[:, 0]

            av = (c1[:, p0] - win(c1)) / n_off
            sd = ((c2[:, p0] - win(c2)) / n_off - av * av).clamp_min(0).sqrt()
            a = (box - w * av) / (sd * math.sqrt(w))
            best = torch.maximum(best, torch.where(sd > 0, a, best))
        out.append(torch.where(best > -math.inf, best, torch.zeros_like(best)))
    return torch.cat(out)


def _exact_median(x, w):
    """Centred running median of a short series, windows cut at the ends."""
    n, h = x.numel(), w // 2
    pad = torch.full((h,), math.inf, dtype=x.dtype, device=x.device)
    win = torch.cat([pad, x, pad]).unfold(0, 2 * h + 1, 1)
    out = torch.empty_like(x)
    per = max(1, (1 << 25) // (2 * h + 1))
    i = torch.arange(n, device=x.device)
    cnt = torch.clamp(i + h, max=n - 1) - torch.clamp(i - h, min=0) + 1
    for a in range(0, n, per):
        s = win[a:a + per].sort(dim=1).values  # values beyond the ends sort last
        c = cnt[a:a + per, None]
        out[a:a + per] = ((s.gather(1, (c - 1) // 2) + s.gather(1, c // 2)) / 2)[:, 0]
    return out


def _exact_search(case, seed):
    x = _input(case, seed).double()
    d0 = case["d0"]
    ts = case["tsamp"] * d0
    x = x[: x.numel() // d0 * d0].view(-1, d0).sum(1)
    p_min = max(1, math.ceil(case["pmin"] / ts - 1e-9))
    p_max = case["pmax"] / ts
    w = min(2 * math.ceil(p_max - 1e-9), 4 * p_min) | 1
    octs, n = [], x.numel()
    while True:
        hi = min(2 * p_min, math.ceil(p_max / 2 ** len(octs) - 1e-9))
        if hi <= p_min or n // p_min < 2:
            break
        octs.append((n, [p for p in range(p_min, hi) if n // p >= 2]))
        n //= 2
    bins = sum(_rows(n // p) * p * math.log2(_rows(n // p)) for n, ps in octs for p in ps)
    if sum(n for n, _ in octs) * w > 4e8 or sum(len(ps) for _, ps in octs) > 1500 or bins > 1e10:
        return None
    snr = []
    for n, ps in octs:
        x = x[:n]
        r = x - _exact_median(x, w)
        z = (r - r.mean()) / r.std(correction=0)
        if case["clip"] > 0:
            z = z.clamp(-case["clip"], case["clip"])
        if case["i8"]:
            z = (z * 16).round().clamp(-127, 127)
        for p in ps:
            widths = _widths(p, case["duty"]) if case["duty"] > 0 else [1, 2, 4, 8, 16]
            snr.append(_exact_score1(_plain_fold(z, p, n // p, _rows(n // p)), widths))
        x = x[: n // 2 * 2].view(-1, 2).sum(1)
    out = dict(snr=torch.cat(snr), best=None)
    if case["top_k"]:
        out.update(top=None, top_snr=None, top_period=None, best_trial=None)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "search":
        return _exact_search(case, seed)
    if kind == "fold":
        z = _fold_input(case, seed)
        if case["i8"]:
            return None  # whole numbers
        return _plain_fold(z.double(), case["p0"], case["m_data"], _rows(case["m_data"]))
    if kind == "score":
        prof, widths = _profiles(case, seed), _widths(case["p0"], 0.2)
        return dict(snr=_exact_score2(prof, widths) if case["alg"] == 2 else _exact_score1(prof, widths), best=None)
    return None
