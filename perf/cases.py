"""The work that users of this library have it do, as measurable cases.

Each case is one pass through public entry points of the Python binding (which
issues the C calls of include/tre.h):

  pipeline  PipelinePlan on request records: reduce, calibrate, normalize, select
  events    PipelinePlan on token-level events
  sweep     SweepPlan: several traces x window lengths x rescue thresholds x pacing caps
  score     tss_score on window counts (with a carry: the newest windows of a live trace)
  occupancy tss_window_reduce with window-mean occupancy, then tss_score on the means
  classes   tss_class_models, then reduce, calibrate and normalize per (model, SLO class)
  stage     the stage-aware signal: reduce, split gauges, both boundaries, both scores
  rank      tss_rank: receiver and donor order of every window
  select    tre_select_moves on scored windows, replicas of unequal footprint
  replay    ReplayPlan: the closed loop for several (rescue threshold, pacing cap) settings

Inputs are made on the GPU from the seed, in the shapes of the library's own
workloads: Poisson arrivals per model (flat, or diurnal with a ten-fold burst),
log-normal token counts, Zipf or code/chat model mixes, first-come-first-served
service at 0.8 utilisation with exponential service times, int32 milliseconds.
The queue of a model with c servers is the single queue whose server is c times
as fast (a running maximum gives its start times), so that a ten-million-record
trace takes a fraction of a second. `exact` states every floating output in
64 bits with plain torch from the same inputs.
"""
import math
import random

import numpy as np
import torch

import paper_2609_29160_gb300 as tre

DEV = "cuda"
SLO_MS = (1000, 5000, 20000)          # interactive, best effort, batch
COLS = ("model", "t_arr_ms", "t_start_ms", "t_first_ms", "t_end_ms", "L_in", "L_out")
W_P, W_Q, TAU_CRIT, TAU_SURPLUS = 0.2, 2.0, 0.8, 1.2
OK_FRAC, RELIABILITY = 0.95, 0.95
TAUS = "0.5,0.6,0.7,0.75,0.8,0.85,0.9,0.95"
CAPS = "1,2,3,4,5,6,7,8"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a short window-by-window study of three models (the smallest whole pass)
        {"name": "pipeline_3x10k_f64", "kind": "pipeline", "dtype": "f64", "M": 3, "n": 10_000,
         "dur_s": 600, "win": 1000, "mix": "same", "waves": False},
        # one hour of eight models, diurnal load with a burst: the ordinary trace
        {"name": "pipeline_8x1M_f32", "kind": "pipeline", "dtype": "f32", "M": 8, "n": 1_000_000,
         "dur_s": 3600, "win": 1000, "mix": "same", "waves": True},
        # six hours of sixteen code-like and chat-like models, half-second windows
        {"name": "pipeline_16x10M_f32", "kind": "pipeline", "dtype": "f32", "M": 16,
         "n": 10_000_000, "dur_s": 21600, "win": 500, "mix": "code_chat", "waves": True},
        # a day of 64 models as one event per token, 100 ms windows: the largest
        {"name": "events_64x200M_f32", "kind": "events", "dtype": "f32", "M": 64, "n": 230_000,
         "dur_s": 86400, "win": 100, "mix": "same", "waves": False},
        # the open-loop study: seven traces under every window length, threshold and cap
        {"name": "sweep_7x1M_f32", "kind": "sweep", "dtype": "f32", "M": 8, "n": 1_000_000,
         "dur_s": 3600, "wins": "100,500,1000,2000", "taus": TAUS, "caps": CAPS, "traces": 7,
         "mix": "same", "waves": True},
        # a controller scoring the newest minute of a live trace, state carried along
        {"name": "score_8x60_carry_f64", "kind": "score", "dtype": "f64", "M": 8, "K": 60,
         "win": 1000, "carry": True},
        # window-mean occupancy of an hour at 100 ms, then the score that uses it
        {"name": "occupancy_8x1M_f32", "kind": "occupancy", "dtype": "f32", "M": 8,
         "n": 1_000_000, "dur_s": 3600, "win": 100, "mix": "same", "waves": True},
        # eight models with three SLO classes each, a record count of no round size
        {"name": "classes_8x3x999983_f64", "kind": "classes", "dtype": "f64", "M": 8,
         "classes": 3, "n": 999_983, "dur_s": 3600, "win": 1000, "mix": "same", "waves": True},
        # separate prefill and decode signals of an ordinary trace
        {"name": "stage_8x1M_f32", "kind": "stage", "dtype": "f32", "M": 8, "n": 1_000_000,
         "dur_s": 3600, "win": 1000, "mix": "same", "waves": True},
        # receiver and donor order of four million windows, for reports
        {"name": "rank_8x4M_f32", "kind": "rank", "dtype": "f32", "M": 8, "K": 4_000_000,
         "win": 100},
        # one controller run over an hour of scored windows, replicas of one, two or four units
        {"name": "select_24x36000_f32", "kind": "select", "dtype": "f32", "M": 24, "K": 36_000,
         "win": 100, "cap": 2},
        # ten minutes replayed in closed loop under 64 settings, wake and sleep delays, guards
        {"name": "replay_8x160k_64_f32", "kind": "replay", "dtype": "f32", "M": 8, "n": 160_000,
         "dur_s": 600, "win": 1000, "taus": TAUS, "caps": CAPS, "mix": "same", "waves": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; the record counts, model counts and
    durations are spread over their logarithm, mostly odd."""
    kind = rng.choice(("pipeline", "pipeline", "pipeline", "events", "sweep", "score",
                       "occupancy", "classes", "stage", "rank", "select", "replay"))
    c = {"kind": kind, "dtype": rng.choice(("f32", "f32", "f64"))}
    if kind == "score":
        c.update(M=_log(rng, 1, 64), K=_log(rng, 8, 200_000), win=rng.choice((100, 500, 1000)),
                 carry=rng.random() < 0.5)
        return c
    if kind == "rank":
        c.update(M=_log(rng, 2, 64), K=_log(rng, 1_000, 2_000_000), win=100)
        return c
    if kind == "select":
        c.update(M=_log(rng, 2, 64), K=_log(rng, 1_000, 200_000), win=rng.choice((100, 500, 1000)),
                 cap=rng.randint(1, 8))
        return c
    c.update(M=_log(rng, 2, 64), win=rng.choice((100, 200, 250, 500, 1000, 2000)),
             mix=rng.choice(("same", "code_chat")), waves=rng.random() < 0.5)
    if kind in ("pipeline", "occupancy", "stage"):
        c.update(n=_log(rng, 5_000, 5_000_000), dur_s=_log(rng, 300, 21_600) // 2 * 2)
    elif kind == "classes":
        c.update(M=_log(rng, 2, 32), classes=rng.choice((2, 3, 5)), n=_log(rng, 5_000, 2_000_000),
                 dur_s=_log(rng, 300, 21_600) // 2 * 2)
    elif kind == "events":
        c.update(n=_log(rng, 2_000, 60_000), dur_s=_log(rng, 600, 43_200) // 2 * 2)
    elif kind == "sweep":
        base = rng.choice((100, 200, 250))
        del c["win"]
        wins = [base] + sorted(rng.sample([base * q for q in (2, 4, 5, 10, 20)],
                                          rng.randint(1, 3)))
        c.update(M=_log(rng, 2, 16), n=_log(rng, 20_000, 700_000), traces=rng.randint(1, 7),
                 dur_s=_log(rng, 300, 3600) // 60 * 60 or 60, wins=",".join(map(str, wins)),
                 taus=",".join(TAUS.split(",")[: rng.randint(1, 8)]),
                 caps=",".join(CAPS.split(",")[: rng.randint(1, 8)]))
    else:
        c.update(M=_log(rng, 2, 16), n=_log(rng, 5_000, 160_000), dur_s=_log(rng, 120, 600),
                 win=rng.choice((500, 1000)), taus=",".join(TAUS.split(",")[: rng.randint(1, 8)]),
                 caps=",".join(CAPS.split(",")[: rng.randint(1, 8)]))
        c["dur_s"] = c["dur_s"] // 2 * 2
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _floats(text):
    return [float(x) for x in text.split(",")]


def _ints(text):
    return [int(x) for x in text.split(",")]


def _split(weights, total):
    """Whole parts of `total` in proportion to the weights, each at least one."""
    w = np.asarray(weights, np.float64)
    part = np.maximum(1, np.floor(w / w.sum() * total).astype(np.int64))
    while part.sum() > total:
        part[int(np.argmax(part))] -= 1
    while part.sum() < total:
        part[int(np.argmax(w / w.sum() * total - part))] += 1
    return part


def _load(case, seed):
    """Per-model rates over the trace, lengths, service scale, budget, replicas."""
    M, T = case["M"], case["dur_s"]
    i = np.arange(M)
    share = 1.0 / (i % 8 + 1.0) if case["mix"] == "code_chat" else 1.0 / (i + 1.0)
    cost = 20.0 ** (i / max(M - 1, 1))
    if case["mix"] == "code_chat":
        li = [(8.0, 1.0) if m < (M + 1) // 2 else (5.0, 1.0) for m in range(M)]
        lo = [(4.0, 1.0) if m < (M + 1) // 2 else (6.0, 0.8) for m in range(M)]
    else:
        li, lo = [(6.0, 1.0)] * M, [(5.0, 0.8)] * M
    work = np.array([0.2 * math.exp(a + b * b / 2) + math.exp(x + y * y / 2)
                     for (a, b), (x, y) in zip(li, lo)])
    t = np.arange(T) + 0.5
    rate = np.repeat(share[:, None], T, 1)
    if case["waves"]:
        rate = rate * (1.0 + 0.5 * np.sin(2 * np.pi * t / T + 2 * np.pi * i[:, None] / M))
        rng = random.Random(int(seed))
        b, b0 = rng.randrange(M), rng.uniform(T / 6, 3 * T / 4)
        rate[b] = np.where((t >= b0) & (t < b0 + T / 12), rate[b] * 10, rate[b])
    budget = 8 * M
    r0 = _split(share * cost * work, budget)
    lam = case["n"] * share / rate.sum()                    # requests per second
    u = 0.8 * budget / float((lam * cost * work).sum())     # seconds per unit of work
    counts = _split(rate.sum(1), case["n"])
    return rate, li, lo, u * cost * work, budget, r0, counts


def _requests(case, seed, latent=False):
    """Records sorted by arrival (or latent requests), the budget and replicas."""
    g = _gen(seed)
    rate, li, lo, svc_mean, budget, r0, counts = _load(case, seed)
    span_us = case["dur_s"] * 1_000_000
    rows = []
    for m in range(case["M"]):
        n = int(counts[m])
        cum = torch.as_tensor(np.concatenate(([0.0], np.cumsum(rate[m]) / rate[m].sum())),
                              device=DEV)
        x = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        k = torch.searchsorted(cum, x, right=True).sub_(1).clamp_(0, case["dur_s"] - 1)
        frac = (x - cum[k]) / (cum[k + 1] - cum[k]).clamp_min(1e-300)
        arr = ((k + frac) * 1e6).long().clamp_(0, span_us - 1).sort().values
        L = [torch.empty(n, device=DEV).log_normal_(*p, generator=g).round_().clamp_(1, 131072)
             for p in (li[m], lo[m])]
        svc = (torch.empty(n, device=DEV, dtype=torch.float64).exponential_(1.0, generator=g) *
               (svc_mean[m] * 1e6)).long()
        pre = 0.2 * L[0].double()
        d_first = (svc * (pre / (pre + L[1].double()))).long()
        one = L[1] == 1
        if latent:
            total = torch.where(one, d_first // 1000, svc // 1000)
            rows.append((arr, [torch.full_like(arr, m), arr // 1000, d_first // 1000, total, *L]))
            continue
        fast = svc // int(r0[m])                            # the queue's own service
        before = torch.cumsum(fast, 0) - fast
        start = before + torch.cummax(arr - before, 0).values
        first, end = (start + d_first) // 1000, (start + svc) // 1000
        rows.append((arr, [torch.full_like(arr, m), arr // 1000, start // 1000, first,
                           torch.where(one, first, end), *L]))
    order = torch.cat([a for a, _ in rows]).sort(stable=True).indices
    keys = tre.LATENT_KEYS if latent else COLS
    out = {}
    for j, k in enumerate(keys):
        v = torch.cat([r[j].long() for _, r in rows])[order]
        out[k] = v.clamp_(max=2_000_000_000).int().contiguous()
    return out, budget, r0


def _events(case, seed):
    """One event per prompt token (uniform over [start, first token]) and per
    output token (normalised exponential gaps from first to last token, that is
    sorted uniforms), sorted by time, with the per-request table."""
    rec, budget, r0 = _requests(case, seed)
    g = _gen(seed + 7919)
    n = rec["model"].numel()
    rid = torch.arange(n, device=DEV)
    t = {k: rec[k].double() / 1000 for k in ("t_start_ms", "t_first_ms", "t_end_ms")}
    req, time, phase = [], [], []
    for ph, (length, a, b) in enumerate((("L_in", "t_start_ms", "t_first_ms"),
                                         ("L_out", "t_first_ms", "t_end_ms"))):
        r = torch.repeat_interleave(rid, rec[length].long())
        u = torch.rand(r.numel(), generator=g, device=DEV)
        if ph:
            stop = torch.cumsum(rec[length].long(), 0)
            u[stop - 1] = 1.0                               # the last token, then the first
            u[stop - rec[length].long()] = 0.0
        time.append((t[a][r] + u * (t[b] - t[a])[r]).float())
        req.append(r.int())
        phase.append(torch.full((r.numel(),), ph, dtype=torch.uint8, device=DEV))
    time, req, phase = torch.cat(time), torch.cat(req), torch.cat(phase)
    time, order = time.sort(stable=True)
    req, phase = req[order].contiguous(), phase[order].contiguous()
    del order
    ev = {"model": rec["model"][req.long()].contiguous(), "req": req, "t_s": time,
          "phase": phase, "req_model": rec["model"], "req_t_arr_ms": rec["t_arr_ms"],
          "req_ttft_ms": (rec["t_first_ms"] - rec["t_arr_ms"]).contiguous()}
    return ev, budget, r0


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _alpha(win):
    return min(1.0, win / 5000.0)


def _profile(M, win, tdt, theta=None):
    v = {"w_p": W_P, "w_q": W_Q, "alpha": _alpha(win), "tau_crit": TAU_CRIT,
         "tau_surplus": TAU_SURPLUS}
    prof = {k: torch.full((M,), x, dtype=tdt, device=DEV) for k, x in v.items()}
    prof["theta"] = torch.ones(M, dtype=tdt, device=DEV) if theta is None else theta
    return prof


def _slo(M):
    return np.array([SLO_MS[m % 3] for m in range(M)], np.int32)


def _K(case):
    return case["dur_s"] * 1000 // case["win"]


def _window_counts(case, seed):
    """Counts of a live trace's windows: quiet and busy models, a tenth idle."""
    g = _gen(seed)
    K, M = case["K"], case["M"]
    busy = 1.0 / (torch.arange(M, device=DEV) + 1.0)
    idle = torch.rand((K, M), generator=g, device=DEV) < 0.1
    draw_ = lambda mean: torch.poisson((busy * mean).expand(K, M).contiguous(), generator=g)
    scale = case["win"] / 1000.0
    out = {}
    for k, mean in (("P", 40000 * scale), ("D", 15000 * scale), ("A", 24.0), ("W", 3.0)):
        out[k] = torch.where(idle, torch.zeros((), device=DEV), draw_(mean)).int().contiguous()
    return out


def prepare(case, seed):
    kind, M, tdt = case["kind"], case["M"], _dtype(case)
    st = {"kind": kind, "case": dict(case)}
    ones = np.ones(M, np.int32)
    if kind in ("pipeline", "events"):
        ev, rec = None, None
        if kind == "events":
            ev, budget, r0 = _events(case, seed)
        else:
            rec, budget, r0 = _requests(case, seed)
        st["plan"] = tre.PipelinePlan(M, case["win"], _K(case), _profile(M, case["win"], tdt),
                                      _slo(M), budget, r0, ones, ones, requests=rec, events=ev,
                                      dtype=case["dtype"])
    elif kind == "sweep":
        traces, wins = [], _ints(case["wins"])
        for i in range(case["traces"]):
            rec, budget, r = _requests(case, seed * 1000 + i)
            traces.append(rec)
        st["plan"] = tre.SweepPlan(traces, M, case["dur_s"] * 1000, wins,
                                   [_alpha(w) for w in wins], _floats(case["taus"]),
                                   _ints(case["caps"]), W_P, W_Q, TAU_SURPLUS, _slo(M), budget, r,
                                   ones, ones, dtype=case["dtype"])
    elif kind == "score":
        st["counts"] = _window_counts(case, seed)
        st["prof"] = _profile(M, case["win"], tdt, _score_theta(case, tdt))
        st["carry"] = None
        if case["carry"]:
            x = torch.rand(M, generator=_gen(seed + 1), device=DEV, dtype=torch.float64) + 0.5
            st["carry"] = {"S": (x * 800).to(tdt),
                           "init": torch.ones(M, dtype=torch.uint8, device=DEV)}
    elif kind in ("occupancy", "stage"):
        st["rec"], _, _ = _requests(case, seed)
        st["prof"] = _profile(M, case["win"], tdt, torch.full((M,), 300.0, dtype=tdt, device=DEV))
        st["slo"] = torch.as_tensor(_slo(M)).to(DEV)
        st["tpot"] = torch.full((M,), 50, dtype=torch.int32, device=DEV)
    elif kind == "classes":
        st["rec"], _, _ = _requests(case, seed)
        pairs = M * case["classes"]
        st["cls"] = torch.randint(0, case["classes"], (case["n"],), generator=_gen(seed + 1),
                                  device=DEV, dtype=torch.int32)
        st["prof"] = _profile(pairs, case["win"], tdt)
        st["slo"] = torch.as_tensor(_slo(pairs)).to(DEV)
    elif kind in ("rank", "select"):
        st["Z"], st["cls"] = _ranked(case, seed)
        fp = np.array([1, 2, 4], np.int32)[np.arange(M) % 3]
        st["fp"], st["r"] = (torch.as_tensor(v).to(DEV) for v in (fp, 4 * ones))
        st["r_min"], st["budget"] = torch.as_tensor(ones).to(DEV), int(4 * fp.sum() + M)
        st["prof"] = _profile(M, case["win"], tdt)
        st["moves"] = np.zeros(4096 * tre.MOVE_DTYPE.itemsize, np.uint8)
    else:
        lat, budget, r0 = _requests(case, seed, latent=True)
        prof = _profile(M, case["win"], tdt)
        rate, _, _, svc, _, _, _ = _load(case, seed)
        # tokens a server emits per second of service, scaled to a boundary below it
        prof["theta"] = torch.as_tensor(0.5 * 300.0 / svc).to(device=DEV, dtype=tdt)
        st["plan"] = tre.ReplayPlan(lat, M, case["win"], _K(case), prof, budget, r0, ones, ones,
                                    tau_list=_floats(case["taus"]), cap_list=_ints(case["caps"]),
                                    wake_ms=1310, sleep_ms=1870, slo_ttft_ms=_slo(M),
                                    guard_ttft_ms=2 * _slo(M), dtype=case["dtype"])
    return st


def _score_theta(case, tdt):
    return torch.full((case["M"],), 700.0, dtype=tdt, device=DEV)


def _ranked(case, seed):
    """Scored windows: Z around 1, a tenth of the cells idle."""
    g = _gen(seed)
    K, M = case["K"], case["M"]
    Z = torch.empty((K, M), device=DEV, dtype=_dtype(case)).log_normal_(0.0, 0.3, generator=g)
    cls = torch.where(Z < TAU_CRIT, tre.CRIT, torch.where(Z > TAU_SURPLUS, tre.SURP, tre.NOM))
    idle = torch.rand((K, M), generator=g, device=DEV) < 0.1
    return Z, torch.where(idle, tre.IDLE, cls).to(torch.uint8)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    case, kind = st["case"], st["kind"]
    M, dt = case["M"], case["dtype"]
    if kind in ("pipeline", "events"):
        p = st["plan"].run()
        return {**p.counts, "theta": p.theta, "S": p.S, "Z": p.Z, "cls": p.cls, "recv": p.recv,
                "moves": p.moves, "n_moves": p.n_moves, "r_final": p.r}
    if kind == "sweep":
        out = st["plan"].run()
        return {k: out[k] for k in ("theta", "Z", "cls", "moves", "n_moves", "r_final")}
    if kind == "score":
        out = tre.tss_score(st["counts"], st["prof"], case["win"], dtype=dt, carry=st["carry"])
        return {**out, "carry": st["carry"]["S"]} if st["carry"] else out
    if kind == "occupancy":
        c = tre.tss_window_reduce(M, case["win"], _K(case), requests=st["rec"],
                                  mean_occupancy=True)
        return {**c, **tre.tss_score(c, st["prof"], case["win"], dtype=dt)}
    if kind == "classes":
        pairs, K, win = M * case["classes"], _K(case), case["win"]
        ids = tre.tss_class_models(st["rec"]["model"], st["cls"], M, case["classes"])
        rec = {**st["rec"], "model": ids}
        c = tre.tss_window_reduce(pairs, win, K, requests=rec)
        S = torch.empty((K, pairs), dtype=_dtype(case), device=DEV)
        idle = torch.empty((K, pairs), dtype=torch.uint8, device=DEV)
        theta = tre.tss_calibrate(c, st["prof"], win, st["slo"], requests=rec, dtype=dt, S_out=S,
                                  cls_out=idle)
        z = tre.tss_normalize(S, idle, {**st["prof"], "theta": theta}, win)
        return {**c, "S": S, "theta": theta, **z}
    if kind == "stage":
        K, win = _K(case), case["win"]
        c = tre.tss_window_reduce(M, win, K, requests=st["rec"])
        Ap, Ad = tre.tss_stage_gauges(M, win, K, st["rec"])
        th = tre.tss_stage_calibrate(c, Ap, Ad, st["prof"], win, st["slo"], st["tpot"], st["rec"],
                                     dtype=dt)
        pre, dec = tre.tss_stage_score(c, Ap, Ad, st["prof"], win, th[0], th[1], dtype=dt)
        return {**c, "A_prefill": Ap, "A_decode": Ad, "theta": list(th), "prefill": pre,
                "decode": dec}
    if kind == "rank":
        return tre.tss_rank(st["Z"], st["cls"], case["win"])
    if kind == "select":
        moves, r, n, _ = tre.tre_select_moves(st["Z"], st["cls"], st["prof"], case["win"],
                                              st["budget"], st["r"], st["r_min"], st["fp"],
                                              pacing_cap=case["cap"])
        rows, used = st["moves"], moves.size * tre.MOVE_DTYPE.itemsize
        rows[:used], rows[used:] = moves.view(np.uint8), 0
        return {"moves": rows, "r": r, "n": n}
    return st["plan"].run()


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Every input read once and every output written once."""
    kind, M, sz = case["kind"], case["M"], 8 if case["dtype"] == "f64" else 4
    scored = 2 * sz + 1
    if kind == "score":
        cells, per = case["K"] * M, 16 + scored
        return {"bytes": cells * per + 4 * case["K"], "flops": 10 * cells}
    if kind == "rank":
        cells = case["K"] * M
        return {"bytes": cells * (sz + 1) + 36 * case["K"], "flops": 10 * cells}
    if kind == "select":
        # the controller reads the windows at its fast ticks (5 s)
        cells = case["K"] * M * case["win"] // 5000
        return {"bytes": max(cells, M) * (sz + 1) + 12 * M, "flops": 10 * max(cells, M)}
    if kind == "sweep":
        cells = sum(case["dur_s"] * 1000 // w for w in _ints(case["wins"])) * M * case["traces"]
        inst = case["traces"] * len(_ints(case["wins"])) * len(_floats(case["taus"])) * \
            len(_ints(case["caps"]))
        return {"bytes": 28 * case["n"] * case["traces"] + cells * (sz + 1) + inst * (4 * M + 8),
                "flops": 10 * cells}
    if kind == "replay":
        inst = len(_floats(case["taus"])) * len(_ints(case["caps"]))
        cells = _K(case) * M * inst
        return {"bytes": 24 * case["n"] + inst * (20 * M + 8), "flops": 10 * cells}
    K, n = _K(case), case["n"]
    if kind == "events":
        # tokens per request: the means of the rounded log-normal lengths
        if case["mix"] == "same":
            per = math.exp(6.5) + math.exp(5.32)
        else:
            per = 0.5 * (math.exp(8.5) + math.exp(4.5) + math.exp(5.5) + math.exp(6.32))
        return {"bytes": 13 * n * per + 12 * n + K * M * (16 + scored) + 4 * K,
                "flops": 10 * K * M}
    cells = K * M
    if kind == "occupancy":
        return {"bytes": 28 * n + cells * (32 + scored) + 4 * K, "flops": 10 * cells}
    if kind == "classes":
        cells *= case["classes"]
        return {"bytes": 36 * n + cells * (16 + scored) + 4 * K, "flops": 10 * cells}
    if kind == "stage":
        return {"bytes": 28 * n + cells * (24 + 2 * scored), "flops": 20 * cells}
    return {"bytes": 28 * n + cells * (16 + scored) + 4 * K, "flops": 10 * cells}


def tolerance(case):
    """The library promises one correctly rounded operation per step in the
    order of the sequential definitions, reproducible bit for bit: another
    correct implementation returns the same bits."""
    return "exact"


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _hist(k, m, v, K, M):
    out = torch.zeros(K * M, dtype=torch.int64, device=DEV)
    out.index_add_(0, k * M + m, v)
    return out.view(K, M)


def _gauge(a, b, m, K, M):
    """Members of [a, b) at each window's last millisecond (window indices)."""
    one = torch.ones_like(m)
    d = _hist(a.clamp(max=K), m, one, K + 1, M) - _hist(b.clamp(max=K), m, one, K + 1, M)
    return torch.cumsum(d, 0)[:K]


def _counts64(rec, M, win, K):
    m, ta, ts, tf, te, Li, Lo = (rec[k].long() for k in COLS)
    in_ = tf < K * win
    P = _hist(tf[in_] // win, m[in_], Li[in_], K, M)
    D = torch.zeros((K, M), dtype=torch.int64, device=DEV)
    step = 1_000_000
    for i in range(0, m.numel(), step):
        s = slice(i, i + step)
        ok = in_[s]
        mm, f, e, L = m[s][ok], tf[s][ok], te[s][ok], Lo[s][ok]
        kf, ke = f // win, (e // win).clamp(max=K - 1)
        rep = ke - kf + 1
        i_ = torch.repeat_interleave(torch.arange(mm.numel(), device=DEV), rep)
        at = torch.arange(i_.numel(), device=DEV) - torch.repeat_interleave(
            torch.cumsum(rep, 0) - rep, rep)
        k = kf[i_] + at

        def before(T):
            f_, e_, L_ = f[i_], e[i_], L[i_]
            dur = (e_ - f_).clamp(min=1)
            mid = ((T - f_) * (L_ - 1) + dur - 1) // dur
            mid = torch.where(L_ == 1, torch.ones_like(mid), mid)
            return torch.where(T <= f_, 0, torch.where(T > e_, L_, mid))

        D += _hist(k, mm[i_], before((k + 1) * win) - before(k * win), K, M)
    A = _gauge(ts // win, te // win, m, K, M)
    W = _gauge(ta // win, ts // win, m, K, M)
    return P, D, A, W


def _mean_ms(a, b, m, win, K, M):
    """Milliseconds of [a, b) inside each window."""
    out = torch.zeros((K, M), dtype=torch.int64, device=DEV)
    b = b.clamp(max=K * win)
    ok = a < b
    a, b, m = a[ok], b[ok], m[ok]
    ka, kb = a // win, (b - 1) // win
    same = ka == kb
    out += _hist(ka, m, torch.where(same, b - a, (ka + 1) * win - a), K, M)
    out += _hist(kb, m, torch.where(same, torch.zeros_like(b), b - kb * win), K, M)
    far = kb > ka
    one = torch.ones_like(m[far])
    d = _hist(ka[far] + 1, m[far], one, K + 1, M) - _hist(kb[far], m[far], one, K + 1, M)
    return out + torch.cumsum(d, 0)[:K] * win


def _smooth64(raw, idle, alpha, S0=None):
    """S = alpha raw + (1 - alpha) S_prev through the non-idle windows, started
    at the first one (or at S0), as a doubling scan of affine maps."""
    started = torch.cumsum((~idle).to(torch.int32), 0) > 0
    first = started & (torch.cumsum(started.to(torch.int32), 0) == 1) if S0 is None else \
        torch.zeros_like(idle)
    a = torch.full_like(raw, 1.0 - alpha).masked_fill_(idle, 1.0).masked_fill_(first, 0.0)
    b = (alpha * raw).masked_fill_(idle, 0.0)
    b = torch.where(first, raw, b)
    if S0 is not None:
        b[0] = a[0] * S0 + b[0]
        a[0] = 0.0
    else:
        a[0] = 0.0
    d = 1
    while d < raw.shape[0]:
        b[d:] = a[d:] * b[:-d] + b[d:]
        a[d:] = a[d:] * a[:-d]
        d *= 2
    return b


def _raw64(P, D, A, W, win, w_p=W_P, w_q=W_Q):
    P, D, A, W = (x.double() for x in (P, D, A, W))
    dt = win / 1000.0
    return (w_p * (P / dt) + D / dt) / torch.clamp(A + w_q * W, min=1.0)


def _theta64(S, idle, n_arr, n_met):
    out = np.ones(S.shape[1])
    for m in range(S.shape[1]):
        cand = (n_arr[:, m] >= 1) & ~idle[:, m] & (S[:, m] > 0)
        s = S[:, m][cand]
        if s.numel() == 0:
            continue
        h = (n_met[:, m][cand].double() >= OK_FRAC * n_arr[:, m][cand].double()).long()
        s, o = s.sort(descending=True, stable=True)
        H = torch.cumsum(h[o], 0).double()
        C = torch.arange(1, s.numel() + 1, device=DEV).double()
        last = torch.ones_like(s, dtype=torch.bool)
        last[:-1] = s[1:] != s[:-1]
        good = last & (H >= RELIABILITY * C)
        out[m] = float(s[good][-1]) if bool(good.any()) else float(s[0])
    return torch.as_tensor(out, device=DEV)


def _slo_counts(rec, M, win, K, slo):
    m, k = rec["model"].long(), rec["t_arr_ms"].long() // win
    met = (rec["t_first_ms"] - rec["t_arr_ms"]).long() <= torch.as_tensor(slo, device=DEV)[m]
    return _hist(k, m, torch.ones_like(m), K, M), _hist(k, m, met.long(), K, M)


def _scored64(counts, n_arr, n_met, win):
    P, D, A, W = counts
    idle = (P == 0) & (D == 0) & (A == 0) & (W == 0)
    S = _smooth64(_raw64(P, D, A, W, win), idle, _alpha(win))
    theta = _theta64(S, idle, n_arr, n_met)
    return {"S": S, "theta": theta, "Z": S / theta}


def _np(d):
    return {k: _np(v) if isinstance(v, dict) else [x.cpu().numpy() for x in v]
            if isinstance(v, list) else v.cpu().numpy() for k, v in d.items()}


def exact(case, seed):
    kind, M = case["kind"], case["M"]
    if kind in ("rank", "select", "replay"):
        return None                       # whole numbers only
    if kind == "score":
        c = {k: v.long() for k, v in _window_counts(case, seed).items()}
        idle = (c["P"] == 0) & (c["D"] == 0) & (c["A"] == 0) & (c["W"] == 0)
        raw = _raw64(c["P"], c["D"], c["A"], c["W"], case["win"])
        S0 = None
        if case["carry"]:
            x = torch.rand(M, generator=_gen(seed + 1), device=DEV, dtype=torch.float64) + 0.5
            S0 = (x * 800).to(_dtype(case)).double()
        S = _smooth64(raw, idle, _alpha(case["win"]), S0)
        out = {"S": S, "Z": S / _score_theta(case, torch.float64)}
        if case["carry"]:
            out["carry"] = S[-1]
        return _np(out)
    if kind == "sweep":
        wins, parts, thetas = _ints(case["wins"]), [], []
        for i in range(case["traces"]):
            rec, _, _ = _requests(case, seed * 1000 + i)
            for w in wins:
                K = case["dur_s"] * 1000 // w
                o = _scored64(_counts64(rec, M, w, K), *_slo_counts(rec, M, w, K, _slo(M)), w)
                parts.append(o["Z"].reshape(-1))
                thetas.append(o["theta"])
        return _np({"theta": torch.stack(thetas), "Z": torch.cat(parts)})
    win, K = case["win"], _K(case)
    if kind == "events":
        ev, _, _ = _events(case, seed)
        # milliseconds: the exact product of a float and 1000, rounded down
        tick = (ev["t_s"].double() * 1000.0).floor().long()
        ok = tick < K * win
        m, rq, k, t = ev["model"][ok].long(), ev["req"][ok].long(), tick[ok] // win, tick[ok]
        del tick
        pre = (ev["phase"][ok] == 0).long()
        P = _hist(k, m, pre, K, M)
        D = _hist(k, m, 1 - pre, K, M)
        n = ev["req_model"].numel()
        first = torch.full((n,), 1 << 40, dtype=torch.int64, device=DEV)
        first.scatter_reduce_(0, rq, t, "amin")
        last = torch.full((n,), -1, dtype=torch.int64, device=DEV)
        last.scatter_reduce_(0, rq, t, "amax")
        del m, rq, k, t, pre, ok
        rm, ta = ev["req_model"].long(), ev["req_t_arr_ms"].long()
        seen = (last >= 0) & (ta <= first)
        A = _gauge(first[seen] // win, last[seen] // win, rm[seen], K, M)
        W = _gauge(ta[seen] // win, first[seen] // win, rm[seen], K, M)
        met = ev["req_ttft_ms"].long() <= torch.as_tensor(_slo(M), device=DEV)[rm]
        n_arr = _hist(ta // win, rm, torch.ones_like(rm), K, M)
        n_met = _hist(ta // win, rm, met.long(), K, M)
        return _np(_scored64((P, D, A, W), n_arr, n_met, win))
    rec, _, _ = _requests(case, seed)
    if kind == "classes":
        cls = torch.randint(0, case["classes"], (case["n"],), generator=_gen(seed + 1),
                            device=DEV, dtype=torch.int32)
        rec["model"] = rec["model"] * case["classes"] + cls
        M *= case["classes"]
    P, D, A, W = _counts64(rec, M, win, K)
    if kind == "occupancy":
        m, ta, ts, te = (rec[k].long() for k in ("model", "t_arr_ms", "t_start_ms", "t_end_ms"))
        Am, Wm = _mean_ms(ts, te, m, win, K, M), _mean_ms(ta, ts, m, win, K, M)
        idle = (P == 0) & (D == 0) & (Am == 0) & (Wm == 0)
        S = _smooth64(_raw64(P, D, Am.double() / win, Wm.double() / win, win), idle, _alpha(win))
        return _np({"S": S, "Z": S / 300.0})
    if kind == "stage":
        m, ts, tf, te = (rec[k].long() for k in ("model", "t_start_ms", "t_first_ms", "t_end_ms"))
        Ap = _gauge(ts // win, tf // win, m, K, M)
        Ad = _gauge(tf // win, te // win, m, K, M)
        out, th = {}, []
        for name, n_, a, w, met in (("prefill", P, Ap, W, None), ("decode", D, Ad, W * 0, 50)):
            idle = (n_ == 0) & (a == 0) & (w == 0)
            S = _smooth64(_raw64(n_, D * 0, a, w, win, w_p=1.0), idle, _alpha(win))
            if met is None:
                n_arr, n_met = _slo_counts(rec, M, win, K, _slo(M))
            else:
                two = rec["L_out"] > 1
                k = rec["t_arr_ms"].long()[two] // win
                fine = (te - tf)[two] <= met * (rec["L_out"].long()[two] - 1)
                n_arr = _hist(k, m[two], torch.ones_like(k), K, M)
                n_met = _hist(k, m[two], fine.long(), K, M)
            th.append(_theta64(S, idle, n_arr, n_met))
            out[name] = {"S": S, "Z": S / th[-1]}
        return _np({**out, "theta": th})
    n_arr, n_met = _slo_counts(rec, M, win, K, _slo(M))
    return _np(_scored64((P, D, A, W), n_arr, n_met, win))
