"""GPU parity of move selection (Sec. IV-B rescue / rebalance, Eq. 3, Sec. IV-C
bounded transfer) on every walk variant of the library, against the oracle's
walk, bit for bit: the lane walk (nested cadences, up to 64 models) at the
edges of its tick chunks and staged slabs, the warp walk beyond 64 models, the
walks that visit every tick (cadences that are not nested, or a fast tick
shorter than a window), and pacing caps above 32 on few models."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

LEVELS = np.array([0.3, 0.5, 0.6, 0.8, 0.8, 0.85, 0.95, 1.0, 1.0, 1.1, 1.2, 1.3, 2.0])


@pytest.fixture(scope="module")
def tre():
    import torch
    import paper_2609_29160_gb300 as lib
    lib.load()
    torch.cuda.set_device(0)
    return lib


def _np(t):
    return t.detach().cpu().numpy()


def _case(seed, K, M, idle=0.1, hetero=False, dtype=np.float32):
    rng = np.random.default_rng(seed)
    Z = rng.choice(LEVELS, (K, M)).astype(dtype)            # many exact ties
    # a few models sit low for long stretches, so rescues repeat on them
    for m in rng.choice(M, max(1, M // 8), replace=False):
        a = int(rng.integers(0, K))
        Z[a: a + K // 5, m] = dtype(0.4)
    cls = np.where(rng.random((K, M)) < idle, oracle.IDLE, oracle.NOM).astype(np.uint8)
    g = rng.integers(1, 4, M).astype(np.int32) if hetero else np.ones(M, np.int32)
    r0 = rng.integers(1, 6, M).astype(np.int32)
    budget = int((g * r0).sum()) + int(rng.integers(0, 4))
    r_min = (rng.random(M) < 0.5).astype(np.int32)
    return Z, cls, g, r0, budget, r_min


def _check(tre, Z, cls, g, r0, budget, r_min, win, cap, fast_ms=5000, slow_ms=10000):
    import torch
    prof = {"w_p": 0.2, "w_q": 2.0, "alpha": 0.2, "theta": 1.0, "tau_crit": 0.8,
            "tau_surplus": 1.2}
    om, orf, _ = oracle.select_moves(Z, cls, 0.8, 1.2, win, budget, r0, r_min, g, fast_ms,
                                     slow_ms, cap)
    Zc, Cc = torch.as_tensor(Z).cuda(), torch.as_tensor(cls).cuda()
    mv, rf, n, diag = tre.tre_select_moves(Zc, Cc, prof, win, budget, r0, r_min, g,
                                           fast_ms=fast_ms, slow_ms=slow_ms, pacing_cap=cap,
                                           moves_cap=len(om) + 8)
    assert n == len(om) and n > 0
    np.testing.assert_array_equal(_np(rf), orf)
    got = np.stack([mv[f].astype(np.int32) for f in ("window", "recv", "donor", "kind", "seq")], 1)
    ref = np.stack([om[f] for f in ("window", "recv", "donor", "kind", "seq")], 1)
    np.testing.assert_array_equal(got, ref)
    assert tre.read_diag(diag)["err"] == 0
    return n


# 17-32 models: one model per lane; 33-64: two; 100: the warp walk, four per
# lane, on rank tables in shared memory.
@pytest.mark.parametrize("M", [17, 24, 32, 33, 40, 48, 64, 100])
@pytest.mark.parametrize("cap", [1, 3])
def test_warp_walk_many_models(tre, M, cap):
    Z, cls, g, r0, budget, r_min = _case(1000 + M * 7 + cap, 3000, M)
    _check(tre, Z, cls, g, r0, budget, r_min, 1000, cap)


@pytest.mark.parametrize("M", [20, 64])
def test_warp_walk_heterogeneous_footprints(tre, M):
    Z, cls, g, r0, budget, r_min = _case(77 + M, 2000, M, hetero=True)
    _check(tre, Z, cls, g, r0, budget, r_min, 1000, 2)


def test_warp_walk_f64(tre):
    Z, cls, g, r0, budget, r_min = _case(91, 2500, 36, dtype=np.float64)
    _check(tre, Z, cls, g, r0, budget, r_min, 1000, 2)


def test_warp_walk_long_series_sixty_four_models(tre):
    """64 models over 86,400 windows of 100 ms (the streaming workload's model
    count and window length over a tenth of its day): tick tables far beyond
    shared memory."""
    Z, cls, g, r0, budget, r_min = _case(5, 86400, 64, idle=0.05)
    r0 = np.full(64, 8, np.int32)
    budget = 512
    _check(tre, Z, cls, g, r0, budget, r_min, 100, 1)


@pytest.mark.parametrize("M", [6, 12])
@pytest.mark.parametrize("fast_ms,slow_ms,win", [(3000, 10000, 1000), (500, 10000, 1000),
                                                 (700, 2100, 100)])
def test_thread_walk_every_tick(tre, M, fast_ms, slow_ms, win):
    """Cadences that are not nested (slow not a multiple of fast) or a fast
    tick shorter than a window: the walk visits every tick, one thread per
    controller instance."""
    Z, cls, g, r0, budget, r_min = _case(300 + M + fast_ms, 3000, M)
    _check(tre, Z, cls, g, r0, budget, r_min, win, 2, fast_ms, slow_ms)


@pytest.mark.parametrize("M", [5, 16])
def test_pacing_cap_above_thirty_two(tre, M):
    """Few models with a pacing cap of 40 transitions per tick (the sweep's
    caps stop at 8): receivers drain every usable donor in one tick."""
    Z, cls, g, r0, budget, r_min = _case(500 + M, 3000, M)
    r0 = r0 * 12
    budget = int((g * r0).sum())
    _check(tre, Z, cls, g, r0, budget, r_min, 1000, 40)


@pytest.mark.parametrize("caps", [None, list(range(1, 13))])
def test_sweep_twenty_four_models(tre, caps):
    """The sweep's walk launch with more than 16 models: one warp per
    (trace, window length, rescue threshold, pacing cap) instance, eight
    caps to a block (twelve caps: two blocks per (series, threshold))."""
    import tracegen
    sw = tracegen.sweep_workload(scale=0.02, n_traces=1, duration_s=600.0)
    rng = np.random.default_rng(8)
    M0, M = sw["M"], 24
    t = sw["traces"][0]
    t["model"] = (t["model"] + M0 * rng.integers(0, 3, len(t["model"]))).astype(np.int32)
    ext = lambda a: np.resize(np.asarray(a), M)
    sw["M"] = M
    for k in ("w_p", "w_q", "tau_surplus", "slo_ttft_ms", "r0", "r_min", "footprint"):
        if np.ndim(sw[k]):
            sw[k] = ext(sw[k]).astype(np.asarray(sw[k]).dtype)
    sw["budget"] = int(sw["r0"].sum()) + 2
    sw["tau_crit"] = sw["tau_crit"][::3]
    sw["pacing_cap"] = (sw["pacing_cap"][::3] if caps is None
                        else np.asarray(caps, dtype=np.asarray(sw["pacing_cap"]).dtype))
    alpha = [min(1.0, w / 5000.0) for w in sw["window_ms"]]
    import torch
    ref = oracle.sweep(sw["traces"], M, sw["duration_ms"], sw["window_ms"], sw["tau_crit"],
                       sw["pacing_cap"], sw["w_p"], sw["w_q"], sw["tau_surplus"], alpha,
                       sw["slo_ttft_ms"], sw["budget"], sw["r0"], sw["r_min"], sw["footprint"],
                       dtype=np.float32)
    out = tre.tre_sweep([{k: torch.as_tensor(v).cuda() for k, v in t.items()}], M,
                        sw["duration_ms"], sw["window_ms"], alpha, sw["tau_crit"],
                        sw["pacing_cap"], sw["w_p"], sw["w_q"], sw["tau_surplus"],
                        sw["slo_ttft_ms"], sw["budget"], sw["r0"], sw["r_min"], sw["footprint"],
                        moves_cap=512)
    moves = tre.sweep_moves(out, len(ref["instances"]), 512)
    rf = _np(out["r_final"])
    total = 0
    for i, inst in enumerate(ref["instances"]):
        np.testing.assert_array_equal(rf[i], inst["r_final"], err_msg=f"instance {i}")
        om = inst["moves"]
        assert int(_np(out["n_moves"])[i]) == len(om), f"instance {i}"
        got = np.stack([moves[i][f].astype(np.int32)
                        for f in ("window", "recv", "donor", "kind", "seq")], 1) \
            if len(om) else np.zeros((0, 5), np.int32)
        ref_m = np.stack([om[f] for f in ("window", "recv", "donor", "kind", "seq")], 1) \
            if len(om) else np.zeros((0, 5), np.int32)
        np.testing.assert_array_equal(got, ref_m, err_msg=f"instance {i}")
        total += len(om)
    assert total > 0


def test_jump_walk_long_series_sixteen_models(tre):
    """Sixteen models over 43,200 windows of 500 ms (the code/chat workload's
    shape): 4,320 ticks, five slabs of the lane walk in two buffers."""
    Z, cls, g, r0, budget, r_min = _case(16, 43200, 16, idle=0.05)
    for cap in (1, 2):
        _check(tre, Z, cls, g, r0, budget, r_min, 500, cap)


@pytest.mark.parametrize("M", [24, 40])
@pytest.mark.parametrize("fast_ms,slow_ms,win", [(3000, 10000, 1000), (500, 10000, 1000),
                                                 (700, 2100, 100)])
def test_warp_walk_cadences(tre, M, fast_ms, slow_ms, win):
    """More than 16 models on cadences that are not nested or with a fast tick
    shorter than a window (the warp walk, every tick visited in order), and on
    nested ones (the lane walk)."""
    Z, cls, g, r0, budget, r_min = _case(900 + M + fast_ms, 3000, M)
    for cap in (1, 3):
        _check(tre, Z, cls, g, r0, budget, r_min, win, cap, fast_ms, slow_ms)


# One tick per window. Ticks are ranked in chunks of 128 and staged 1024 at a time
# (768 for more than 16 models, 384 for more than 32), series of one slab in one
# buffer; row words hold 3 to 6 rank bits for 8, 16, 32 and 64 models. Infinite Z and zeros of both signs (equal, so the lower
# index goes first) sit among the ties.
@pytest.mark.parametrize("hetero,cap", [(False, 1), (False, 5), (True, 3)])
@pytest.mark.parametrize("M,ticks", [(2, 129), (8, 127), (8, 128), (8, 1025), (9, 2200),
                                     (16, 1024), (16, 1025), (17, 129), (32, 768), (32, 769),
                                     (32, 1153), (33, 384), (33, 769), (64, 384), (64, 385),
                                     (64, 768), (64, 1700)])
def test_lane_walk_chunk_and_slab_edges(tre, M, ticks, hetero, cap):
    dtype = np.float64 if ticks % 2 else np.float32
    Z, cls, g, r0, budget, r_min = _case(40 + M + ticks, ticks, M, hetero=hetero, dtype=dtype)
    rng = np.random.default_rng(M)
    for v in (np.inf, 0.0, -0.0):
        Z[rng.random(Z.shape) < 0.04] = v
    budget += 2
    _check(tre, Z, cls, g, r0, budget, r_min, 1000, cap, 1000, 2000)


# A Z that is no number (a zero theta under a zero series) has a place of its own in
# every order: the walk ends, and its moves, final replicas, floors and budget agree
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("M,hetero,cap", [(8, False, 1), (16, False, 4), (16, True, 2),
                                          (33, False, 2), (64, True, 1)])
def test_lane_walk_nan_values(tre, dtype, M, hetero, cap):
    import torch
    K = 1500
    Z, cls, g, r0, budget, r_min = _case(M + cap, K, M, hetero=hetero, dtype=dtype)
    Z[np.random.default_rng(M).random(Z.shape) < 0.1] = np.nan
    prof = {"w_p": 0.2, "w_q": 2.0, "alpha": 0.2, "theta": 1.0, "tau_crit": 0.8,
            "tau_surplus": 1.2}
    mv, rf, n, diag = tre.tre_select_moves(torch.as_tensor(Z).cuda(), torch.as_tensor(cls).cuda(),
                                           prof, 1000, budget, r0, r_min, g, fast_ms=1000,
                                           slow_ms=2000, pacing_cap=cap, moves_cap=1 << 15)
    assert 0 < n == len(mv) and tre.read_diag(diag)["err"] == 0
    r, floor = r0.astype(int), np.minimum(r_min, r0)
    same = lambda a, b: (a["window"], a["seq"], a["recv"]) == (b["window"], b["seq"], b["recv"])
    for i, x in enumerate(mv):
        assert x["window"] >= mv[max(i - 1, 0)]["window"] and x["donor"] != x["recv"]
        assert cls[x["window"], x["recv"]] != 3
        if x["donor"] >= 0:
            r[x["donor"]] -= 1
            assert r[x["donor"]] >= floor[x["donor"]]
        if i + 1 == n or not same(x, mv[i + 1]):
            r[x["recv"]] += 1
            assert (g * r).sum() <= budget
    np.testing.assert_array_equal(_np(rf), r)


# A warp logs 256 moves before it writes them out. Idle pools of whole multiples
# of that, and one fewer and more, are drawn on one a tick within the first slab of
# staged ticks (1024 for 8 models, 384 for 40), with donors' moves behind them;
# the caps' warps lie side by side, cap 1 in the first or in the last of a block.
@pytest.mark.parametrize("caps", [[1, 2, 3, 4, 5, 6, 7, 8], [2, 3, 4, 5, 6, 7, 8, 1]])
@pytest.mark.parametrize("M,pool", [(8, 255), (8, 256), (8, 257), (8, 512), (40, 255), (40, 256)])
def test_lane_walk_full_log(tre, M, pool, caps):
    import torch
    import tracegen
    sw = tracegen.sweep_workload(scale=0.02, n_traces=1, duration_s=200.0)
    t = sw["traces"][0]
    more = np.random.default_rng(8).integers(0, M // 8, len(t["model"]))
    t["model"] = (t["model"] + 8 * more).astype(np.int32)
    r0, r_min, foot, slo = (np.resize(sw[k], M).astype(np.int32)
                            for k in ("r0", "r_min", "footprint", "slo_ttft_ms"))
    args = (M, sw["duration_ms"])
    rest = (sw["w_p"], sw["w_q"], sw["tau_surplus"])
    ctrl = (int(r0.sum()) + pool, r0, r_min, foot)
    ref = oracle.sweep(sw["traces"], *args, [100], [0.8], caps, *rest, [0.02], slo, *ctrl,
                       fast_ms=100, slow_ms=100)["instances"]
    first = ref[caps.index(1)]["moves"]
    drawn = first["donor"] < 0
    slab = 1024 if M <= 16 else 384
    assert drawn.sum() == pool and ((first["window"] < slab) & ~drawn).sum() > 100
    out = tre.tre_sweep([{k: torch.as_tensor(v).cuda() for k, v in t.items()}], *args, [100],
                        [0.02], [0.8], caps, *rest, slo, *ctrl, fast_ms=100, slow_ms=100,
                        moves_cap=4096)
    moves = tre.sweep_moves(out, len(ref), 4096)
    for i, inst in enumerate(ref):
        assert int(_np(out["n_moves"])[i]) == len(inst["moves"]) <= 4096
        for f in ("window", "recv", "donor", "kind", "seq"):
            np.testing.assert_array_equal(moves[i][f], inst["moves"][f], err_msg=f"{i} {f}")
        np.testing.assert_array_equal(_np(out["r_final"])[i], inst["r_final"])
