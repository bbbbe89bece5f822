"""The work a user of the planner has it do, as cases that can be timed.

A case names what is called and on what window.  Windows are drawn on the GPU from the seed alone:
lengths from the families of `paper_2608_12146_b200.windows` and routing counts that keep the
conservation law sum_e a[i][l][e] = k * t_i exactly.  What is called (`kind`):

  plan      one optimizer step's plan, as a planner runs it for every new window: load, place, pack,
            (with `candidates` > 0: initial population by Algorithm 2), anneal, best, destroy
  place     expert placement only (the "reorder" arm of the paper): load, place, pack, destroy
  score     rp_eval_population on `n` explicit layouts of a packed window
  noalloc   rp_eval_layouts_noalloc on `n` device-resident layouts
  diagnose  rp_diagnostics of one layout of a packed window
"""
import math
import random

import numpy as np
import torch

import paper_2608_12146_b200.binding as rp

# ---- cases -------------------------------------------------------------------------------------------


def _case(kind, n_samples, layers, experts, top_k, cap, dp, shards, ranks, family, scale, topics=1, pop=8, sweeps=0,
          candidates=0, n=0, **kw):
    c = dict(kind=kind, n_samples=n_samples, layers=layers, experts=experts, top_k=top_k, cap=cap, dp=dp, shards=shards,
             ranks=ranks, family=family, scale=scale, topics=topics, pop=pop, sweeps=sweeps, candidates=candidates, n=n)
    c.update(kw)
    return c


def listed():
    return [
        # The five windows of paper_2608_12146_b200/windows.py, whole plans from the length-only seed.
        # tiny: a debugging or unit-test sized step; launches and host work decide.
        _case("plan", 64, 4, 16, 2, 4096, 2, 2, 4, "lognormal", 1096, pop=8, sweeps=200, name="plan tiny"),
        # medium: an ordinary RL step of 512 sequences.
        _case("plan", 512, 16, 64, 4, 32768, 8, 8, 8, "lognormal", 2981, pop=256, sweeps=2000, name="plan medium"),
        # large: long-context mixture, 24 layers of 128 experts on 16 ranks.
        _case("plan", 2048, 24, 128, 8, 65536, 16, 16, 16, "mixture", 1096, pop=1024, sweeps=5000, name="plan large"),
        # wide: 48 layers of 256 experts; the demand tensor and the rank loads are at their widest.
        _case("plan", 4096, 48, 256, 8, 131072, 32, 32, 32, "lognormal", 4915, pop=4096, sweeps=5000, name="plan wide"),
        # heavy: 8192 heavy-tailed samples, the largest search budget (the benchmark's headline window).
        _case("plan", 8192, 32, 128, 8, 131072, 16, 16, 32, "pareto", 256, pop=8192, sweeps=20000, name="plan heavy"),
        # The shape of the paper's runs: 64 prompt groups x 8 rollouts, token cap 8192, two EDP shards,
        # samples of different prompts routed differently.
        _case("plan", 512, 24, 64, 8, 8192, 8, 2, 8, "lognormal", 900, topics=4, pop=256, sweeps=2000, name="plan two shards"),
        # Nothing a power of two: rank count, shard map, odd sample and layer counts.
        _case("plan", 1531, 17, 96, 6, 24000, 12, 4, 12, "lognormal", 2500, topics=4, pop=300, sweeps=1500, name="plan ragged"),
        # Initial population by Algorithm 2 (trials, pairing, selection), then a short search.
        _case("plan", 2048, 24, 128, 8, 65536, 16, 16, 16, "mixture", 1096, topics=4, pop=512, sweeps=1000, candidates=256,
              name="plan with candidates"),
        # Expert reordering alone on the widest window.
        _case("place", 4096, 48, 256, 8, 131072, 32, 32, 32, "lognormal", 4915, topics=4, name="place wide"),
        # Scoring a batch of alternative layouts.
        _case("score", 2048, 24, 128, 8, 65536, 16, 16, 16, "mixture", 1096, topics=4, n=256, name="score 256 layouts"),
        # Rescoring a few layouts inside a training loop that may not allocate.
        _case("noalloc", 512, 16, 64, 4, 32768, 8, 8, 8, "lognormal", 2981, n=3, name="score 3 layouts"),
        # Load-balance metrics of the committed layout, logged every step.
        _case("diagnose", 8192, 32, 128, 8, 131072, 16, 16, 32, "pareto", 256, name="diagnose heavy"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same ranges: any kind, sizes spread over their logarithm, odd ones among them."""
    kind = rng.choices(("plan", "plan2", "place", "score", "noalloc", "diagnose"), (10, 2, 3, 3, 1, 1))[0]
    while True:
        dp = rng.choice((2, 3, 4, 6, 8, 8, 12, 16, 16, 24, 32))
        shards = rng.choice([dp, dp, dp, 1, 2] + [g for g in (3, 4, 6, 8) if dp % g == 0])
        rows = _log_int(rng, 2, 14)
        per_cell = math.exp(rng.uniform(math.log(2.5), math.log(170)))
        n_samples = int(rows * dp * per_cell) | rng.choice((0, 1))
        ranks = rng.choice((2, 4, 4, 8, 8, 8, 12, 16, 16, 24, 32, 32))
        experts = ranks * rng.choice((2, 4, 4, 8, 8, 6))
        layers = _log_int(rng, 3, 48)
        cap = rng.choice((4096, 8192, 20000, 32768, 65536, 131072))
        top_k = rng.choice((2, 4, 6, 8))
        # a family's mean length is about 1.9 (lognormal) or 2.7 (pareto) scales; cells come out about 0.95 full
        family = rng.choice(("lognormal", "lognormal", "mixture", "pareto"))
        mean = 0.93 * cap / per_cell
        scale = int(mean / {"lognormal": 1.9, "mixture": 1.0, "pareto": 2.7}[family])
        if family == "mixture":
            scale = int((mean - 0.3 * cap * 5 / 16) / 0.7 / 1.38)
        if not 48 <= n_samples <= 8192 or scale < 4 or experts > 256 or n_samples * layers * experts > 5.1e7:
            continue
        if top_k * cap * -(-dp // shards) >= 2 ** 30 or top_k > experts:
            continue
        c = _case("plan" if kind == "plan2" else kind, n_samples, layers, experts, top_k, cap, dp, shards, ranks, family, scale,
                  topics=rng.choice((1, 4)))
        lp = layers * ranks
        if kind in ("plan", "plan2"):
            c["pop"] = _log_int(rng, 8, 4096)
            c["sweeps"] = 20 * _log_int(rng, 10, 500 if kind == "plan" else 100)
            if kind == "plan2":
                c["candidates"] = _log_int(rng, 16, 300)
            # within a quarter of the largest search, and rank loads of the population within a few GB
            if c["pop"] * c["sweeps"] * lp > 8192 * 20000 * 1024 / 4 or c["pop"] * rows * shards * lp * 8 > 8e9:
                continue
        if kind == "score":
            c["n"] = _log_int(rng, 1, 1000)
            if c["n"] * n_samples * lp > 256 * 8192 * 1024:
                continue
        if kind == "noalloc":
            c["n"] = _log_int(rng, 1, 64)
            if c["n"] * n_samples > 5e5 or c["n"] * 2 * rows * shards > 32768:
                continue
        return c


# ---- inputs -------------------------------------------------------------------------------------------


def _lengths(c, rng):
    n, cap, s = c["n_samples"], c["cap"], float(c["scale"])
    if c["family"] == "lognormal":
        t = np.clip(rng.lognormal(math.log(s), 1.2, n), 16, cap // 4 if cap > 8192 else cap // 2)
    elif c["family"] == "mixture":      # 70 % short, 30 % long sequences
        short = np.clip(rng.lognormal(math.log(s), 0.8, n), 16, cap)
        long_ = rng.integers(cap // 8, cap // 2, n, endpoint=True).astype(np.float64)
        t = np.where(rng.random(n) < 0.7, short, long_)
    else:                               # heavy tail
        t = np.clip(s * (1.0 + rng.pareto(1.5, n)), s, cap // 2)
    return np.clip(np.floor(t), 1, cap).astype(np.int32)


def _demand(c, lengths, rng, seed):
    """Routing counts [N][L][E]: k * t_i assignments per layer, multinomial over the layer's popularity
    (one popularity, or one of `topics` sharpened and rotated copies of it per sample)."""
    L, E = c["layers"], c["experts"]
    pop = rng.dirichlet(np.full(E, 0.2), size=L)
    tp = np.stack([np.roll(pop, 3 * k + 1, axis=1) ** (1.0 + 0.5 * k) for k in range(4)]) if c["topics"] == 4 else pop[None]
    tp = np.maximum(tp, 1e-9)
    tp /= tp.sum(axis=2, keepdims=True)
    tail = np.cumsum(tp[:, :, ::-1], axis=2)[:, :, ::-1]
    cond = torch.from_numpy(np.clip(tp / tail, 0.0, 1.0)).cuda()            # P(expert e | not an earlier one)
    topic = torch.from_numpy(rng.integers(0, tp.shape[0], c["n_samples"])).cuda()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 13)
    left = (lengths.double() * c["top_k"])[:, None].expand(-1, L).contiguous()
    out = torch.empty((c["n_samples"], L, E), dtype=torch.int32, device="cuda")
    for e in range(E - 1):
        x = torch.binomial(left, cond[:, :, e][topic], generator=gen)
        out[:, :, e] = x
        left -= x
    out[:, :, E - 1] = left
    return out


def _load(s):
    c = s["case"]
    return rp.rp_window_load(s["lengths"], s["demand"], top_k=c["top_k"], token_cap=c["cap"], dp_width=c["dp"],
                             ep_width=c["ranks"], pop_size=c["pop"], edp_of_dp=s["edp"], seed=s["seed"],
                             stream=torch.cuda.current_stream())


def prepare(case, seed):
    rng = np.random.default_rng([int(seed), 2608])
    lengths = torch.from_numpy(_lengths(case, rng)).cuda()
    s = dict(case=case, seed=int(seed), lengths=lengths, demand=_demand(case, lengths, rng, seed))
    s["edp"] = None if case["shards"] == case["dp"] else [d * case["shards"] // case["dp"] for d in range(case["dp"])]
    if case["kind"] in ("score", "noalloc", "diagnose"):
        # a packed window and layouts like those a search visits: the seed with rows and slots exchanged
        # and some samples swapped
        ctx = s["ctx"] = _load(s)
        rp.rp_place_experts(ctx)
        rows, _ = rp.rp_pack_rows(ctx)
        seed_layout = torch.from_numpy(rp.rp_best(ctx)[0]).cuda().long()
        n, N, K = max(1, case["n"]), case["n_samples"], rows * case["dp"]
        perm = torch.from_numpy(np.stack([rng.permutation(K) for _ in range(n)])).cuda()
        lay = perm[:, seed_layout]
        i = torch.from_numpy(rng.integers(0, N, (n, N // 8 + 1))).cuda()
        lay = lay.scatter(1, i, lay.gather(1, (i * 5 + 1) % N))
        s["layouts"] = lay.to(torch.int32).contiguous()
        if case["kind"] != "diagnose":
            s["score_fx"] = torch.empty((n, 3), dtype=torch.int64, device="cuda")
            s["score_f64"] = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


# ---- one pass -----------------------------------------------------------------------------------------


def run(s):
    c = s["case"]
    if c["kind"] == "score":
        return rp.rp_eval_population(s["ctx"], s["layouts"], s["score_fx"], s["score_f64"])
    if c["kind"] == "noalloc":
        return rp.rp_eval_layouts_noalloc(s["ctx"], s["layouts"], s["score_fx"], s["score_f64"])
    if c["kind"] == "diagnose":
        return rp.rp_diagnostics(s["ctx"], s["layouts"])
    ctx = _load(s)
    pi, rank_load = rp.rp_place_experts(ctx)
    rows, certified = rp.rp_pack_rows(ctx)
    out = dict(pi=pi, rank_load=rank_load, rows=rows, certified=certified)
    if c["kind"] == "plan":
        if c["candidates"]:
            out["distinct"], out["picked"] = rp.rp_init_population(ctx, c["candidates"])
        st = rp.rp_anneal(ctx, n_levels=20, steps_per_level=c["sweeps"] // 20, t0=1e-3, t_ratio=10.0 ** (-3.0 / 19.0),
                          p_reloc=0.25, p_guide=0.8)
        out["counts"] = [st.proposed, st.feasible, st.accepted, st.improved]
        out["layout"], out["score_fx"], out["score_f64"] = rp.rp_best(ctx)
    rp.rp_destroy(ctx)
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------------


def work(case):
    """Bytes: inputs once, outputs once.  "flops": the integer additions and comparisons of the method: every
    count of the demand tensor once for the totals and once for the projection; two tentative rank-load slices
    (add and compare) for each proposal that fits, taken as a quarter of the proposals; a demand row per sample
    and layout scored, candidate paired or diagnosed."""
    N, LE, LP = case["n_samples"], case["layers"] * case["experts"], case["layers"] * case["ranks"]
    if case["kind"] in ("score", "noalloc", "diagnose"):
        n = max(1, case["n"])
        out = 64.0 if case["kind"] == "diagnose" else 48.0 * n
        return {"bytes": 4.0 * N * LP + 4.0 * n * N + 4.0 * N + out, "flops": float(n) * N * LP}
    b = 4.0 * N * LE + 4.0 * N + 4.0 * LE + 8.0 * LP
    f = 2.0 * N * LE
    if case["kind"] == "plan":
        b += 4.0 * N + 48.0
        f += 4.0 * LP * 0.25 * case["pop"] * case["sweeps"] + 2.0 * case["candidates"] * N * LP
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Every decision and score is integer arithmetic, and the reported doubles are one correctly rounded
    division of those integers.  Only the coefficients of variation of the diagnostics are floating-point sums
    (64 bits, at most a few thousand terms, one square root): another order of the terms moves them by a few
    1e-16 each."""
    return {"rel": 1e-13} if case["kind"] == "diagnose" else "exact"
