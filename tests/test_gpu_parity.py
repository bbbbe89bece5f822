"""Parity of the CUDA path (through the C ABI) with the CPU oracle, element by element.

Integers, indices, placements, layouts and the whole annealing trajectory must be bit-exact;
the reported fp64 objective must agree with the oracle's real-valued evaluation to 1e-9
relative (the tolerance the benchmark spec states).
"""
import os

import numpy as np
import pytest

import oracle
import paper_2608_12146_b200.binding as rp
from paper_2608_12146_b200.windows import Window, custom_spec, make_window

pytestmark = pytest.mark.gpu
F64_RTOL = 1e-9


def load(w, pop=None, edp=None, min_rows=0, device_inputs=False):
    s = w.spec
    t, a = w.lengths, w.demand
    if device_inputs:
        import torch
        t, a = torch.from_numpy(t).cuda(), torch.from_numpy(a).cuda()
    ctx = rp.rp_window_load(t, a, top_k=s.top_k, token_cap=s.token_cap, dp_width=s.dp_width,
                            ep_width=s.ep_width, pop_size=pop or s.pop_size, edp_of_dp=edp,
                            alpha=s.alpha, beta=s.beta, min_rows=min_rows, seed=s.anneal_seed)
    rp.rp_debug_set_trace(ctx, True)          # the parity checks read the per-level traces
    return ctx


def oracle_front(w, edp=None, min_rows=0):
    s = w.spec
    Lagg = oracle.aggregate(w.demand)
    pi, G = oracle.lpt(Lagg, s.ep_width)
    q = oracle.project(w.demand, pi, s.ep_width)
    R, cert, seed = oracle.pack_ffd(w.lengths, s.token_cap, s.dp_width, min_rows)
    return dict(Lagg=Lagg, pi=pi, G=G, q=q, R=R, cert=cert, seed=seed)


def check_front(w, ctx, ref):
    s = w.spec
    pi, load_ = rp.rp_place_experts(ctx)
    assert (rp.rp_debug_dump(ctx, "LAGG", (s.n_layers, s.n_experts), np.int64) == ref["Lagg"]).all()
    assert (pi == ref["pi"]).all()
    assert (load_ == ref["G"]).all()
    q = rp.rp_debug_dump(ctx, "Q", (s.n_samples, s.n_layers, s.ep_width), np.int32)
    assert (q == ref["q"]).all()
    R, cert = rp.rp_pack_rows(ctx)
    assert (R, cert) == (ref["R"], ref["cert"])
    assert (rp.rp_debug_dump(ctx, "SEED_LAYOUT", (s.n_samples,), np.int32) == ref["seed"]).all()
    return R


def check_eval(w, ctx, ref, edp, n=6, seed=0):
    s = w.spec
    R, D = ref["R"], s.dp_width
    rng = np.random.default_rng(seed)
    lays = rng.integers(0, R * D, (n, s.n_samples)).astype(np.int32)
    lays[0] = ref["seed"]
    fx, f64 = rp.rp_eval_population(ctx, lays)
    ev = oracle.eval_layouts(w.lengths, ref["q"], lays, R, s.token_cap, D, edp, s.alpha, s.beta)
    assert (fx == ev["score"]).all()
    G = 1 + (max(edp) if edp is not None else D - 1)
    for j in range(n):
        Wj = rp.rp_debug_dump(ctx, "EVAL_W", (R, G, s.n_layers, s.ep_width), np.int32, index=j)
        assert (Wj == ev["W"][j]).all()
        real = oracle.eval_f64(w.lengths, ref["q"], lays[j], R, s.token_cap, D, edp, s.alpha, s.beta)
        np.testing.assert_allclose(f64[j], real, rtol=F64_RTOL, atol=0)


def check_anneal(w, ctx, ref, edp, pop, levels, steps, threads=8, t_ratio=None, check_members=3, init=None, t0=None):
    s = w.spec
    t0 = s.t0 if t0 is None else t0
    R, D = ref["R"], s.dp_width
    ratio = s.t_ratio if t_ratio is None else t_ratio
    if init is None:
        init = np.tile(ref["seed"], (pop, 1))
    want = oracle.anneal(w.lengths, ref["q"], init, R, s.token_cap, D, n_levels=levels, steps=steps, t0=t0,
                         t_ratio=ratio, p_reloc=s.p_reloc, p_guide=s.p_guide, seed=s.anneal_seed,
                         edp_of_dp=edp, alpha=s.alpha, beta=s.beta, n_threads=threads)
    assert want["status"] == 0
    stats = rp.rp_anneal(ctx, n_levels=levels, steps_per_level=steps, t0=t0, t_ratio=ratio,
                         p_reloc=s.p_reloc, p_guide=s.p_guide)
    got_counters = [stats.proposed, stats.feasible, stats.accepted, stats.improved]
    assert got_counters == want["counters"].tolist()
    # the whole trajectory, level by level
    assert (rp.rp_debug_dump(ctx, "TRACE_DIGEST", (levels, pop), np.uint64) == want["digest"]).all()
    assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (levels, pop, 3), np.int64) == want["term"]).all()
    assert (rp.rp_debug_dump(ctx, "TRACE_BEST", (levels, pop, 3), np.int64) == want["best"]).all()
    assert (rp.rp_debug_dump(ctx, "TRACE_BEST_STEP", (levels, pop), np.int32) == want["best_step"]).all()
    if levels > 1:
        assert (rp.rp_debug_dump(ctx, "TRACE_ANC", (levels - 1, pop), np.int32) == want["anc"]).all()
    assert (rp.rp_debug_dump(ctx, "TRACE_INCUMBENT", (levels, 3), np.int64) == want["incumbent"]).all()
    # final population and the incumbent
    popl = rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32)
    assert (popl == want["final_pop"]).all()
    layout, fx, f64 = rp.rp_best(ctx)
    assert (layout == want["best_layout"]).all() and (fx == want["best_score"]).all()
    real = oracle.eval_f64(w.lengths, ref["q"], layout, R, s.token_cap, D, edp, s.alpha, s.beta)
    np.testing.assert_allclose(f64, real, rtol=F64_RTOL, atol=0)
    # incrementally maintained state of a few members equals the oracle's full evaluation
    G = 1 + (max(edp) if edp is not None else D - 1)
    for j in sorted(set([0, pop // 2, pop - 1]))[:check_members]:
        ev = oracle.eval_layouts(w.lengths, ref["q"], popl[j], R, s.token_cap, D, edp, s.alpha, s.beta)
        assert (rp.rp_debug_dump(ctx, "W", (R, G, s.n_layers, s.ep_width), np.int32, index=j) == ev["W"][0]).all()
        assert (rp.rp_debug_dump(ctx, "CELL_T", (R * D,), np.int64, index=j) == ev["T"][0]).all()
        assert (rp.rp_debug_dump(ctx, "CELL_Q", (R * D,), np.int64, index=j) == ev["Q"][0]).all()
        assert (rp.rp_debug_dump(ctx, "CELL_CNT", (R * D,), np.int32, index=j) == ev["cnt"][0]).all()
        assert (rp.rp_debug_dump(ctx, "ESUM", (R, G), np.int64, index=j) * (256 * s.token_cap) == ev["Efx"][0]).all()
    # scoring the current population from scratch agrees with the last terminal scores
    fx_pop, _ = rp.rp_eval_population(ctx)
    assert (fx_pop == want["term"][-1]).all()
    # load-balance diagnostics of the incumbent and of the seed
    pi = oracle.lpt(ref["Lagg"], s.ep_width)[0]
    for lay, arg in ((want["best_layout"], None), (ref["seed"], ref["seed"])):
        d_want = oracle.diagnostics(w.lengths, ref["q"], ref["Lagg"], pi, lay, R, s.token_cap, D, edp, s.alpha, s.beta)
        d_got = rp.rp_diagnostics(ctx, arg)
        for key in ("s_ep", "t_ep", "n_ep"):
            assert d_got[key] == d_want[key], key
        for key in ("cv_identity", "cv_placed", "eta_ep", "attention", "joint"):
            assert abs(d_got[key] - d_want[key]) <= F64_RTOL * abs(d_want[key]), key
    return want, stats


# ---------------------------------------------------------------------------------------------
def log_boundary_words():
    """Words whose (x+1)'s base-2 logarithm lies within 2^-26 of a 24-bit fraction boundary, powers of two aside: where the
    device leaves the double-precision logarithm for the definition."""
    k = np.arange(1, 1 << 24, dtype=np.float64)
    root = np.exp2(k / (1 << 24))
    found = []
    for e in range(25, 32):
        exact = root * float(1 << e)
        near = np.abs(np.rint(exact) - exact) < 2.0 ** -17          # (a superset: one part in 2^49 of up to 2^32)
        v, kk = np.rint(exact[near]).astype(np.uint64), k[near].astype(np.longdouble)
        y = (np.log2(v.astype(np.longdouble)) - e) * (1 << 24)
        found.append(v[np.abs(y - kk) < np.longdouble(2.0) ** -26])
    return (np.unique(np.concatenate(found)) - 1).astype(np.uint32)


def test_device_integer_functions_bit_exact():
    rng = np.random.default_rng(0)
    ctr = rng.integers(0, 2 ** 32, (4096, 4), dtype=np.uint64).astype(np.uint32)
    ctr[0] = 0
    ctr[1] = 0xFFFFFFFF
    key = np.array([0xA4093822, 0x299F31D0], np.uint32)
    got = rp.rp_debug_philox(ctr, key)
    for i in list(range(64)) + [4095]:
        assert (got[i] == oracle.philox4x32_10(ctr[i], key)).all()
    x = np.concatenate([rng.integers(0, 2 ** 32, 20000, dtype=np.uint64).astype(np.uint32),
                        np.array([0, 1, 2, 3, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 2, 2 ** 32 - 1], np.uint32),
                        (2 ** np.arange(1, 32, dtype=np.uint64) - 1).astype(np.uint32)])
    near = log_boundary_words()
    assert near.size > 100                 # one word in 2^25 is expected to lie there
    x = np.concatenate([x, near, near - 1, near + 1])
    got = rp.rp_debug_nl2(x)
    assert got.tolist() == [oracle.nl2(int(v)) for v in x]
    z = np.concatenate([rng.integers(0, 34 << 32, 20000, dtype=np.uint64),
                        np.array([0, 1, 255, 256, 2 ** 32 - 1, 2 ** 32, 32 << 32, (32 << 32) - 1, 2 ** 40, 2 ** 63], np.uint64)])
    got = rp.rp_debug_exp2neg(z)
    assert got.tolist() == [oracle.exp2neg(int(v)) for v in z]


def test_philox_against_the_curand_header(tmp_path):
    """A third implementation: cuRAND's device function, compiled here with nvcc (skipped when the
    toolkit is not on the machine), against the library's and the oracle's words."""
    import ctypes
    import shutil
    import subprocess
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "aux", "philox_curand.cu")
    so = str(tmp_path / "philox_curand.so")
    res = subprocess.run([nvcc, "-O2", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared",
                          "-o", so, src], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    lib = ctypes.CDLL(so)
    rng = np.random.default_rng(12)
    ctr = rng.integers(0, 2 ** 32, (512, 4), dtype=np.uint64).astype(np.uint32)
    ctr[0] = 0
    ctr[1] = 0xFFFFFFFF
    key = np.array([0x243F6A88, 0x85A308D3], np.uint32)
    out = np.zeros_like(ctr)
    assert lib.curand_philox_host(ctr.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint32(int(key[0])), ctypes.c_uint32(int(key[1])),
                                  out.ctypes.data_as(ctypes.c_void_p), ctypes.c_int(len(ctr))) == 0
    assert (rp.rp_debug_philox(ctr, key) == out).all()
    for i in range(32):
        assert (out[i] == oracle.philox4x32_10(ctr[i], key)).all()


@pytest.mark.parametrize("per_level", [2, 1], ids=["one_launch", "launch_per_level"])
@pytest.mark.parametrize("name", ["tiny", "medium"])
def test_named_window_full_budget(name, per_level):
    """The two windows the oracle finishes in seconds, at their full population and sweeps: all
    levels in one launch (every chain is resident at once), and one launch per level."""
    w = make_window(name)
    s = w.spec
    ref = oracle_front(w)
    ctx = load(w, device_inputs=(name == "medium"))
    rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", per_level)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, None)
    check_anneal(w, ctx, ref, None, s.pop_size, s.n_levels, s.steps_per_level)
    rp.rp_destroy(ctx)


EDGE_SPECS = [
    # name, N, L, E, k, C, D, P, edp, min_rows   (ragged sizes, non-power-of-two ranks, shared shards)
    ("ragged", 77, 3, 12, 2, 3000, 3, 3, None, 4),
    ("shared_shards", 96, 5, 16, 2, 4096, 4, 4, [0, 0, 1, 1], 3),
    ("one_shard", 64, 2, 8, 1, 2048, 4, 8, [0, 0, 0, 0], 3),
    ("interleaved", 120, 7, 24, 3, 4096, 6, 6, [0, 1, 2, 0, 1, 2], 2),
    ("one_rank", 50, 4, 5, 2, 2048, 2, 1, None, 4),
    ("wide_ranks", 90, 2, 96, 2, 4096, 2, 48, None, 5),
    ("single_slot", 40, 3, 8, 2, 2048, 1, 4, None, 6),
    ("vector_tail", 130, 9, 40, 2, 8192, 5, 20, [0, 1, 1, 2, 2], 3),
    # L*k*C*(cells per row-shard) >= 2^31: the sums over layers of the busiest ranks need 64 bits
    ("wide_sums", 72, 64, 16, 8, 1 << 20, 4, 4, [0, 0, 0, 0], 3),
    # more ranks than the register-resident placement holds (128): its shared-memory form
    ("many_ranks", 60, 2, 160, 2, 4096, 2, 160, None, 4),
]


@pytest.mark.parametrize("spec", EDGE_SPECS, ids=[e[0] for e in EDGE_SPECS])
def test_edge_shapes(spec):
    name, N, L, E, k, C, D, P, edp, min_rows = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, 24, 400, data_seed=len(name) * 7 + N))
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=24, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, edp)
    want, stats = check_anneal(w, ctx, ref, edp, 24, 8, 50, t_ratio=0.6)
    assert stats.accepted > 50
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("per_level", [2, 1], ids=["one_launch", "launch_per_level"])
def test_resampling_under_selection_pressure_small_population(per_level):
    """A cold schedule on a window whose samples really differ: resampling replaces many members
    every level, so chains adopt other members' states (and others keep theirs on chip when all
    levels run in one launch); several rp_anneal calls in a row continue from one another."""
    w = make_window(custom_spec("pressure", 140, 6, 32, 2, 4096, 4, 8, 100, 400, data_seed=321))
    s = w.spec
    edp = [0, 1, 1, 0]
    ref = oracle_front(w, edp, 3)
    ctx = load(w, pop=100, edp=edp, min_rows=3)
    rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", per_level)
    check_front(w, ctx, ref)
    want, stats = check_anneal(w, ctx, ref, edp, 100, 12, 300, t_ratio=0.5, t0=2e-5, check_members=3)    # 300 steps: two batches of step records
    anc = want["anc"]
    assert any(len(set(a.tolist())) < 60 for a in anc) and stats.gather_bytes > 0
    again = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, s.dp_width, n_levels=5,
                          steps=33, t0=1e-5, t_ratio=0.7, p_reloc=0.4, p_guide=0.8, seed=s.anneal_seed,
                          edp_of_dp=edp, alpha=s.alpha, beta=s.beta)
    rp.rp_anneal(ctx, n_levels=5, steps_per_level=33, t0=1e-5, t_ratio=0.7, p_reloc=0.4, p_guide=0.8)
    assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (5, 100, 3), np.int64) == again["term"]).all()
    assert (rp.rp_debug_dump(ctx, "TRACE_ANC", (4, 100), np.int32) == again["anc"]).all()
    assert (rp.rp_debug_dump(ctx, "POPULATION", (100, s.n_samples), np.int32) == again["final_pop"]).all()
    layout, fx, _ = rp.rp_best(ctx)
    best = min((tuple(want["best_score"]), 0), (tuple(again["best_score"]), 1))
    assert tuple(fx) == best[0]
    assert (layout == (want, again)[best[1]]["best_layout"]).all()
    G = 2
    for j in (0, 57, 99):
        ev = oracle.eval_layouts(w.lengths, ref["q"], again["final_pop"][j], ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
        assert (rp.rp_debug_dump(ctx, "W", (ref["R"], G, s.n_layers, s.ep_width), np.int32, index=j) == ev["W"][0]).all()
    rp.rp_destroy(ctx)


def test_three_attention_stages_and_resume():
    """Three stage types with fractional coefficients; a second rp_anneal call continues from
    the population the first one left (the oracle is restarted from that population)."""
    w = make_window(custom_spec("stages", 100, 4, 16, 2, 4096, 4, 4, 16, 300, data_seed=99,
                                alpha=(0.5, 2.25, 1.0), beta=(0.0, 0.75, 3.0)))
    s = w.spec
    edp = [0, 0, 1, 1]
    ref = oracle_front(w, edp, 3)
    ctx = load(w, pop=16, edp=edp, min_rows=3)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, edp)
    want, _ = check_anneal(w, ctx, ref, edp, 16, 5, 40, t_ratio=0.5)
    # resume
    again = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, s.dp_width, n_levels=3,
                          steps=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed,
                          edp_of_dp=edp, alpha=s.alpha, beta=s.beta)
    rp.rp_anneal(ctx, n_levels=3, steps_per_level=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
    assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (3, 16, 3), np.int64) == again["term"]).all()
    assert (rp.rp_debug_dump(ctx, "POPULATION", (16, s.n_samples), np.int32) == again["final_pop"]).all()
    _, fx, _ = rp.rp_best(ctx)
    assert tuple(fx) == min(tuple(want["best_score"]), tuple(again["best_score"]))
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("kernel", [1, 2], ids=["several_warps_per_chain", "warp_per_chain"])
@pytest.mark.parametrize("name,pop,levels,steps", [("large", 96, 3, 60), ("wide", 48, 2, 40), ("heavy", 64, 2, 80)])
def test_large_windows_full_shapes_reduced_budget(name, pop, levels, steps, kernel):
    """Full N, L, E, P, C, D of the three big windows (so the kernels run in the launch
    configuration of the full-size runs), with a population and step budget the oracle finishes
    quickly, on both chain kernels that take such windows; every trajectory is still compared bit
    for bit."""
    w = make_window(name)
    ref = oracle_front(w)
    ctx = load(w, pop=pop, device_inputs=True)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", kernel)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, None, n=2)
    check_anneal(w, ctx, ref, None, pop, levels, steps, check_members=2)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("name,pop,levels,steps,t0", [("large", 1024, 20, 250, None), ("heavy", 8192, 2, 1000, None),
                                                      ("wide", 4096, 2, 250, 2e-5)])
def test_large_windows_full_population(name, pop, levels, steps, t0, threads=16):
    """The three big windows at the population the benchmark runs them at (large at its whole
    budget, heavy and wide for two levels of their real step count), every trace against the
    oracle: this is where the four-members-per-thread weights, the cumulative weights in global
    memory, the off-chip cell bookkeeping and the multi-wave rank-load free list run.  (Wide starts
    colder than its schedule does, so that already its first resampling replaces members.)"""
    w = make_window(name)
    assert pop == w.spec.pop_size and steps == w.spec.steps_per_level
    ref = oracle_front(w)
    ctx = load(w, pop=pop, device_inputs=True)
    check_front(w, ctx, ref)
    want, stats = check_anneal(w, ctx, ref, None, pop, levels, steps, threads=threads, check_members=2, t0=t0)
    assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row"
    assert stats.accepted > pop            # the levels did move
    if levels > 1:                          # resampling really replaced members and kept others
        anc = want["anc"][0]
        assert 1 < len(set(anc.tolist())) < pop
    rp.rp_destroy(ctx)


BARRIER_CASES = [
    # name, N, L, E, k, C, D, P, edp, min_rows, pop   (first two: warp-per-candidate kernel; last two: cooperative kernel, L*P > 512)
    ("ws_small", 96, 5, 16, 2, 4096, 4, 4, [0, 0, 1, 1], 3, 37),
    ("ws_pow2", 130, 9, 40, 2, 8192, 5, 20, None, 3, 64),
    ("ws_coop", 120, 20, 32, 2, 4096, 4, 32, None, 3, 40),
    ("ws_coop_shared", 150, 17, 64, 2, 4096, 4, 32, [0, 1, 1, 0], 2, 130),
]


@pytest.mark.parametrize("spec", BARRIER_CASES, ids=[e[0] for e in BARRIER_CASES])
@pytest.mark.parametrize("cap", [0, 64])
def test_level_barrier_paths_on_small_windows(spec, cap):
    """The level barrier with all of its shared memory (cap 0) and with next to none (cap 64: the
    cumulative weights, the cell bookkeeping and the incumbent's replay go through global memory,
    as they do for populations of thousands), on windows small enough for many levels; the
    cooperative kernel is reached with L*P > 512."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 11 + N))
    ref = oracle_front(w, edp, min_rows)
    for slices in ((1, 2) if L * P > 512 else (0,)):       # cooperative kernel: rank loads as shared slices, and as cells
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        rp.rp_debug_set_knob(ctx, "BARRIER_WORKSPACE", cap)
        rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", 1)    # the barrier in question is the one between launches
        rp.rp_debug_set_knob(ctx, "RANK_LOAD_SLICES", slices)
        rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 1)        # (L*P > 512: the 128-thread kernel, not one warp per chain)
        check_front(w, ctx, ref)
        want, stats = check_anneal(w, ctx, ref, edp, pop, 10, 40, t_ratio=0.6, check_members=2)
        assert stats.accepted > 50 and stats.improved > 0
        if slices == 1:
            assert stats.gather_bytes == 0          # nothing is copied when members share slices
            # resume: the tables survive between calls
            s_ = w.spec
            again = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s_.token_cap, s_.dp_width, n_levels=3,
                                  steps=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s_.anneal_seed,
                                  edp_of_dp=edp, alpha=s_.alpha, beta=s_.beta)
            rp.rp_anneal(ctx, n_levels=3, steps_per_level=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
            assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (3, pop, 3), np.int64) == again["term"]).all()
            assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s_.n_samples), np.int32) == again["final_pop"]).all()
            G = 1 + (max(edp) if edp is not None else D - 1)
            for j in (0, pop - 1):
                ev = oracle.eval_layouts(w.lengths, ref["q"], again["final_pop"][j], ref["R"], s_.token_cap, D, edp, s_.alpha, s_.beta)
                assert (rp.rp_debug_dump(ctx, "W", (ref["R"], G, L, P), np.int32, index=j) == ev["W"][0]).all()
        rp.rp_destroy(ctx)


OTHER_RANK_CASES = [
    # name, N, L, E, k, C, D, P, edp, min_rows, pop: L*P > 512 with rank counts that are not a power of two from 4 to 128
    ("ranks_48", 100, 12, 48, 2, 4096, 4, 48, None, 3, 30),
    ("ranks_2", 90, 300, 4, 2, 4096, 3, 2, [0, 1, 0], 2, 21),
    ("ranks_3", 64, 180, 6, 1, 3000, 2, 3, None, 4, 9),
]


@pytest.mark.parametrize("spec", OTHER_RANK_CASES, ids=[e[0] for e in OTHER_RANK_CASES])
def test_slice_pool_windows_with_other_rank_counts(spec):
    """Windows whose rank loads live in the slice pool but whose rank count the warp-per-chain
    kernel does not take (its layers must be whole 16-byte chunks): the 128-thread kernel runs them
    by default, with its element-wise scoring loop."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 17 + N))
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    want, stats = check_anneal(w, ctx, ref, edp, pop, 6, 40, t_ratio=0.6, check_members=2)
    assert stats.accepted > 0 and stats.kernel_launches == 6 * 3
    rp.rp_destroy(ctx)


WARP_CHAIN_CASES = [
    # name, N, L, E, k, C, D, P, edp, min_rows, pop: windows with 512 < L*P <= 1024 for the warp-per-chain kernel
    ("wc_ragged", 120, 20, 32, 2, 4096, 4, 32, None, 3, 40),            # 160 chunks of 16 bytes: 5 per lane
    ("wc_shared", 151, 17, 64, 2, 4096, 4, 32, [0, 1, 1, 0], 2, 130),   # two DP slots per shard, odd sample count
    ("wc_p4", 140, 200, 16, 2, 4096, 4, 4, None, 3, 33),                # one lane per layer
    ("wc_p128", 100, 8, 128, 2, 4096, 3, 128, None, 2, 50),             # a whole warp per layer, L*P = 1024
    ("wc_cells", 700, 16, 64, 2, 8192, 64, 64, None, 5, 24),            # 320 cells
]


@pytest.mark.parametrize("spec", WARP_CHAIN_CASES, ids=[e[0] for e in WARP_CHAIN_CASES])
def test_warp_per_chain_kernel_on_small_windows(spec):
    """The chain kernel that full-size windows with thousands of chains use (one warp per chain),
    forced onto small windows: ragged chunk counts, one to 32 chunks per layer, fewer layers than
    lanes and more, shared shards, more than 256 cells; the level barrier as a launch of its own,
    with all of its shared memory and with next to none; a second rp_anneal call that resumes
    from the tables."""
    kernel = 2
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 13 + N))
    ref = oracle_front(w, edp, min_rows)
    for cap in (0, 64):
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", kernel)
        rp.rp_debug_set_knob(ctx, "BARRIER_WORKSPACE", cap)
        check_front(w, ctx, ref)
        want, stats = check_anneal(w, ctx, ref, edp, pop, 8, 40, t_ratio=0.6, check_members=2)
        assert stats.accepted > 50 and stats.improved > 0
        assert stats.gather_bytes == 0 and stats.kernel_launches == 8 * 4       # bookkeeping (2), chains, barrier
        s_ = w.spec
        again = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s_.token_cap, s_.dp_width, n_levels=3,
                              steps=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s_.anneal_seed,
                              edp_of_dp=edp, alpha=s_.alpha, beta=s_.beta)
        rp.rp_anneal(ctx, n_levels=3, steps_per_level=30, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
        assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (3, pop, 3), np.int64) == again["term"]).all()
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s_.n_samples), np.int32) == again["final_pop"]).all()
        G = 1 + (max(edp) if edp is not None else D - 1)
        for j in (0, pop - 1):
            ev = oracle.eval_layouts(w.lengths, ref["q"], again["final_pop"][j], ref["R"], s_.token_cap, D, edp, s_.alpha, s_.beta)
            assert (rp.rp_debug_dump(ctx, "W", (ref["R"], G, L, P), np.int32, index=j) == ev["W"][0]).all()
        rp.rp_destroy(ctx)


PERMUTED_CASES = [
    # name, N, L, E, k, C, D, P, min_rows, pop, knob: one DP slot per shard, but slot d is not shard d
    ("perm_on_chip", 96, 5, 16, 2, 4096, 4, 4, 3, 20, 0),
    ("perm_warp", 120, 20, 32, 2, 4096, 4, 32, 3, 24, 2),
    ("perm_128_threads", 1100, 16, 64, 2, 8192, 64, 64, 8, 8, 1),      # 512 cells: the form without per-cell key caches is in reach
]


@pytest.mark.parametrize("spec", PERMUTED_CASES, ids=[e[0] for e in PERMUTED_CASES])
def test_permuted_shards(spec):
    """As many shards as DP slots, in another order: a cell and its row-shard then differ in index,
    on each chain kernel."""
    name, N, L, E, k, C, D, P, min_rows, pop, kernel = spec
    edp = [(d + 1) % D for d in range(D)]
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 13 + N))
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", kernel)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, edp, pop, 4, 60, t_ratio=0.6, check_members=2)
    assert stats.accepted > 0
    rp.rp_destroy(ctx)


ROW_CASES = [
    # name, N, L, E, k, C, D, P, edp, min_rows, pop: one launch for all levels up to 1184 members, else one per level
    ("row_one_chunk", 70, 32, 8, 2, 4096, 3, 4, None, 3, 21),              # a lane per layer, exactly 32 layers
    ("row_33_layers", 66, 33, 16, 2, 4096, 2, 8, [1, 0], 4, 9),            # two layers per lane, a permuted shard map
    ("row_65_layers", 61, 65, 8, 1, 4096, 2, 4, [0, 0], 4, 5),             # four layers per lane
    ("row_8_chunks", 90, 20, 64, 2, 4096, 4, 32, [0, 1, 1, 0], 3, 160),    # L*P > 512: starts from slices, two chains per CTA
    ("row_padded", 57, 5, 10, 2, 4096, 3, 5, [0, 1, 1], 3, 310),           # rows padded to whole chunks, four chains per CTA
    ("row_8_per_cta", 40, 3, 8, 2, 4096, 2, 8, None, 3, 601),              # no warp left for the step records
    ("row_levels", 60, 24, 32, 2, 4096, 3, 16, [0, 0, 1], 3, 1190),        # one launch per level, four chunks per lane
    ("row_levels_pad", 45, 6, 6, 2, 4096, 2, 3, None, 3, 1201),            # the same with padded rows
    ("row_levels_64", 48, 64, 8, 2, 4096, 2, 4, None, 3, 1185),            # the same, two layers per lane
]


@pytest.mark.parametrize("spec", ROW_CASES, ids=[e[0] for e in ROW_CASES])
def test_one_layer_per_lane_kernel(spec):
    """The chain kernel most windows use, at the edges of its lanes, chunks, chains per CTA and launch
    forms; then the same population annealed on by another kernel and by this one again, so that the
    rank loads change form and back."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 23 + N))
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row"
    want, stats = check_anneal(w, ctx, ref, edp, pop, 3, 40, t_ratio=0.5, check_members=2)
    assert stats.accepted > 0
    for knob in (1, 0):
        rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", knob)
        want = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, D, n_levels=2, steps=33, t0=1e-4,
                             t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed, edp_of_dp=edp, alpha=s.alpha,
                             beta=s.beta, n_threads=8)
        rp.rp_anneal(ctx, n_levels=2, steps_per_level=33, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
        assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (2, pop, 3), np.int64) == want["term"]).all()
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == want["final_pop"]).all()
        G = 1 + (max(edp) if edp is not None else D - 1)
        ev = oracle.eval_layouts(w.lengths, ref["q"], want["final_pop"][pop - 1], ref["R"], s.token_cap, D, edp, s.alpha, s.beta)
        assert (rp.rp_debug_dump(ctx, "W", (ref["R"], G, L, P), np.int32, index=pop - 1) == ev["W"][0]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("spec", [ROW_CASES[0], ROW_CASES[6]], ids=["one_launch", "launch_per_level"])
def test_a_wait_of_the_one_layer_per_lane_kernel_that_runs_out(spec):
    """Its bounded waits, cut short while one chain waits for something that never comes: a time-out
    status, a context that is refused until it is packed again and then anneals as the oracle does."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 23 + N))
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    rp.rp_debug_set_knob(ctx, "WAIT_POLLS", 10000)
    rp.rp_debug_set_knob(ctx, "STALL_ONE_CHAIN", 1)
    for status in (-8, -7):
        with pytest.raises(rp.RpError) as e:
            rp.rp_anneal(ctx, n_levels=3, steps_per_level=20, t0=s.t0, t_ratio=0.6, p_reloc=s.p_reloc, p_guide=s.p_guide)
        assert e.value.status == status
    rp.rp_debug_set_knob(ctx, "STALL_ONE_CHAIN", 0)
    rp.rp_debug_set_knob(ctx, "WAIT_POLLS", 0)
    assert rp.rp_pack_rows(ctx) == (ref["R"], ref["cert"])
    check_anneal(w, ctx, ref, edp, pop, 3, 20, t_ratio=0.6, check_members=1)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("spec", [BARRIER_CASES[0], BARRIER_CASES[2], WARP_CHAIN_CASES[0]],
                         ids=["warp_per_candidate", "cooperative", "warp_per_chain"])
def test_a_wait_that_runs_out_is_reported_and_the_context_survives(spec):
    """One chain waits on a barrier phase that nothing completes, with the poll limit cut to 10^4:
    the wait gives up, the kernels return, rp_anneal reports RP_ERR_TIMEOUT, the calls that make no
    sense afterwards are refused, and after rp_pack_rows the same context anneals again, bit for
    bit as the oracle does.  Nothing traps, faults or spins without a limit."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 11 + N))
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 2 if name.startswith("wc_") else 1)
    rp.rp_debug_set_knob(ctx, "WAIT_POLLS", 10000)
    rp.rp_debug_set_knob(ctx, "STALL_ONE_CHAIN", 1)
    for _ in range(2):                      # the second call finds the arrival counter and the status words clean
        with pytest.raises(rp.RpError) as e:
            rp.rp_anneal(ctx, n_levels=4, steps_per_level=30, t0=s.t0, t_ratio=0.6, p_reloc=s.p_reloc, p_guide=s.p_guide)
        assert e.value.status == -8
        with pytest.raises(rp.RpError) as e:    # the population is gone: annealing on needs rp_pack_rows first
            rp.rp_anneal(ctx, n_levels=1, steps_per_level=5, t0=s.t0, t_ratio=0.6, p_reloc=s.p_reloc, p_guide=s.p_guide)
        assert e.value.status == -7
        assert rp.rp_pack_rows(ctx) == (ref["R"], ref["cert"])
    rp.rp_debug_set_knob(ctx, "STALL_ONE_CHAIN", 0)
    rp.rp_debug_set_knob(ctx, "WAIT_POLLS", 0)
    check_anneal(w, ctx, ref, edp, pop, 4, 30, t_ratio=0.6, check_members=1)
    rp.rp_destroy(ctx)


def test_full_size_properties_large():
    """Large at its full population and sweeps: properties that hold at any size (feasibility
    of every member, cached scores equal to a full rescoring, monotone incumbent, conserved
    rank loads), plus the oracle's evaluation of sampled members."""
    w = make_window("large")
    s = w.spec
    ref = oracle_front(w)
    ctx = load(w, device_inputs=True)
    R = check_front(w, ctx, ref)
    stats = rp.rp_anneal(ctx, n_levels=s.n_levels, steps_per_level=s.steps_per_level, t0=s.t0, t_ratio=s.t_ratio,
                         p_reloc=s.p_reloc, p_guide=s.p_guide)
    assert stats.proposed == s.pop_size * s.sweeps
    K = R * s.dp_width
    popl = rp.rp_debug_dump(ctx, "POPULATION", (s.pop_size, s.n_samples), np.int32)
    assert popl.min() >= 0 and popl.max() < K
    for j in range(0, s.pop_size, 37):
        assert (np.bincount(popl[j], minlength=K) >= 1).all()
        assert (np.bincount(popl[j], weights=w.lengths, minlength=K) <= s.token_cap).all()
    term = rp.rp_debug_dump(ctx, "TRACE_TERM", (s.n_levels, s.pop_size, 3), np.int64)
    fx_pop, _ = rp.rp_eval_population(ctx)
    assert (fx_pop == term[-1]).all()
    inc = [tuple(x) for x in rp.rp_debug_dump(ctx, "TRACE_INCUMBENT", (s.n_levels, 3), np.int64)]
    assert all(b <= a for a, b in zip(inc, inc[1:]))
    for j in (0, 511, 1023):
        ev = oracle.eval_layouts(w.lengths, ref["q"], popl[j], R, s.token_cap, s.dp_width)
        assert tuple(ev["score"][0]) == tuple(term[-1, j])
        Wj = rp.rp_debug_dump(ctx, "W", (R, s.dp_width, s.n_layers, s.ep_width), np.int32, index=j)
        assert (Wj == ev["W"][0]).all()
        assert (Wj.sum(axis=(0, 1)) == ref["G"]).all()          # aggregate invariance
    layout, fx, f64 = rp.rp_best(ctx)
    ev = oracle.eval_layouts(w.lengths, ref["q"], layout, R, s.token_cap, s.dp_width)
    assert tuple(ev["score"][0]) == tuple(fx) == inc[-1]
    seed_score = oracle.eval_layouts(w.lengths, ref["q"], ref["seed"], R, s.token_cap, s.dp_width)["score"][0]
    assert tuple(fx) <= tuple(seed_score)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("case,width", [("medium", 4), ("shared", 8), ("ragged", 1), ("large", 3)])
def test_randomized_seed_population(case, width):
    """Algorithm 2's trial loop: every member's seed layout, which trials were dropped, the scores
    of the seeded population and the annealing that starts from it, all against the oracle."""
    edp, min_rows, pop = None, 0, 48
    if case == "medium":
        w = make_window("medium")
    elif case == "large":
        w = make_window("large")
    elif case == "shared":
        w = make_window(custom_spec("seeds_shared", 96, 5, 16, 2, 4096, 4, 4, pop, 400, data_seed=5))
        edp, min_rows = [0, 0, 1, 1], 3
    else:
        w = make_window(custom_spec("seeds_ragged", 77, 3, 12, 2, 3000, 3, 3, pop, 400, data_seed=6))
        min_rows = 4
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, s.dp_width, pop, width, s.anneal_seed)
    own = rp.rp_seed_population(ctx, width)
    assert own == int(ok.sum())
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == lays).all()
    ev = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
    fx, _ = rp.rp_eval_population(ctx)
    assert (fx == ev["score"]).all()
    best = min(range(pop), key=lambda j: (tuple(ev["score"][j]), j))
    layout, bfx, _ = rp.rp_best(ctx)
    assert (layout == lays[best]).all() and tuple(bfx) == tuple(ev["score"][best])
    check_anneal(w, ctx, ref, edp, pop, 4, 40, t_ratio=0.5, check_members=2, init=lays)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("case,width", [("shared", 1), ("shared", 4), ("interleaved", 3), ("one_shard", 8),
                                        ("identity", 4), ("medium", 4), ("no_trials", 2)])
def test_edp_aware_pairing(case, width):
    """Algorithm 2's pairing operator on a randomized seed population: every member's re-paired
    layout, the scores, the incumbent and the annealing that starts from it, against the oracle."""
    pop, edp, min_rows = 40, None, 3
    if case == "medium":
        w = make_window("medium")
        min_rows = 0
    elif case in ("shared", "no_trials"):
        w = make_window(custom_spec("pair_shared", 96, 5, 16, 2, 4096, 4, 4, pop, 400, data_seed=15))
        edp = [0, 0, 1, 1]
    elif case == "interleaved":
        w = make_window(custom_spec("pair_inter", 120, 7, 24, 3, 4096, 6, 6, pop, 400, data_seed=16))
        edp, min_rows = [0, 1, 2, 0, 1, 2], 2
    elif case == "one_shard":
        w = make_window(custom_spec("pair_one", 64, 2, 8, 1, 2048, 4, 8, pop, 400, data_seed=17))
        edp = [0, 0, 0, 0]
    else:
        w = make_window(custom_spec("pair_ident", 77, 3, 12, 2, 3000, 3, 3, pop, 400, data_seed=18))
        min_rows = 4
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    if case == "no_trials":                 # straight on the length-only seed: the x_paired candidates
        lays = np.tile(ref["seed"], (pop, 1)).astype(np.int32)
    else:
        lays, _ = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, s.dp_width, pop, 4, s.anneal_seed)
        rp.rp_seed_population(ctx, 4)
    want = oracle.edp_pair(ref["q"], lays, ref["R"], s.dp_width, width, s.anneal_seed, edp)
    changed = rp.rp_pair_population(ctx, width)
    assert changed == int((want != lays).any(axis=1).sum())
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == want).all()
    ev = oracle.eval_layouts(w.lengths, ref["q"], want, ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
    fx, _ = rp.rp_eval_population(ctx)
    assert (fx == ev["score"]).all()
    best = min(range(pop), key=lambda j: (tuple(ev["score"][j]), j))
    layout, bfx, _ = rp.rp_best(ctx)
    assert (layout == want[best]).all() and tuple(bfx) == tuple(ev["score"][best])
    check_anneal(w, ctx, ref, edp, pop, 3, 40, t_ratio=0.5, check_members=2, init=want)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("case,eta", [("shared", 1 << 16), ("shared", 0), ("interleaved", 1 << 18),
                                      ("identity", 1 << 16), ("medium", 1 << 14), ("copies", 1 << 16)])
def test_canonical_map_and_quality_diversity_selection(case, eta):
    """Algorithm 2's last lines over a seeded and paired population: which members are one plan,
    the order the selection takes the distinct ones in, the plan distances, the new population,
    its scores, the incumbent and the annealing that starts from it, against the oracle."""
    pop, edp, min_rows, n_proj = 40, None, 3, 6
    if case == "medium":
        w = make_window("medium")
        min_rows = 0
    elif case in ("shared", "copies"):
        w = make_window(custom_spec("sel_shared", 96, 5, 16, 2, 4096, 4, 4, pop, 400, data_seed=25))
        edp = [0, 0, 1, 1]
    elif case == "interleaved":
        w = make_window(custom_spec("sel_inter", 120, 7, 24, 3, 4096, 6, 6, pop, 400, data_seed=26))
        edp, min_rows = [0, 1, 2, 0, 1, 2], 2
    else:
        w = make_window(custom_spec("sel_ident", 77, 3, 12, 2, 3000, 3, 3, pop, 400, data_seed=28))
        min_rows = 4
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    if case == "copies":            # no trials: every member is the length-only seed, re-paired with width 1 -> few classes
        lays = np.tile(ref["seed"], (pop, 1)).astype(np.int32)
        width = 2
    else:
        lays, _ = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, s.dp_width, pop, 4, s.anneal_seed)
        rp.rp_seed_population(ctx, 4)
        width = 3
    lays = oracle.edp_pair(ref["q"], lays, ref["R"], s.dp_width, width, s.anneal_seed, edp)
    rp.rp_pair_population(ctx, width)
    sc = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)["score"]
    want = oracle.select_population(w.lengths, ref["q"], lays, sc, ref["R"], s.token_cap, s.dp_width, s.top_k, n_proj, eta,
                                    s.anneal_seed, edp, want_dist=True)
    nd, order = rp.rp_select_population(ctx, n_proj, eta)
    assert nd == want["n_distinct"]
    if case == "copies":
        assert nd < pop
    assert (order == want["order"]).all()
    got = rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32)
    assert (got == want["layouts"]).all()
    dist = rp.rp_debug_dump(ctx, "SELECT_DIST", (pop, pop), np.int64)
    reps = sorted(set(order[:nd].tolist()))
    assert (dist[np.ix_(reps, reps)] == want["dist"][np.ix_(reps, reps)]).all()
    ev = oracle.eval_layouts(w.lengths, ref["q"], want["layouts"], ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
    fx, _ = rp.rp_eval_population(ctx)
    assert (fx == ev["score"]).all()
    layout, bfx, _ = rp.rp_best(ctx)
    assert (layout == want["layouts"][0]).all() and tuple(bfx) == tuple(ev["score"][0])     # the winner leads
    check_anneal(w, ctx, ref, edp, pop, 3, 40, t_ratio=0.5, check_members=2, init=want["layouts"])
    rp.rp_destroy(ctx)


def oracle_init_population(w, ref, edp, M, pop, width, n_proj, eta):
    """Algorithm 2 over M candidates, composed from the oracle's stages: x_length, x_paired, M - 2
    trials (shuffle -> best fit -> pairing), CanonicalMap + QualityDiversitySelect, cyclic fill."""
    s = w.spec
    R, D = ref["R"], s.dp_width
    lays, _ = oracle.seed_trials(w.lengths, ref["seed"], R, s.token_cap, D, M, width, s.anneal_seed)
    lays[1] = ref["seed"]                                  # candidate 1 starts as the length-only seed too
    cand = oracle.edp_pair(ref["q"], lays, R, D, width, s.anneal_seed, edp)
    score = lambda l: oracle.eval_layouts(w.lengths, ref["q"], l, R, s.token_cap, D, edp, s.alpha, s.beta)["score"]
    if not tuple(score(cand[1])[0]) < tuple(score(ref["seed"])[0]):
        cand[1] = ref["seed"]                              # x_paired = min_Score{x_length, pairing of x_length}
    sel = oracle.select_population(w.lengths, ref["q"], cand, score(cand), R, s.token_cap, D, s.top_k, n_proj, eta,
                                   s.anneal_seed, edp)
    nd = sel["n_distinct"]
    picked = np.array([sel["order"][m % nd] for m in range(pop)], np.int32)
    return nd, picked, cand[picked]


@pytest.mark.parametrize("case,M,pop", [("shared", 60, 24), ("shared", 10, 24), ("interleaved", 33, 33), ("medium", 80, 48),
                                        ("identity", 2, 5), ("copies", 40, 16), ("slices", 12, 40), ("slices_shared", 9, 30)])
def test_algorithm_2_as_one_call(case, M, pop):
    """rp_init_population against the composition of the oracle's stages: how many candidates are
    distinct, which candidate every member is, the members' layouts and scores, the incumbent, and
    the annealing that starts from them; with fewer, as many and more candidates than members."""
    edp, min_rows, width, n_proj, eta = None, 3, 3, 6, 1 << 16
    if case == "medium":
        w = make_window("medium")
        min_rows = 0
    elif case in ("shared", "copies"):
        w = make_window(custom_spec("a2_shared", 96, 5, 16, 2, 4096, 4, 4, pop, 400, data_seed=45))
        edp = [0, 0, 1, 1]
        if case == "copies":
            width = 1                                       # no randomness: few distinct candidates
    elif case == "interleaved":
        w = make_window(custom_spec("a2_inter", 120, 7, 24, 3, 4096, 6, 6, pop, 400, data_seed=46))
        edp, min_rows = [0, 1, 2, 0, 1, 2], 2
    elif case in ("slices", "slices_shared"):
        # rank loads in the slice pool, fewer candidates than members: the repeated members share
        # their original's slices until they rewrite them
        w = make_window(custom_spec("a2_slices", 120, 20, 32, 2, 4096, 4, 32, pop, 400, data_seed=47))
        edp = [0, 1, 1, 0] if case == "slices_shared" else None
    else:
        w = make_window(custom_spec("a2_ident", 77, 3, 12, 2, 3000, 3, 3, pop, 400, data_seed=48))
        min_rows = 4
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    nd_want, picked_want, lays_want = oracle_init_population(w, ref, edp, M, pop, width, n_proj, eta)
    nd, picked = rp.rp_init_population(ctx, M, width, n_proj, eta)
    assert nd == nd_want and (picked == picked_want).all()
    if case == "copies":
        assert nd < M
    got = rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32)
    assert (got == lays_want).all()
    ev = oracle.eval_layouts(w.lengths, ref["q"], lays_want, ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
    fx, _ = rp.rp_eval_population(ctx)
    assert (fx == ev["score"]).all()
    best = min(range(pop), key=lambda j: (tuple(ev["score"][j]), j))
    layout, bfx, _ = rp.rp_best(ctx)
    assert (layout == lays_want[best]).all() and tuple(bfx) == tuple(ev["score"][best])
    check_anneal(w, ctx, ref, edp, pop, 3, 40, t_ratio=0.5, check_members=2, init=lays_want)
    rp.rp_destroy(ctx)


def test_fuzz_random_small_windows():
    """Random shapes and search parameters (rank counts 1..48 including non powers of two, shared
    and interleaved shards, swap-only and relocation-only proposals, unguided and fully guided,
    one to four attention stages, hot and cold schedules): every trajectory against the oracle."""
    rng = np.random.default_rng(2024)
    for trial in range(24):
        P = int(rng.choice([1, 2, 3, 4, 6, 8, 16, 24, 32, 48]))
        H = int(rng.choice([1, 2, 3]))
        E = P * H
        L = int(rng.integers(1, 7))
        D = int(rng.choice([1, 2, 3, 4, 6]))
        N = int(rng.integers(max(12, 4 * D), 160))
        k = int(rng.choice([1, 2, 4]))
        C = int(rng.choice([512, 3000, 8192]))
        G = int(rng.integers(1, D + 1))
        edp = None if G == D else sorted(int(x) for x in np.concatenate([np.arange(G), rng.integers(0, G, D - G)]))
        if edp is not None and trial % 2:
            edp = [int(x) for x in rng.permutation(edp)]
        S = int(rng.integers(1, 5))
        alpha = tuple(float(x) for x in np.round(rng.uniform(0, 3, S) * 256) / 256)
        beta = tuple(float(x) for x in np.round(rng.uniform(0, 3, S) * 256) / 256)
        pop = int(rng.choice([1, 2, 5, 9, 33]))
        spec = custom_spec(f"fuzz{trial}", N, L, E, k, C, D, P, pop, 0, data_seed=1000 + trial, alpha=alpha, beta=beta,
                           p_reloc=float(rng.choice([0.0, 0.25, 0.6, 1.0])), p_guide=float(rng.choice([0.0, 0.5, 0.8, 1.0])),
                           t0=float(rng.choice([1e-5, 1e-3, 5e-2])), anneal_seed=int(rng.integers(0, 2 ** 62)))
        w = make_window(spec)
        min_rows = int(rng.integers(1, 4))
        ref = oracle_front(w, edp, min_rows)
        if ref["R"] == 0:
            continue
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        check_front(w, ctx, ref)
        levels, steps = int(rng.integers(1, 5)), int(rng.choice([1, 7, 33, 130]))
        check_anneal(w, ctx, ref, edp, pop, levels, steps, t_ratio=float(rng.choice([0.3, 0.7, 1.0])), check_members=1)
        rp.rp_destroy(ctx)


def test_fuzz_warp_per_chain_kernel():
    """Random windows whose rank loads live in the slice pool (L*P of 600 to 2000 with 4 to 64
    ranks), random shard maps, attention stages, proposal mixes and schedules, on the
    warp-per-chain kernel: every trajectory against the oracle."""
    rng = np.random.default_rng(77)
    for trial in range(12):
        P = int(rng.choice([4, 8, 16, 32, 64]))
        L = int(rng.integers(600 // P + 1, 2000 // P + 1))
        H = int(rng.choice([1, 2]))
        E = P * H
        D = int(rng.choice([1, 2, 3, 4, 6]))
        N = int(rng.integers(max(16, 4 * D), 140))
        k = int(rng.choice([1, 2, 4]))
        C = int(rng.choice([3000, 8192]))
        G = int(rng.integers(1, D + 1))
        edp = None if G == D else [int(x) for x in rng.permutation(np.concatenate([np.arange(G), rng.integers(0, G, D - G)]))]
        S = int(rng.integers(1, 4))
        alpha = tuple(float(x) for x in np.round(rng.uniform(0, 3, S) * 256) / 256)
        beta = tuple(float(x) for x in np.round(rng.uniform(0, 3, S) * 256) / 256)
        pop = int(rng.choice([1, 3, 9, 40]))
        spec = custom_spec(f"wfuzz{trial}", N, L, E, k, C, D, P, pop, 0, data_seed=3000 + trial, alpha=alpha, beta=beta,
                           p_reloc=float(rng.choice([0.0, 0.25, 0.6, 1.0])), p_guide=float(rng.choice([0.0, 0.5, 0.8, 1.0])),
                           t0=float(rng.choice([1e-5, 1e-3, 5e-2])), anneal_seed=int(rng.integers(0, 2 ** 62)))
        w = make_window(spec)
        min_rows = int(rng.integers(1, 4))
        ref = oracle_front(w, edp, min_rows)
        if ref["R"] == 0:
            continue
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 2)
        check_front(w, ctx, ref)
        levels, steps = int(rng.integers(1, 5)), int(rng.choice([1, 7, 33, 70]))
        _, stats = check_anneal(w, ctx, ref, edp, pop, levels, steps, t_ratio=float(rng.choice([0.3, 0.7, 1.0])), check_members=1)
        assert stats.kernel_launches == levels * 4
        rp.rp_destroy(ctx)


def test_windows_planned_at_once_on_separate_streams():
    """Four different windows (two with more layers or ranks than stay on chip, one that does, one of
    240 cells) planned, and their candidate stages run, at the same
    time by four host threads, each on its own stream and context, several plans each: every
    plan equals the oracle's, so nothing process-wide (shared-memory limits of the kernels, memory
    pools, launch counters) is upset by another context."""
    import threading
    import torch
    cases = [("conc_a", 90, 40, 32, 2, 4096, 4, 32, None, 3, 37),        # L*P = 1280
             ("conc_b", 120, 20, 32, 2, 4096, 4, 32, [0, 1, 1, 0], 3, 25),
             ("conc_c", 96, 5, 16, 2, 4096, 4, 4, None, 3, 40),
             ("conc_d", 300, 6, 16, 2, 4096, 16, 4, None, 15, 20)]        # 240 cells: larger candidate stages than the others'
    jobs = []
    for name, N, L, E, k, C, D, P, edp, min_rows, pop in cases:
        w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 19 + N))
        s = w.spec
        ref = oracle_front(w, edp, min_rows)
        want = oracle.anneal(w.lengths, ref["q"], np.tile(ref["seed"], (pop, 1)), ref["R"], s.token_cap, D, n_levels=6, steps=40,
                             t0=s.t0, t_ratio=0.6, p_reloc=s.p_reloc, p_guide=s.p_guide, seed=s.anneal_seed, edp_of_dp=edp,
                             alpha=s.alpha, beta=s.beta)
        cand = oracle_init_population(w, ref, edp, 12, pop, 4, 8, 1 << 16)
        jobs.append((w, edp, min_rows, pop, want, cand))
    errors = []

    def worker(job):
        try:
            w, edp, min_rows, pop, want, cand = job
            s = w.spec
            stream = torch.cuda.Stream()
            for _ in range(6):
                ctx = rp.rp_window_load(w.lengths, w.demand, top_k=s.top_k, token_cap=s.token_cap, dp_width=s.dp_width,
                                        ep_width=s.ep_width, pop_size=pop, edp_of_dp=edp, alpha=s.alpha, beta=s.beta,
                                        min_rows=min_rows, seed=s.anneal_seed, stream=stream)
                rp.rp_place_experts(ctx)
                rp.rp_pack_rows(ctx)
                st = rp.rp_anneal(ctx, n_levels=6, steps_per_level=40, t0=s.t0, t_ratio=0.6, p_reloc=s.p_reloc, p_guide=s.p_guide)
                layout, fx, _ = rp.rp_best(ctx)
                assert [st.proposed, st.feasible, st.accepted, st.improved] == want["counters"].tolist()
                assert (layout == want["best_layout"]).all() and (fx == want["best_score"]).all()
                assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == want["final_pop"]).all()
                rp.rp_pack_rows(ctx)                     # and the candidate stages
                nd, picked = rp.rp_init_population(ctx, 12, 4, 8, 1 << 16)
                assert nd == cand[0] and (picked == cand[1]).all()
                assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == cand[2]).all()
                rp.rp_destroy(ctx)
        except Exception as e:          # reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=worker, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


@pytest.mark.parametrize("name,pop", [("tiny", 8), ("medium", 256), ("medium", 100), ("large", 300)])
def test_annealing_without_the_inspection_hook(name, pop):
    """The per-level traces are an inspection hook: counters, final population, incumbent and
    scores without them must be those of the traced run (itself checked against the oracle
    elsewhere), over many levels, and again when rp_anneal continues from the population."""
    w = make_window(name)
    s = w.spec
    outs = []
    for trace in (True, False):
        ctx = load(w, pop=pop)
        rp.rp_debug_set_trace(ctx, trace)
        rp.rp_place_experts(ctx)
        rp.rp_pack_rows(ctx)
        res = []
        for levels, steps in ((12, 25), (5, 40)):
            st = rp.rp_anneal(ctx, n_levels=levels, steps_per_level=steps, t0=s.t0, t_ratio=0.7, p_reloc=s.p_reloc, p_guide=s.p_guide)
            layout, fx, _ = rp.rp_best(ctx)
            res.append(([st.proposed, st.feasible, st.accepted, st.improved], layout.copy(), fx.copy(),
                        rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32),
                        rp.rp_eval_population(ctx)[0]))
        outs.append(res)
        rp.rp_destroy(ctx)
    for a, b in zip(*outs):
        assert a[0] == b[0]
        for x, y in zip(a[1:], b[1:]):
            assert (x == y).all()


def test_repeated_front_end_calls_recompute():
    """rp_window_load already queues placement and packing; a second rp_place_experts or
    rp_pack_rows computes them again itself, and rp_best without a preceding rp_anneal validates
    on its own: same results on every route."""
    w = make_window(custom_spec("twice", 96, 5, 16, 2, 4096, 4, 4, 12, 400, data_seed=31))
    edp = [0, 0, 1, 1]
    ref = oracle_front(w, edp, 3)
    ctx = load(w, pop=12, edp=edp, min_rows=3)
    pi1, load1 = rp.rp_place_experts(ctx)
    pi2, load2 = rp.rp_place_experts(ctx)
    assert (pi1 == pi2).all() and (load1 == load2).all() and (pi1 == ref["pi"]).all()
    r1 = rp.rp_pack_rows(ctx)
    lay1, fx1, _ = rp.rp_best(ctx)                  # no rp_anneal yet: the seed, validated here
    r2 = rp.rp_pack_rows(ctx)
    lay2, fx2, _ = rp.rp_best(ctx)
    assert r1 == r2 and r1[0] == ref["R"]
    assert (lay1 == lay2).all() and (lay1 == ref["seed"]).all() and tuple(fx1) == tuple(fx2)
    check_eval(w, ctx, ref, edp)
    check_anneal(w, ctx, ref, edp, 12, 3, 40, t_ratio=0.5)
    lay3, fx3, _ = rp.rp_best(ctx)                  # handed over by rp_anneal
    lay4, fx4, _ = rp.rp_best(ctx)
    assert (lay3 == lay4).all() and tuple(fx3) == tuple(fx4)
    rp.rp_destroy(ctx)


def test_fuzz_seeding_stages():
    """Random shapes (one to six DP slots, one to all shards, 1..48 ranks, populations of 1..33,
    choice widths 1..32, one to nine projections, zero to large eta): trial loop, pairing and
    selection against the oracle, stage by stage."""
    rng = np.random.default_rng(77)
    done = 0
    for trial in range(16):
        P = int(rng.choice([1, 2, 3, 4, 8, 16, 48]))
        E = P * int(rng.choice([1, 2]))
        L = int(rng.integers(1, 6))
        D = int(rng.choice([1, 2, 3, 4, 6]))
        N = int(rng.integers(max(12, 4 * D), 140))
        k = int(rng.choice([1, 2, 4]))
        C = int(rng.choice([512, 3000, 8192]))
        G = int(rng.integers(1, D + 1))
        edp = None if G == D else [int(x) for x in rng.permutation(np.concatenate([np.arange(G), rng.integers(0, G, D - G)]))]
        pop = int(rng.choice([1, 2, 7, 20, 33]))
        spec = custom_spec(f"seedfuzz{trial}", N, L, E, k, C, D, P, pop, 0, data_seed=3000 + trial,
                           anneal_seed=int(rng.integers(0, 2 ** 62)))
        w = make_window(spec)
        s = w.spec
        min_rows = int(rng.integers(1, 4))
        ref = oracle_front(w, edp, min_rows)
        if ref["R"] == 0:
            continue
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        check_front(w, ctx, ref)
        w1, w2 = int(rng.choice([1, 2, 5, 32])), int(rng.choice([1, 3, 32]))
        n_proj, eta = int(rng.integers(1, 10)), int(rng.choice([0, 1 << 12, 1 << 16, 1 << 24]))
        lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, s.dp_width, pop, w1, s.anneal_seed)
        assert rp.rp_seed_population(ctx, w1) == int(ok.sum())
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == lays).all()
        paired = oracle.edp_pair(ref["q"], lays, ref["R"], s.dp_width, w2, s.anneal_seed, edp)
        assert rp.rp_pair_population(ctx, w2) == int((paired != lays).any(axis=1).sum())
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == paired).all()
        sc = oracle.eval_layouts(w.lengths, ref["q"], paired, ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)["score"]
        want = oracle.select_population(w.lengths, ref["q"], paired, sc, ref["R"], s.token_cap, s.dp_width, s.top_k, n_proj, eta,
                                        s.anneal_seed, edp)
        nd, order = rp.rp_select_population(ctx, n_proj, eta)
        assert nd == want["n_distinct"] and (order == want["order"]).all()
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, s.n_samples), np.int32) == want["layouts"]).all()
        check_anneal(w, ctx, ref, edp, pop, 2, 20, t_ratio=0.5, check_members=1, init=want["layouts"])
        rp.rp_destroy(ctx)
        done += 1
    assert done >= 10


def test_bad_inputs_are_host_side_errors():
    w = make_window("tiny")
    s = w.spec
    kw = dict(top_k=s.top_k, token_cap=s.token_cap, dp_width=s.dp_width, ep_width=s.ep_width, pop_size=4)
    bad = w.demand.copy()
    bad[7, 2, 3] += 1
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths, bad, **kw)
    assert e.value.status == -3
    neg = w.demand.copy()
    neg[3, 0, 0] -= 5
    neg[3, 0, 1] += 5
    if neg[3, 0, 0] < 0:
        with pytest.raises(rp.RpError) as e:
            rp.rp_window_load(w.lengths, neg, **kw)
        assert e.value.status == -3
    long_ = w.lengths.copy()
    long_[0] = s.token_cap + 1
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(long_, w.demand, **kw)
    assert e.value.status == -3
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths, w.demand, **dict(kw, ep_width=3))
    assert e.value.status == -2
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths[:1], w.demand[:1], **kw)
    assert e.value.status == -2
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths, w.demand, edp_of_dp=[0, 2], **kw)      # shard 1 unused
    assert e.value.status == -2
    # rank loads are 32-bit: k * C * (DP slots of one shard) must stay below 2^31; the cap itself below 2^24
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths, w.demand, **dict(kw, top_k=64, token_cap=1 << 24, edp_of_dp=[0, 0]))
    assert e.value.status == -5
    with pytest.raises(rp.RpError) as e:
        rp.rp_window_load(w.lengths, w.demand, **dict(kw, token_cap=(1 << 24) + 1))
    assert e.value.status == -5
    with pytest.raises(rp.RpError) as e:                                     # score range: (2^8*C*L*k + ...) * sum t >= 2^62
        rp.rp_window_load(w.lengths, w.demand, **dict(kw, token_cap=1 << 24, alpha=(1e6,), beta=(0.0,)))
    assert e.value.status == -5
    ctx = rp.rp_window_load(w.lengths, w.demand, **kw)
    with pytest.raises(rp.RpError) as e:
        rp.rp_pack_rows(ctx)                                                 # before rp_place_experts
    assert e.value.status == -7
    rp.rp_place_experts(ctx)
    with pytest.raises(rp.RpError) as e:
        rp.rp_anneal(ctx, n_levels=1, steps_per_level=1, t0=1e-3, t_ratio=0.5, p_reloc=0.2, p_guide=0.8)
    assert e.value.status == -7
    for call in (lambda: rp.rp_seed_population(ctx, 4), lambda: rp.rp_pair_population(ctx, 4),
                 lambda: rp.rp_select_population(ctx, 4, 1 << 16), lambda: rp.rp_init_population(ctx, 8)):
        with pytest.raises(rp.RpError) as e:
            call()                                                           # before rp_pack_rows
        assert e.value.status == -7
    R, _ = rp.rp_pack_rows(ctx)
    for call in (lambda: rp.rp_seed_population(ctx, 0), lambda: rp.rp_pair_population(ctx, 33),
                 lambda: rp.rp_select_population(ctx, 0, 1 << 16), lambda: rp.rp_select_population(ctx, 4, -1),
                 lambda: rp.rp_init_population(ctx, 1), lambda: rp.rp_init_population(ctx, 8, 0),
                 lambda: rp.rp_init_population(ctx, 8, 4, 65), lambda: rp.rp_init_population(ctx, 8, 4, 8, -1)):
        with pytest.raises(rp.RpError) as e:
            call()
        assert e.value.status == -1
    lay = np.zeros((1, s.n_samples), np.int32)
    lay[0, 5] = R * s.dp_width
    with pytest.raises(rp.RpError) as e:
        rp.rp_eval_population(ctx, lay)
    assert e.value.status == -1
    with pytest.raises(rp.RpError) as e:
        rp.rp_anneal(ctx, n_levels=0, steps_per_level=1, t0=1e-3, t_ratio=0.5, p_reloc=0.2, p_guide=0.8)
    assert e.value.status == -1
    rp.rp_anneal(ctx, n_levels=1, steps_per_level=4, t0=1e-3, t_ratio=0.5, p_reloc=0.2, p_guide=0.8)
    with pytest.raises(rp.RpError) as e:
        rp.rp_pair_population(ctx, 4)                                        # the seeding stages end with rp_anneal
    assert e.value.status == -7
    rp.rp_destroy(ctx)
    # infeasible: more DP slots than one-sample cells can fill at this cap is fine, but a window
    # whose samples cannot be split into non-empty cells within the cap is reported, not trapped
    t = np.full(6, 10, np.int32)
    a = np.zeros((6, 1, 2), np.int32)
    a[:, 0, 0] = 10
    ctx = rp.rp_window_load(t, a, top_k=1, token_cap=10, dp_width=4, ep_width=2, pop_size=2)
    rp.rp_place_experts(ctx)
    with pytest.raises(rp.RpError) as e:
        rp.rp_pack_rows(ctx)          # 6 samples of a full cell each need 6 cells; 4 and 8 are the only shapes
    assert e.value.status == -4
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("E,P,N,L", [(128, 32, 70, 5), (256, 16, 37, 9), (384, 4, 33, 2), (1024, 8, 19, 3), (128, 1, 41, 3),
                                     (128, 8, 100, 2), (512, 32, 35, 4), (256, 32, 300, 3), (128, 64, 50, 2),
                                     (128, 32, 301, 32), (128, 4, 296, 32), (256, 16, 297, 48)])
def test_wide_expert_rows_front_end(E, P, N, L):
    """Rows of whole multiples of 128 experts take the 16-byte-load forms of the check + reduce and
    projection kernels (ragged sample counts: the last group of rows is partial; two shapes with 32 layers
    of 128 experts take the sequential-stream form of the check + reduce): aggregate demand,
    placement, rank demand and seed against the oracle, and every kind of bad input is still caught."""
    w = make_window(custom_spec(f"rows{E}", N, L, E, 4, 4096, 2, P, 6, 100, data_seed=E + N))
    s = w.spec
    ref = oracle_front(w, None, 2)
    for device_inputs in (False, True):
        ctx = load(w, pop=6, min_rows=2, device_inputs=device_inputs)
        check_front(w, ctx, ref)
        check_eval(w, ctx, ref, None, n=2)
        rp.rp_destroy(ctx)
    kw = dict(top_k=s.top_k, token_cap=s.token_cap, dp_width=s.dp_width, ep_width=s.ep_width, pop_size=2)
    for i, l, e in ((0, 0, 0), (N - 1, L - 1, E - 1), (N // 2, L // 2, 129 % E)):
        bad = w.demand.copy()
        bad[i, l, e] += 1                                   # row sum off by one
        with pytest.raises(rp.RpError) as err:
            rp.rp_window_load(w.lengths, bad, **kw)
        assert err.value.status == -3
        neg = w.demand.copy()                               # row sum right, one count negative
        neg[i, l, e] -= neg[i, l, e] + 3
        neg[i, l, (e + 5) % E] += w.demand[i, l, e] + 3
        with pytest.raises(rp.RpError) as err:
            rp.rp_window_load(w.lengths, neg, **kw)
        assert err.value.status == -3
        big = w.demand.copy()                               # sums right modulo 2^32, counts far out of range
        big[i, l, e] += 2 ** 30
        big[i, l, (e + 1) % E] += 2 ** 30
        big[i, l, (e + 2) % E] += 2 ** 30
        big[i, l, (e + 3) % E] += 2 ** 30
        with pytest.raises(rp.RpError) as err:
            rp.rp_window_load(w.lengths, big, **kw)
        assert err.value.status == -3
    long_ = w.lengths.copy()
    long_[N - 1] = 0
    with pytest.raises(rp.RpError) as err:
        rp.rp_window_load(long_, w.demand, **kw)
    assert err.value.status == -3


def test_smallest_window_and_empty_moves():
    """N == D, one row, one sample per cell: every proposal is infeasible (same cell, or a
    relocation that would empty a cell, or a swap over the cap) or a legal swap."""
    t = np.array([5, 9, 3, 7], np.int32)
    a = np.zeros((4, 2, 4), np.int32)
    rng = np.random.default_rng(5)
    for i in range(4):
        for l in range(2):
            a[i, l] = rng.multinomial(2 * t[i], [0.1, 0.2, 0.3, 0.4])
    pi, G = oracle.lpt(oracle.aggregate(a), 2)
    q = oracle.project(a, pi, 2)
    R, cert, seed = oracle.pack_ffd(t, 16, 4)
    assert R == 1
    ctx = rp.rp_window_load(t, a, top_k=2, token_cap=16, dp_width=4, ep_width=2, pop_size=3, seed=11)
    rp.rp_debug_set_trace(ctx, True)
    rp.rp_place_experts(ctx)
    assert rp.rp_pack_rows(ctx) == (R, cert)
    want = oracle.anneal(t, q, np.tile(seed, (3, 1)), R, 16, 4, n_levels=4, steps=30, t0=1e-2, t_ratio=0.5,
                         p_reloc=0.3, p_guide=0.8, seed=11)
    stats = rp.rp_anneal(ctx, n_levels=4, steps_per_level=30, t0=1e-2, t_ratio=0.5, p_reloc=0.3, p_guide=0.8)
    assert [stats.proposed, stats.feasible, stats.accepted, stats.improved] == want["counters"].tolist()
    assert (rp.rp_debug_dump(ctx, "TRACE_DIGEST", (4, 3), np.uint64) == want["digest"]).all()
    layout, fx, _ = rp.rp_best(ctx)
    assert (layout == want["best_layout"]).all() and (fx == want["best_score"]).all()
    rp.rp_destroy(ctx)


# Both orders (sort in the packing CTA up to 512 samples and above 32768, counting on the whole GPU between), up to 1024 cells and
# more, keys in shared and global memory, one-token samples that fill a cell by the run.
@pytest.mark.parametrize("N,D,min_rows,cap,longest", [
    (33, 1, 0, 40, 40), (512, 4, 0, 64, 64), (513, 4, 0, 64, 20), (700, 7, 0, 4096, 1), (2100, 4, 256, 64, 40),
    (2100, 5, 205, 64, 40), (2049, 2, 1024, 100, 100), (8193, 8, 120, 64, 4),
    (9000, 8, 0, 4096, 300), (32770, 8, 0, 1 << 20, 4096)])
def test_packing_at_the_edges_of_its_forms(N, D, min_rows, cap, longest):
    rng = np.random.default_rng(N + D)
    t = rng.integers(1, longest + 1, N).astype(np.int32)
    a = np.zeros((N, 1, 2), np.int32)
    a[np.arange(N), 0, rng.integers(0, 2, N)] = t
    R, cert, seed = oracle.pack_ffd(t, cap, D, min_rows)
    ctx = rp.rp_window_load(t, a, top_k=1, token_cap=cap, dp_width=D, ep_width=2, pop_size=2, min_rows=min_rows)
    rp.rp_place_experts(ctx)
    assert rp.rp_pack_rows(ctx) == (R, cert)
    assert (rp.rp_debug_dump(ctx, "SEED_LAYOUT", (N,), np.int32) == seed).all()
    rp.rp_destroy(ctx)


# Cells on both sides of the numbers the sorted keys of a trial are kept for (64, 256, 512 in registers, more in shared memory),
# several and one slot per row-shard beyond one a thread, and pair counts of the distances in 32, 16 and 8 bits, whole and in blocks.
@pytest.mark.parametrize("N,D,min_rows,edp,longest,full", [
    (200, 8, 8, None, 60, 0), (200, 5, 13, [0, 0, 1, 1, 1], 60, 0), (700, 8, 32, [0, 1] * 4, 60, 0), (700, 1, 257, None, 60, 0),
    (1300, 4, 128, [0, 0, 0, 0], 60, 0), (1300, 3, 171, [0, 1, 1], 60, 0), (2300, 4, 300, [0, 0, 1, 1], 60, 0),
    (3150, 8, 20, None, 1, 150), (3240, 10, 25, [0, 1] * 5, 1, 240)])
def test_candidate_stages_at_the_edges_of_their_forms(N, D, min_rows, edp, longest, full):
    rng = np.random.default_rng(N + D)
    cap, pop, L, E, k = 600, 4, 2, 8, 2
    t = rng.integers(1, longest + 1, N).astype(np.int32)
    t[:full] = cap
    a = np.stack([[rng.multinomial(k * int(ti), np.full(E, 1 / E)) for _ in range(L)] for ti in t]).astype(np.int32)
    ref_pi, _ = oracle.lpt(oracle.aggregate(a), 2)
    q = oracle.project(a, ref_pi, 2)
    R, cert, seed = oracle.pack_ffd(t, cap, D, min_rows)
    ctx = rp.rp_window_load(t, a, top_k=k, token_cap=cap, dp_width=D, ep_width=2, pop_size=pop, min_rows=min_rows, edp_of_dp=edp, seed=5)
    rp.rp_debug_set_trace(ctx, True)
    rp.rp_place_experts(ctx)
    assert rp.rp_pack_rows(ctx) == (R, cert)
    lays, ok = oracle.seed_trials(t, seed, R, cap, D, pop, 5, 5)
    assert rp.rp_seed_population(ctx, 5) == int(ok.sum())
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == lays).all()
    pairs = oracle.edp_pair(q, lays, R, D, 4, 5, edp)
    rp.rp_pair_population(ctx, 4)
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == pairs).all()
    sc = oracle.eval_layouts(t, q, pairs, R, cap, D, edp)["score"]
    want = oracle.select_population(t, q, pairs, sc, R, cap, D, k, 9, 1 << 16, 5, edp, want_dist=True)
    nd, order = rp.rp_select_population(ctx, 9, 1 << 16)
    assert nd == want["n_distinct"] and (order == want["order"]).all()
    dist = rp.rp_debug_dump(ctx, "SELECT_DIST", (pop, pop), np.int64)
    reps = sorted(set(order[:nd].tolist()))
    assert (dist[np.ix_(reps, reps)] == want["dist"][np.ix_(reps, reps)]).all()
    rp.rp_destroy(ctx)


# From level to level in one launch: fewer members than CTAs and several per thread, more row-shards than threads and a few, slices
# in one piece and several; the same with the parts as launches of their own.
@pytest.mark.parametrize("N,D,min_rows,edp,pop,levels", [(600, 4, 140, None, 2, 6), (600, 4, 140, None, 37, 5), (60, 2, 2, [0, 0], 1200, 5),
                                                         (48, 2, 3, None, 5003, 3)])
def test_between_two_levels_at_the_edges(N, D, min_rows, edp, pop, levels):
    w = make_window(custom_spec("turn", N, 24, 32, 2, 4096, D, 16, pop, 400, data_seed=N + pop))
    ref = oracle_front(w, edp, min_rows)
    for knob in (0, 1):
        ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
        rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", knob)
        check_front(w, ctx, ref)
        if knob == 0:
            assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row"
        _, stats = check_anneal(w, ctx, ref, edp, pop, levels, 20, t_ratio=0.5, check_members=2)
        if knob == 0:
            assert stats.kernel_launches == 2 * levels + 2
        rp.rp_destroy(ctx)


def one_heavy_expert(name, t, L, E, k, C, D, P, pop, share, **kw):
    """A window of given lengths whose first expert takes `share` of every sample's routing."""
    s = custom_spec(name, len(t), L, E, k, C, D, P, pop, 0, **kw)
    a = np.zeros((len(t), L, E), np.int64)
    rng = np.random.default_rng(len(t) + L)
    total = k * t.astype(np.int64)
    a[:, :, 0] = (share * total).astype(np.int64)[:, None]
    rest = (total - a[:, 0, 0])[:, None, None] // (E + 3) + rng.integers(0, 50, (len(t), L, E - 1))
    a[:, :, 1:] = rest
    a[:, :, E - 1] += total[:, None] - a.sum(axis=2)
    assert (a >= 0).all() and (a.sum(axis=2) == total[:, None]).all()
    return Window(s, t.astype(np.int32), np.ascontiguousarray(a.astype(np.int32)))


UNEVEN = [0] * 17 + list(range(1, 16))


@pytest.mark.parametrize("n", [5, 1300])
@pytest.mark.parametrize("case", ["uneven_shards", "overfull_cells"])
def test_busiest_loads_that_add_up_beyond_32_bits(case, n):
    """A row-shard's busiest loads over all layers pass 32 bits: a shard with 17 of 32 slots where the even share is two,
    and layouts that put everything into one cell; both scoring forms."""
    rng = np.random.default_rng(n)
    if case == "uneven_shards":
        w = one_heavy_expert(case, rng.integers(300_000, 340_000, 40), 120, 4, 8, 1 << 20, 32, 4, 2, 0.55)
        edp, slots = UNEVEN, 17
    else:
        w = one_heavy_expert(case, rng.integers(300_000, 500_000, 64), 100, 8, 2, 1 << 20, 4, 4, 2, 0.9)
        edp, slots = None, 1
    s = w.spec
    ref = oracle_front(w, edp)
    ctx = load(w, pop=2, edp=edp)
    check_front(w, ctx, ref)
    K = ref["R"] * s.dp_width
    lays = rng.integers(0, K, (n, s.n_samples)).astype(np.int32)
    lays[1::2] = rng.integers(0, slots, (n // 2, s.n_samples))       # all of it in the first shard of the first row
    fx, _ = rp.rp_eval_population(ctx, lays)
    some = np.r_[0:5, n - 3:n]
    ev = oracle.eval_layouts(w.lengths, ref["q"], lays[some], ref["R"], s.token_cap, s.dp_width, edp, s.alpha, s.beta)
    assert ev["W"].max(axis=-1).sum(axis=-1, dtype=np.int64).max() >= 1 << 32
    assert (fx[some] == ev["score"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("kernel", [0, 1, 2])
def test_annealing_of_a_shard_with_most_of_the_slots(kernel):
    """The same map under annealing: rank loads and slacks of the large shard beyond 2^31 on every chain kernel."""
    rng = np.random.default_rng(3)
    w = one_heavy_expert("uneven_anneal", rng.integers(250_000, 420_000, 40), 120, 4, 8, 1 << 20, 32, 4, 12, 0.9)
    s = w.spec
    ref = oracle_front(w, UNEVEN)
    ev = oracle.eval_layouts(w.lengths, ref["q"], ref["seed"], ref["R"], s.token_cap, s.dp_width, UNEVEN, s.alpha, s.beta)
    assert ev["W"].max(axis=-1).sum(axis=-1, dtype=np.int64).max() >= 1 << 32
    ctx = load(w, pop=12, edp=UNEVEN)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", kernel)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, UNEVEN, 12, 4, 60, t_ratio=0.6)
    assert stats.accepted > 0
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("stage", ["selection", "packing"])
def test_kernels_with_window_sized_shared_memory_on_two_threads(stage):
    """Two host threads, each with a window of its own size, the same stage over and over: the shared-memory limit of a
    kernel that asks for as much as its window needs must not follow the other thread's window."""
    import threading
    import torch

    def call(ctx):
        if stage == "packing":
            return np.array(rp.rp_pack_rows(ctx))
        nd, order = rp.rp_select_population(ctx)
        return np.r_[nd, order]

    jobs = []
    for N, D, min_rows in ((500, 16, 15), (220, 10, 10)) if stage == "selection" else ((5000, 8, 0), (3000, 8, 0)):
        w = make_window(custom_spec("two_threads", N, 2, 8, 2, 4096, D, 4, 6, 0, data_seed=N))
        s = w.spec
        pair = []
        for _ in range(2):                       # one for the reference run, one for the thread
            ctx = rp.rp_window_load(torch.from_numpy(w.lengths).cuda(), torch.from_numpy(w.demand).cuda(), top_k=s.top_k,
                                    token_cap=s.token_cap, dp_width=D, ep_width=4, pop_size=6, min_rows=min_rows, seed=3,
                                    stream=torch.cuda.Stream())
            rp.rp_place_experts(ctx)
            rp.rp_pack_rows(ctx)
            if stage == "selection":
                rp.rp_seed_population(ctx, 4)
            pair.append(ctx)
        jobs.append((pair[1], [call(pair[0]) for _ in range(5)]))
    errors = []

    def worker(ctx, want):
        try:
            for n in range(3000):
                got = call(ctx)
                if n < len(want):
                    assert (got == want[n]).all()
        except Exception as e:          # reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=worker, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


SHARD31 = list(range(31)) + [0]
PERM32 = [(d + 1) % 32 for d in range(32)]


@pytest.mark.parametrize("N,L,P,min_rows,edp,S,row", [
    (2400, 24, 32, 72, SHARD31, 2, False),      # 235 KB a chain with one layer per lane: more than an SM has
    (1300, 24, 16, 36, PERM32, 8, False),       # 241 KB
    (1300, 24, 16, 32, PERM32, 2, True), (1300, 24, 16, 36, PERM32, 2, False),      # two chains to an SM, and no longer two
    (700, 24, 16, 16, PERM32, 4, True), (700, 24, 16, 17, PERM32, 4, False)])       # three
def test_windows_whose_chains_do_not_fit_one_layer_per_lane(N, L, P, min_rows, edp, S, row):
    """Many cells under a shard map that is not the identity: the one-layer-per-lane kernel is chosen by the shared memory
    of its chain, and what it does not take is annealed by the kernels for such windows."""
    w = make_window(custom_spec("big_maps", N, L, P, 2, 8192, 32, P, 5, 0, data_seed=N + S, alpha=(1.0,) * S,
                                beta=tuple(x / S for x in range(S))))
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, edp=edp, min_rows=min_rows)
    check_front(w, ctx, ref)
    assert (rp.rp_debug_chain_kernel(ctx) == "k_anneal_row") == row
    _, stats = check_anneal(w, ctx, ref, edp, 5, 3, 50, t_ratio=0.6, check_members=1)
    assert stats.accepted > 0
    rp.rp_destroy(ctx)


def test_a_call_that_fails_for_memory_leaves_the_population_as_it_is():
    """51000 members whose rank loads fit the GPU as compressed rows (6 GB) and not in full form (200 GB): a kernel that
    needs the full form is refused, before any level has run and after some, and the next call goes on from where the
    population stands, as in a context that was never asked for more."""
    import torch
    N, L, P, D, R, pop = 200, 32, 128, 8, 15, 51000
    rng = np.random.default_rng(8)
    t = rng.integers(20, 200, N).astype(np.int32)
    p = np.full((L, P), 0.35 / (P - 3))
    for l in range(L):
        p[l, rng.choice(P, 3, replace=False)] = (0.3, 0.2, 0.15)
    a = rng.multinomial((20 * t.astype(np.int64))[:, None], p).astype(np.int32)
    runs = []
    for refused in (True, False):
        ctx = rp.rp_window_load(t, a, top_k=20, token_cap=2048, dp_width=D, ep_width=P, pop_size=pop, min_rows=R, seed=4)
        rp.rp_place_experts(ctx)
        assert rp.rp_pack_rows(ctx)[0] == R
        out = []
        for levels in (2, 3):
            if refused:
                rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 1)
                with pytest.raises(rp.RpError) as err:
                    rp.rp_anneal(ctx, n_levels=2, steps_per_level=5, t0=1e-3, t_ratio=0.5, p_reloc=0.2, p_guide=0.8)
                assert err.value.status == -6
                rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 0)
                torch.zeros(1, device="cuda").add_(1)            # the failure does not turn up in the caller's next launch
            st = rp.rp_anneal(ctx, n_levels=levels, steps_per_level=8, t0=1e-3, t_ratio=0.5, p_reloc=0.2, p_guide=0.8)
            assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row" and st.accepted > 0
            out += [np.array([st.proposed, st.feasible, st.accepted, st.improved]), rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32),
                    *rp.rp_best(ctx)]
        runs.append(out)
        rp.rp_destroy(ctx)
        rp.rp_release_cached_memory()
    for x, y in zip(*runs):
        assert (x == y).all()


@pytest.mark.parametrize("spec,when", [(ROW_CASES[0], "before"), (ROW_CASES[3], "before"), (ROW_CASES[0], "after"), (ROW_CASES[3], "after"),
                                       (ROW_CASES[4], "after"), (ROW_CASES[5], "resumed"), (ROW_CASES[4], "resumed"),
                                       (ROW_CASES[6], "after"), (ROW_CASES[7], "resumed")])
def test_launches_that_need_more_sms_than_are_free(spec, when):
    """Launches whose CTAs wait for one another where only three SMs can hold them: known when the population is built
    (more chains per CTA, or another form), found out at the launch, and found out by a later call."""
    name, N, L, E, k, C, D, P, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, k, C, D, P, pop, 400, data_seed=len(name) * 29 + N))
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    if when == "before":
        rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 3)
    check_front(w, ctx, ref)
    if when == "after":
        rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 3)
    want, stats = check_anneal(w, ctx, ref, edp, pop, 4, 40, t_ratio=0.5, check_members=2)
    assert stats.accepted > 0
    if when == "before":
        assert (stats.kernel_launches == 1) == (pop <= 24)
    elif when == "after":
        assert stats.kernel_launches >= 4
    rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 3)
    want = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, D, n_levels=3, steps=33, t0=1e-4,
                         t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed, edp_of_dp=edp, alpha=s.alpha,
                         beta=s.beta, n_threads=8)
    stats = rp.rp_anneal(ctx, n_levels=3, steps_per_level=33, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
    assert stats.kernel_launches >= 3 or pop <= 24
    assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (3, pop, 3), np.int64) == want["term"]).all()
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == want["final_pop"]).all()
    G = 1 + (max(edp) if edp is not None else D - 1)
    ev = oracle.eval_layouts(w.lengths, ref["q"], want["final_pop"][pop - 1], ref["R"], s.token_cap, D, edp, s.alpha, s.beta)
    assert (rp.rp_debug_dump(ctx, "W", (ref["R"], G, L, P), np.int32, index=pop - 1) == ev["W"][0]).all()
    layout, fx, _ = rp.rp_best(ctx)
    assert (layout == want["best_layout"]).all() and (fx == want["best_score"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("P,kernel", [(3, 0), (3, 1), (16, 2)])
def test_more_members_than_one_scoring_launch_takes(P, kernel):
    """17000 members with seeds of their own, more than a launch of the scoring kernels takes: every member's rank loads
    are its own, and annealing goes on from them."""
    pop, N, L, D, min_rows = 17000, 24, 40, 2, 3
    w = make_window(custom_spec("many_members", N, L, P, 1, 2048, D, P, pop, 0, data_seed=P))
    s = w.spec
    ref = oracle_front(w, None, min_rows)
    ctx = load(w, min_rows=min_rows)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", kernel)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, D, pop, 5, s.anneal_seed)
    assert rp.rp_seed_population(ctx, 5) == int(ok.sum())
    for j in (0, 16383, 16384, pop - 1):
        ev = oracle.eval_layouts(w.lengths, ref["q"], lays[j], ref["R"], s.token_cap, D, None, s.alpha, s.beta)
        assert (rp.rp_debug_dump(ctx, "W", (ref["R"], D, L, P), np.int32, index=j) == ev["W"][0]).all()
    check_anneal(w, ctx, ref, None, pop, 2, 12, t_ratio=0.6, init=lays)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("n", [1, 3, 150, 2500, 4000, 16400])
def test_a_refused_layout_leaves_the_outputs_alone(n):
    """One bad cell id among n layouts: RP_ERR_ARG, and neither device nor host outputs are written; good layouts are
    scored by the next call (few and many layouts, more than the pinned block and more than one launch holds)."""
    import torch
    w = make_window(custom_spec("refused", 40, 3, 8, 2, 4096, 4, 4, 2, 0, data_seed=n))
    s = w.spec
    ref = oracle_front(w, None, 2)
    ctx = load(w, min_rows=2)
    check_front(w, ctx, ref)
    rng = np.random.default_rng(n)
    good = rng.integers(0, ref["R"] * 4, (n, 40)).astype(np.int32)
    want = oracle.eval_layouts(w.lengths, ref["q"], good[-2:], ref["R"], s.token_cap, 4, None, s.alpha, s.beta)["score"]
    for value in (-1, ref["R"] * 4):
        lays = good.copy()
        lays[rng.integers(0, n), rng.integers(0, 40)] = value
        for dev in (True, False):
            fx, f64 = torch.full((n, 3), -7, dtype=torch.int64), torch.full((n, 3), -7.0, dtype=torch.float64)
            if dev:
                fx, f64 = fx.cuda(), f64.cuda()
            for out64 in (f64, None, np.full((n, 3), -7.0)):
                with pytest.raises(rp.RpError) as e:
                    rp._check(rp.lib().rp_eval_population(ctx.handle, rp._ptr(lays), n, rp._ptr(fx), rp._ptr(out64)), "eval")
                assert e.value.status == -1
                assert bool((fx == -7).all()) and (out64 is None or bool((out64 == -7).all()))
            rp.rp_eval_population(ctx, good, fx, f64)
            assert (fx[-2:].cpu().numpy() == want).all()
            np.testing.assert_allclose(f64[-2:].cpu().numpy(), want / (256.0 * s.token_cap ** 2), rtol=F64_RTOL)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,L,E,P", [(1, 3, 8, 4), (7, 2, 8, 8), (5, 4, 64, 32), (300, 2, 128, 16), (9, 2, 128, 128), (4, 1, 512, 256), (6, 3, 1024, 8)])
def test_windows_with_negative_counts_are_refused(N, L, E, P):
    """Placement and projection are queued before the verdict on the counts: aggregate loads below zero must not upset them,
    and a good window behind is planned as ever."""
    t = np.full(N, 3, np.int32)
    good = np.zeros((N, L, E), np.int32)
    good[:, :, 0] = 6
    kw = dict(top_k=2, token_cap=64, dp_width=1, ep_width=P, pop_size=2)
    for value in (-1, -(1 << 31), -3):
        for bad in (np.full((N, L, E), value, np.int32), np.where(np.arange(E) % 3 == 0, 1 << 20, value).astype(np.int32) + 0 * good):
            with pytest.raises(rp.RpError) as e:
                rp.rp_window_load(t, bad, **kw)
            assert e.value.status == -3
        ctx = rp.rp_window_load(t, good, **kw)
        pi, load_ = rp.rp_place_experts(ctx)
        want, G = oracle.lpt(oracle.aggregate(good), P)
        assert (pi == want).all() and (load_ == G).all()
        assert (rp.rp_debug_dump(ctx, "Q", (N, L, P), np.int32) == oracle.project(good, pi, P)).all()
        rp.rp_destroy(ctx)


@pytest.mark.parametrize("P,L", [(864, 5), (1000, 2), (1024, 16)])
def test_diagnostics_of_many_ranks(P, L):
    """Rows of rank loads of up to the most ranks there are, one per warp in shared memory."""
    w = make_window(custom_spec("many_ranks", 24, L, P, 2, 2048, 2, P, 3, 0, data_seed=P))
    s = w.spec
    ref = oracle_front(w, None, 2)
    ctx = load(w, min_rows=2)
    check_front(w, ctx, ref)
    want = oracle.diagnostics(w.lengths, ref["q"], ref["Lagg"], ref["pi"], ref["seed"], ref["R"], s.token_cap, 2, None, s.alpha, s.beta)
    got = rp.rp_diagnostics(ctx)
    for key in ("s_ep", "t_ep", "n_ep"):
        assert got[key] == want[key], key
    for key in ("cv_identity", "cv_placed", "eta_ep", "attention", "joint"):
        assert abs(got[key] - want[key]) <= F64_RTOL * abs(want[key]), key
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,L,P,D,R,edp,ns", [
    (40, 3, 132, 2, 2, None, (1, 2, 400)),              # layers of 33 chunks: more than a warp has lanes
    (60, 5, 256, 3, 2, [0, 1, 1], (1, 7, 300)), (30, 9, 1020, 2, 2, None, (1, 2, 90)),
    (64, 4, 4, 2, 3, None, (256, 270, 290)),            # both sides of the line between few and many layouts
    (2048, 6, 16, 16, 15, None, (1, 2, 3, 4)), (3000, 3, 8, 2, 3, [0, 0], (1, 150, 240)),
    (4096, 2, 4, 32, 40, None, (1, 2))])                # 1280 row-shards of 4096 samples: many from the first layout on
def test_scoring_at_the_edges_of_its_forms(N, L, P, D, R, edp, ns):
    w = make_window(custom_spec("forms", N, L, P, 2, 4096, D, P, 2, 0, data_seed=N + P))
    ref = oracle_front(w, edp, R)
    ctx = load(w, edp=edp, min_rows=R)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, edp, n=3)
    s = w.spec
    rng = np.random.default_rng(P)
    for n in ns:
        lays = rng.integers(0, ref["R"] * D, (n, N)).astype(np.int32)
        some = sorted({0, n // 2, n - 1})
        want = oracle.eval_layouts(w.lengths, ref["q"], lays[some], ref["R"], s.token_cap, D, edp, s.alpha, s.beta)["score"]
        for _ in range(2):                              # the scratch is clear again after a call
            fx, _f64 = rp.rp_eval_population(ctx, lays)
            assert (fx[some] == want).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,D,edp", [(600, 32, [0] * 32), (600, 33, [0] * 33), (600, 64, None), (700, 80, [0, 1] * 40)])
def test_cell_statistics_that_meet_in_a_cluster(N, D, edp):
    """Scoring by clusters of eight: 32 slots, a lane for every CTA of a slot, and more; the scores, and the statistics a search
    starts from."""
    w = make_window(custom_spec("statistics", N, 3, 8, 2, 2048, D, 8, 3, 0, data_seed=D))
    ref = oracle_front(w, edp, 2)
    ctx = load(w, pop=3, edp=edp, min_rows=2)
    check_front(w, ctx, ref)
    check_eval(w, ctx, ref, edp, n=1)
    check_anneal(w, ctx, ref, edp, 3, 2, 20, t_ratio=0.6)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,D", [(255, 5), (256, 4)])
def test_squared_lengths_that_reach_48_bits(N, D):
    """Cap times tokens just below 2^48, where squares are added up in two halves (all samples in one cell: the upper half just fits
    32 bits), and at it, where they are not."""
    t = np.full(N, 1 << 20)
    if N == 255:
        t[3::7] -= 3
    w = one_heavy_expert("squares", t, 2, 4, 2, 1 << 20, D, 4, 2, 0.4)
    s = w.spec
    assert (s.token_cap * int(w.lengths.sum()) < 1 << 48) == (N == 255)
    ref = oracle_front(w, None)
    ctx = load(w, pop=2)
    check_front(w, ctx, ref)
    lays = np.random.default_rng(N).integers(0, ref["R"] * D, (2, N)).astype(np.int32)
    lays[1] = ref["R"] * D - 1
    fx, _ = rp.rp_eval_population(ctx, lays)
    want = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, D, None, s.alpha, s.beta)["score"]
    assert (fx == want).all()
    check_eval(w, ctx, ref, None, n=3)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("L,P,D,edp,pop,mixes,kernel", [
    (32, 4, 4, [1, 2, 3, 0], 9, 4, "k_anneal_wpc"), (8, 8, 3, [2, 0, 1], 256, 4, "k_anneal_wpc"),
    (8, 8, 3, [2, 0, 1], 257, 4, "k_anneal_row"), (5, 12, 3, [2, 0, 1], 20, 4, "k_anneal_row"),
    (6, 16, 4, None, 30, 4, "k_anneal_wpc"), (3, 32, 2, None, 60, 4, "k_anneal_wpc"), (7, 16, 4, None, 30, 4, "k_anneal_row"),
    (12, 4, 2, None, 20, 4, "k_anneal_wpc"), (13, 4, 2, None, 20, 4, "k_anneal_row"), (12, 4, 2, None, 20, 1, "k_anneal_row"),
    (6, 16, 4, None, 30, 1, "k_anneal_row"), (3, 32, 2, None, 200, 1, "k_anneal_row"), (4, 32, 4, [0, 0, 1, 1], 12, 4, "k_anneal_row")])
def test_windows_that_stay_with_the_warp_per_candidate_kernel(L, P, D, edp, pop, mixes, kernel):
    """Permuted one-slot shards, and few layers of many ranks whose row-shards differ in their busiest ranks: both sides of the
    rules, first call and a second one that goes on."""
    if mixes == 1:
        w = one_heavy_expert("stay", np.random.default_rng(L).integers(20_000, 60_000, 70), L, 2 * P, 2, 1 << 19, D, P, pop, 0.4)
    else:
        w = make_window(custom_spec("stay", 70, L, 2 * P, 2, 4096, D, P, pop, 0, data_seed=L * P))
    s = w.spec
    ref = oracle_front(w, edp, 4)
    ctx = load(w, pop=pop, edp=edp, min_rows=4)
    check_front(w, ctx, ref)
    want, stats = check_anneal(w, ctx, ref, edp, pop, 3, 340, t_ratio=0.6, check_members=2)
    assert rp.rp_debug_chain_kernel(ctx) == kernel and stats.accepted > 0
    want = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, D, n_levels=2, steps=33, t0=1e-4,
                         t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed, edp_of_dp=edp, alpha=s.alpha, beta=s.beta)
    rp.rp_anneal(ctx, n_levels=2, steps_per_level=33, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
    assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (2, pop, 3), np.int64) == want["term"]).all()
    assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, 70), np.int32) == want["final_pop"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,L,P,D,R,edp,pop", [(70, 32, 4, 3, 3, None, 21), (900, 24, 2, 8, 31, None, 200), (90, 20, 32, 4, 3, [0, 1, 1, 0], 160)])
@pytest.mark.parametrize("seeds", ["length_only", "trials", "two_plans"])
def test_launch_form_asked_for_after_packing(N, L, P, D, R, edp, pop, seeds):
    """RP_KNOB_LAUNCH_PER_LEVEL set when the population has been built, or even seeded: the same kernel and launches as set before,
    and the population is what it was."""
    w = make_window(custom_spec("late_knob", N, L, 2 * P, 2, 4096, D, P, pop, 0, data_seed=N))
    s = w.spec
    ref = oracle_front(w, edp, R)
    forms = []
    for early in (True, False):
        ctx = load(w, pop=pop, edp=edp, min_rows=R)
        if early:
            rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", 1)
        check_front(w, ctx, ref)
        if seeds == "trials":
            rp.rp_seed_population(ctx, 4)
        elif seeds == "two_plans":
            rp.rp_init_population(ctx, 2)
        if not early:
            before = rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32)
            rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", 1)
            assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == before).all()
        init = rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32)
        _, stats = check_anneal(w, ctx, ref, edp, pop, 3, 30, t_ratio=0.6, check_members=2, init=init)
        forms.append((rp.rp_debug_chain_kernel(ctx), stats.kernel_launches))
        rp.rp_destroy(ctx)
    assert forms[0] == forms[1]


COMPRESSED_CASES = [
    # name, N, L, E, P, D, edp, min_rows, pop: rows of three ranks and a bound per layer, whatever they leave undecided
    ("comp_33_layers", 90, 33, 64, 32, 3, None, 3, 20),            # two layers per lane
    ("comp_65_layers", 60, 65, 32, 32, 2, None, 4, 9),             # four
    ("comp_128_layers", 40, 128, 32, 32, 2, [1, 0], 3, 5),         # a permuted shard map
    ("comp_48_ranks", 70, 12, 96, 48, 3, [0, 1, 1], 3, 30),        # ranks in two passes, shards of two slots
    ("comp_128_ranks", 50, 5, 128, 128, 4, None, 2, 40),
    ("comp_20_ranks", 64, 40, 40, 20, 4, [0, 0, 1, 1], 2, 16),
    ("comp_long", 1500, 6, 48, 48, 2, None, 1, 6),                 # 700 samples a row-shard: collected a piece at a time
    ("comp_one_shard", 900, 9, 40, 40, 3, [0, 0, 0], 1, 1200)]


def compressed_window(spec):
    name, N, L, E, P, D, edp, min_rows, pop = spec
    w = make_window(custom_spec(name, N, L, E, 2, 4096 if N < 1000 else 1 << 18, D, P, pop, 0, data_seed=len(name) + N))
    if N >= 900:                                    # short samples: all of a row-shard's in a few cells
        rng = np.random.default_rng(N)
        w.lengths[:] = rng.integers(1, 3 if N < 1000 else 150, N)
        mixes = rng.dirichlet(np.full(E, 0.3), size=(4, L))
        w.demand[:] = rng.multinomial((2 * w.lengths.astype(np.int64))[:, None], mixes[rng.integers(0, 4, N)])
    return w


@pytest.mark.parametrize("spec", COMPRESSED_CASES, ids=[e[0] for e in COMPRESSED_CASES])
def test_compressed_rows_with_open_layers(spec):
    """Compressed rows on windows of four routing mixes, where many layers are left open and added up from the samples; whole
    trajectories, then on by another kernel and back."""
    name, N, L, E, P, D, edp, min_rows, pop = spec
    w = compressed_window(spec)
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    check_front(w, ctx, ref)
    steps = 60 if pop < 1000 else 12
    want, stats = check_anneal(w, ctx, ref, edp, pop, 3, steps, t_ratio=0.6, check_members=2, t0=1e-2)
    assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row" and stats.accepted > 0
    for knob in (1, 3):
        rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", knob)
        want = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, D, n_levels=2, steps=steps, t0=1e-4,
                             t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed, edp_of_dp=edp, alpha=s.alpha, beta=s.beta,
                             n_threads=8)
        rp.rp_anneal(ctx, n_levels=2, steps_per_level=steps, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
        assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (2, pop, 3), np.int64) == want["term"]).all()
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == want["final_pop"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,L,P,D,edp", [(40, 16, 8, 2, None), (40, 9, 16, 3, [0, 0, 1]), (44, 17, 16, 2, None), (36, 40, 8, 3, [1, 0, 1]),
                                         (36, 31, 16, 2, [1, 0]), (30, 64, 8, 2, None), (48, 7, 12, 2, None), (48, 32, 12, 3, [0, 0, 1])])
def test_rows_dealt_out_to_the_lanes(N, L, P, D, edp):
    """One launch per level with whole rows: 16-byte chunks dealt out to the lanes in turn, one to four of them to a lane, the last
    ones of some lanes missing; and the three chunks of twelve ranks, whole layers to a lane."""
    pop = 1190
    w = make_window(custom_spec("dealt", N, L, 2 * P, 2, 4096, D, P, pop, 400, data_seed=N + L))
    ref = oracle_front(w, edp, 3)
    ctx = load(w, pop=pop, edp=edp, min_rows=3)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, edp, pop, 3, 21, t_ratio=0.5, check_members=2)
    assert rp.rp_debug_chain_form(ctx) == ("whole layers" if P == 12 else "dealt out") and stats.accepted > 0
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("case", ["small", "beyond_16_bits", "beyond_32_bits"])
def test_slacks_of_few_row_shards(case):
    """Hundreds of samples to a row-shard: sums of 16-bit halves, whose lower or upper one alone is used, or both up to a sum
    beyond 32 bits; as scored, and as the moves leave them."""
    rng = np.random.default_rng(len(case))
    edp = None
    if case == "small":
        w = make_window(custom_spec(case, 700, 3, 16, 2, 1 << 17, 2, 8, 6, 0, data_seed=5))
        w.lengths[:] = rng.integers(1, 120, 700)
        w.demand[:] = rng.multinomial((2 * w.lengths.astype(np.int64))[:, None], rng.dirichlet(np.full(16, 0.3), size=3))
    elif case == "beyond_16_bits":
        w = one_heavy_expert(case, rng.integers(20_000, 60_000, 2000), 4, 8, 4, 1 << 23, 2, 8, 6, 0.7)
    else:
        w = one_heavy_expert(case, rng.integers(250_000, 420_000, 40), 120, 4, 8, 1 << 20, 32, 4, 6, 0.9)
        edp = UNEVEN
    s = w.spec
    ref = oracle_front(w, edp)
    ctx = load(w, pop=6, edp=edp)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    check_front(w, ctx, ref)
    G = 1 + (max(edp) if edp is not None else s.dp_width - 1)
    of = np.asarray(edp if edp is not None else range(s.dp_width))
    fixed = ref["G"].argmax(axis=1)                                  # (of equal ones the lowest)
    f = ref["q"].astype(np.int64)[:, np.arange(s.n_layers), fixed].sum(axis=1)
    for init, steps in ((None, 1), ("now", 25)):
        init = rp.rp_debug_dump(ctx, "POPULATION", (6, s.n_samples), np.int32) if init else None
        check_anneal(w, ctx, ref, edp, 6, 2, steps, t_ratio=0.6, check_members=1, init=init, t0=1e-2)
        assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row"
        layouts = rp.rp_debug_dump(ctx, "POPULATION", (6, s.n_samples), np.int32)
        for j in range(6):
            rg = layouts[j] // s.dp_width * G + of[layouts[j] % s.dp_width]
            sums = np.zeros(ref["R"] * G, np.int64)
            np.add.at(sums, rg, f)
            want = rp.rp_debug_dump(ctx, "ESUM", (ref["R"] * G,), np.int64, index=j) - sums
            assert (rp.rp_debug_dump(ctx, "SLACK", (ref["R"] * G,), np.int64, index=j) == want).all()
    assert f.max() < 1 << 16 if case == "small" else f.max() >= 1 << 16
    assert (sums.max() >= 1 << 32) == (case == "beyond_32_bits")
    rp.rp_destroy(ctx)


PAIR_CASES = [
    # as COMPRESSED_CASES, and the steps of a level: sixteen lanes to a chain, one or two layers to a lane
    (("pair_16_layers", 80, 16, 64, 32, 3, None, 3, 45), 50),
    (("pair_17_layers", 80, 17, 64, 32, 3, None, 3, 100), 33),
    (("pair_32_layers", 60, 32, 48, 24, 2, None, 4, 64), 16),
    (("pair_1_layer", 70, 1, 96, 96, 4, None, 2, 57), 7),
    (("pair_long", 1500, 6, 48, 48, 2, None, 1, 43), 64)]


@pytest.mark.parametrize("spec,steps", PAIR_CASES, ids=[e[0][0] for e in PAIR_CASES])
def test_two_chains_to_a_warp(spec, steps):
    """Compressed rows with more members than two SMs hold with a warp each, an odd one left over, windows of steps that end before
    the sixteenth, whole or with open layers; then on with a warp to a chain and back."""
    name, N, L, E, P, D, edp, min_rows, pop = spec
    w = compressed_window(spec)
    s = w.spec
    ref = oracle_front(w, edp, min_rows)
    ctx = load(w, pop=pop, edp=edp, min_rows=min_rows)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 2)
    check_front(w, ctx, ref)
    want, stats = check_anneal(w, ctx, ref, edp, pop, 3, steps, t_ratio=0.6, check_members=2, t0=1e-2)
    assert rp.rp_debug_chain_form(ctx) == "two to a warp" and stats.accepted > 0
    for sms, form in ((0, "compressed"), (2, "two to a warp")):
        rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", sms)
        want = oracle.anneal(w.lengths, ref["q"], want["final_pop"], ref["R"], s.token_cap, D, n_levels=2, steps=steps, t0=1e-4,
                             t_ratio=0.5, p_reloc=0.5, p_guide=0.3, seed=s.anneal_seed, edp_of_dp=edp, alpha=s.alpha, beta=s.beta,
                             n_threads=8)
        rp.rp_anneal(ctx, n_levels=2, steps_per_level=steps, t0=1e-4, t_ratio=0.5, p_reloc=0.5, p_guide=0.3)
        assert rp.rp_debug_chain_form(ctx) == form
        assert (rp.rp_debug_dump(ctx, "TRACE_TERM", (2, pop, 3), np.int64) == want["term"]).all()
        assert (rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32) == want["final_pop"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("L", [16, 17])
@pytest.mark.parametrize("pop,form", [(32, "compressed"), (33, "two to a warp")])
def test_as_many_members_as_are_resident_keep_a_warp_each(L, pop, form):
    """Sixteen warps of 128 registers fill an SM: two SMs keep 32 chains with a warp each, and share warps from the 33rd on."""
    spec = ("resident", 80, L, 64, 32, 3, None, 3, pop)
    w = compressed_window(spec)
    ref = oracle_front(w, None, 3)
    ctx = load(w, pop=pop, min_rows=3)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 2)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, None, pop, 2, 20, t_ratio=0.6, check_members=2, t0=1e-2)
    assert rp.rp_debug_chain_form(ctx) == form and stats.accepted > 0
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("D,R", [(32, 59), (16, 118), (8, 237)])
def test_two_chains_that_take_more_than_half_an_sm_each(D, R):
    """One chain to a warp where the shared memory of two lies between what a launch may ask for (220 KB) and what an SM has (227):
    112 to 116 KB a chain and one resident, so that two to a warp would be half as many again."""
    spec = ("pair_smem", D * R + 12, 2, 40, 20, D, None, R, 5)
    w = compressed_window(spec)
    ref = oracle_front(w, None, R)
    ctx = load(w, pop=5, min_rows=R)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 3)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, None, 5, 3, 40, t_ratio=0.6, check_members=2, t0=1e-2)
    assert rp.rp_debug_chain_form(ctx) == "compressed" and stats.accepted > 0
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("pop", [2, 303, 304, 307, 308])
def test_selection_with_its_distances_on_chip_and_not(pop):
    """The greedy order where all distances of the candidates just fit on chip, and with one candidate more."""
    w = make_window(custom_spec("greedy", 60, 5, 16, 2, 4096, 3, 4, pop, 0, data_seed=3))
    s = w.spec
    ref = oracle_front(w, None, 3)
    ctx = load(w, pop=pop, min_rows=3)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, 3, pop, 5, s.anneal_seed)
    assert rp.rp_seed_population(ctx, 5) == int(ok.sum())
    sc = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, 3, None, s.alpha, s.beta)["score"]
    want = oracle.select_population(w.lengths, ref["q"], lays, sc, ref["R"], s.token_cap, 3, s.top_k, 4, 1 << 16, s.anneal_seed, None,
                                    want_dist=True)
    nd, order = rp.rp_select_population(ctx, 4, 1 << 16)
    assert nd == want["n_distinct"] and (order == want["order"]).all()
    dist = rp.rp_debug_dump(ctx, "SELECT_DIST", (pop, pop), np.int64)
    assert dist.min() >= 0 and dist.max() <= 1 << 22             # (kept in 32 bits on chip)
    rp.rp_destroy(ctx)


# Samples behind the first of each cell: none, one warp of eight a lane filled and one more, both sides of where a lane holds sixteen
# (5120), a CTA of sixteen a lane filled (16384) and one more; cells on both sides of eight to a phase, and of 31 behind the last; more
# cells than samples behind them; five and ten attempts before a row count that fits.
@pytest.mark.parametrize("N,D,min_rows,cap,longest", [
    (12, 4, 3, 50, 50), (257, 1, 0, 1 << 20, 1000), (264, 8, 1, 4096, 60), (265, 8, 0, 4096, 60), (5160, 8, 5, 1 << 16, 300),
    (5161, 8, 5, 1 << 16, 300), (16424, 8, 5, 1 << 20, 500), (16425, 8, 5, 1 << 20, 500), (36000, 3, 0, 1 << 20, 900),
    (900, 31, 0, 700, 400), (1500, 33, 40, 700, 30), (700, 3, 0, 100, 67), (333, 2, 0, 1000, 520), (2600, 1100, 0, 90, 61)])
def test_first_fit_at_the_edges_of_its_warps(N, D, min_rows, cap, longest):
    rng = np.random.default_rng(N + D)
    t = rng.integers(longest // 2 if longest in (67, 61, 520) else 1, longest + 1, N).astype(np.int32)
    a = np.zeros((N, 1, 2), np.int32)
    a[np.arange(N), 0, rng.integers(0, 2, N)] = t
    R, cert, seed = oracle.pack_ffd(t, cap, D, min_rows)
    ctx = rp.rp_window_load(t, a, top_k=1, token_cap=cap, dp_width=D, ep_width=2, pop_size=2, min_rows=min_rows)
    rp.rp_place_experts(ctx)
    assert rp.rp_pack_rows(ctx) == (R, cert)
    assert (rp.rp_debug_dump(ctx, "SEED_LAYOUT", (N,), np.int32) == seed).all()
    rp.rp_destroy(ctx)


# Scoring from a slice of all rows on chip: chunks of a layer one, three and six (several layers to a slice, the last slice with fewer),
# eight, in two pieces and eleven; as many samples as one chunk a row holds and more (no slice); pieces of a layer with a few layouts
# to a batch; row-shards of more samples than are told apart by their number, and of none; odd batches.
@pytest.mark.parametrize("N,L,P,D,R,edp,n", [
    (300, 11, 4, 4, 3, None, 700), (301, 5, 12, 4, 3, None, 500), (120, 3, 24, 2, 9, [0, 0], 900), (1900, 3, 32, 16, 8, None, 40),
    (900, 2, 64, 16, 6, None, 67), (60, 3, 132, 2, 2, None, 400), (14079, 2, 4, 4, 2, None, 100), (14080, 2, 4, 4, 2, None, 100),
    (2600, 2, 64, 32, 40, None, 5), (3000, 3, 16, 2, 2, [0, 0], 700)])
def test_scoring_from_slices_on_chip(N, L, P, D, R, edp, n):
    w = make_window(custom_spec("slices", N, L, P, 2, 4096, D, P, 2, 0, data_seed=N + P))
    ref = oracle_front(w, edp, R)
    ctx = load(w, edp=edp, min_rows=R)
    check_front(w, ctx, ref)
    s = w.spec
    rng = np.random.default_rng(P + N)
    lays = rng.integers(0, ref["R"] * D, (n, N)).astype(np.int32)
    lays[n // 2] = rng.integers(0, 2, N)                # nearly all row-shards empty
    want = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, D, edp, s.alpha, s.beta)["score"]
    for _ in range(2):                                  # the scratch is clear again after a call
        fx, _f64 = rp.rp_eval_population(ctx, lays)
        assert (fx == want).all()
    if n <= 64:
        check_eval(w, ctx, ref, edp, n=n)               # rank loads too
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,L,P,D,pop", [(200, 5, 12, 6, 220), (900, 3, 64, 4, 200)])
def test_rank_loads_of_members_scored_from_slices(N, L, P, D, pop):
    """The rank loads and statistics that scoring leaves for a population are what a search starts from."""
    w = make_window(custom_spec("slice_loads", N, L, P, 2, 4096, D, P, pop, 0, data_seed=P))
    s = w.spec
    ref = oracle_front(w, None, 4)
    ctx = load(w, pop=pop, min_rows=4)
    check_front(w, ctx, ref)
    rp.rp_seed_population(ctx, 4)
    init, _ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, D, pop, 4, s.anneal_seed)
    check_anneal(w, ctx, ref, None, pop, 2, 20, t_ratio=0.6, init=init)
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("L", [16, 17])
@pytest.mark.parametrize("pop", [8, 9, 24, 25, 48, 49])
def test_instances_by_the_members_of_an_sm(L, pop):
    """On two SMs: chains that start beside the launch before them, four to an SM, and more; twelve warps of 168 registers to an SM,
    with a chain each or with two, and more of 128."""
    R = 3 if pop > 16 else 40                   # (few members: rank loads that do not fit on chip)
    spec = ("instances", 80 if R == 3 else 200, L, 64, 32, 3, None, R, pop)
    w = compressed_window(spec)
    ref = oracle_front(w, None, R)
    ctx = load(w, pop=pop, min_rows=R)
    rp.rp_debug_set_knob(ctx, "CHAIN_KERNEL", 3)
    rp.rp_debug_set_knob(ctx, "RESIDENT_SMS", 2)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, None, pop, 4, 70, t_ratio=0.6, check_members=2, t0=1e-2)
    assert rp.rp_debug_chain_form(ctx) == ("two to a warp" if pop > 32 else "compressed") and stats.accepted > 0
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("pop,eta", [(64, 0), (65, 1 << 16), (128, 1 << 20), (129, 1 << 16), (256, 1 << 16), (257, 1 << 18), (40, 1 << 40), (307, 1 << 40)])
def test_greedy_order_by_one_warp(pop, eta):
    """Two, four, eight and ten candidates a lane, filled and one more; penalties that 30 bits do not hold."""
    w = make_window(custom_spec("greedy_warp", 60, 5, 16, 2, 4096, 3, 4, pop, 0, data_seed=4))
    s = w.spec
    ref = oracle_front(w, None, 3)
    ctx = load(w, pop=pop, min_rows=3)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, 3, pop, 5, s.anneal_seed)
    assert rp.rp_seed_population(ctx, 5) == int(ok.sum())
    sc = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, 3, None, s.alpha, s.beta)["score"]
    want = oracle.select_population(w.lengths, ref["q"], lays, sc, ref["R"], s.token_cap, 3, s.top_k, 4, eta, s.anneal_seed)
    nd, order = rp.rp_select_population(ctx, 4, eta)
    assert nd == want["n_distinct"] and (order == want["order"]).all()
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N,longest,width", [(700, 1, 1), (700, 3, 4), (767, 2, 1), (768, 1, 1)])
def test_trials_whose_cells_outgrow_short_keys(N, longest, width):
    """Six cells of 2^20 tokens: keys of 32 bits count 511 samples of a cell (up to 767 samples in the window); with one cell to
    choose from the fullest takes all of the short samples, more than that."""
    rng = np.random.default_rng(N + width)
    t = rng.integers(1, longest + 1, N)
    t[rng.permutation(N)[:6]] = rng.integers(800_000, 1_000_000, 6)
    s = custom_spec("short_keys", N, 2, 4, 2, 1 << 20, 6, 4, 5, 0)
    a = np.zeros((N, 2, 4), np.int32)
    for l in range(2):
        a[np.arange(N), l, rng.integers(0, 4, N)] = 2 * t
    w = Window(s, t.astype(np.int32), a)
    ref = oracle_front(w, None)
    ctx = load(w, pop=5)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, 6, 5, width, s.anneal_seed)
    assert rp.rp_seed_population(ctx, width) == int(ok.sum())
    assert (rp.rp_debug_dump(ctx, "POPULATION", (5, N), np.int32) == lays).all()
    assert ref["R"] == 1 and (max(np.bincount(x).max() for x in lays[1:]) > 511) == (width == 1)
    rp.rp_destroy(ctx)


def test_weights_next_to_an_integer():
    """Fractions whose power lies so close to an integer that double precision does not decide it, all of them, their neighbours, and
    whole exponents with and without a fraction."""
    f = np.arange(1 << 24, dtype=np.uint64)
    y = np.exp2(32.0 - f * 2.0 ** -24)
    r = y - np.floor(y)
    near = f[(r < 2.0 ** -15) | (r > 1 - 2.0 ** -15)]
    assert 500 < near.size < 2000 and near[0] == 0
    z = np.concatenate([near, near[1:] - 1, near[:-1] + 1, np.random.default_rng(1).integers(0, 1 << 24, 4000, dtype=np.uint64)]) << np.uint64(8)
    z = np.concatenate([z, z + np.uint64(255), z + (np.uint64(3) << np.uint64(32)), z + (np.uint64(31) << np.uint64(32))])
    assert rp.rp_debug_exp2neg(z).tolist() == [oracle.exp2neg(int(v)) for v in z]


@pytest.mark.parametrize("pop", [511, 512, 513, 1024, 1025])
def test_between_two_levels_by_members_a_thread(pop):
    """One member a thread weighed by every worker, two, and more, shared out; full and not."""
    w = make_window(custom_spec("members", 600, 3, 8, 2, 2048, 4, 4, pop, 0, data_seed=140))
    ref = oracle_front(w, None, 140)
    ctx = load(w, pop=pop, min_rows=140)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, None, pop, 4, 24, t_ratio=0.4, check_members=2, t0=3e-3)
    assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row" and stats.kernel_launches == 2 * 4 + 2
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("N", [2047, 2048, 2049])
def test_distances_of_as_many_samples_as_registers_hold(N):
    """Eight samples a thread, and one more."""
    w = make_window(custom_spec("held", N, 2, 8, 2, 1 << 16, 4, 4, 9, 0, data_seed=N))
    s = w.spec
    ref = oracle_front(w, None, 3)
    ctx = load(w, pop=9, min_rows=3)
    check_front(w, ctx, ref)
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], ref["R"], s.token_cap, 4, 9, 5, s.anneal_seed)
    assert rp.rp_seed_population(ctx, 5) == int(ok.sum())
    sc = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, 4, None, s.alpha, s.beta)["score"]
    want = oracle.select_population(w.lengths, ref["q"], lays, sc, ref["R"], s.token_cap, 4, s.top_k, 4, 1 << 16, s.anneal_seed, None,
                                    want_dist=True)
    nd, order = rp.rp_select_population(ctx, 4, 1 << 16)
    assert nd == want["n_distinct"] and (order == want["order"]).all()
    assert (rp.rp_debug_dump(ctx, "SELECT_DIST", (9, 9), np.int64) == want["dist"]).all()
    rp.rp_destroy(ctx)


# Samples exactly as long as the cap: one, two, eight, and all cells but one; caps of a power of two, one less and one more; cells on both
# sides of 64, 128, 256 and 512 (two to sixteen keys a lane, and keys in shared memory); the largest cap, where a length fills 64 bits too.
@pytest.mark.parametrize("C,D,R,n_cap,n_short,width", [
    (4096, 2, 4, 1, 56, 4), (4096, 8, 3, 8, 60, 32), (4096, 8, 8, 63, 70, 4), (4097, 8, 8, 63, 70, 4), (4095, 8, 8, 63, 70, 4),
    (8192, 8, 1, 2, 62, 1), (8192, 8, 1, 2, 62, 4), (8192, 8, 1, 2, 62, 8), (8191, 8, 1, 2, 62, 8), (8193, 8, 1, 2, 62, 8), (8192, 8, 1, 7, 250, 32),
    (131072, 8, 9, 70, 90, 8), (131072, 8, 16, 126, 60, 32), (131072, 8, 17, 133, 60, 8), (131072, 8, 32, 254, 60, 32), (131072, 8, 33, 262, 60, 8),
    (65536, 8, 64, 510, 80, 32), (65536, 8, 65, 518, 80, 32), (1, 4, 3, 12, 0, 4), (2, 4, 3, 8, 8, 4), (1 << 24, 8, 1, 7, 20, 4), (1 << 24, 8, 1, 7, 200, 8)])
def test_trials_with_samples_as_long_as_the_cap(C, D, R, n_cap, n_short, width):
    N, K, pop = n_cap + n_short, D * R, 60
    rng = np.random.default_rng(C + N + width)
    t = np.full(N, C)
    free = K - n_cap                                             # cells that no sample of the cap's length takes
    t[:n_short] = rng.integers(1, max(1, min(C - 1, 2 * free * C // (3 * max(1, n_short)))) + 1, n_short)
    t = t[rng.permutation(N)].astype(np.int32)
    s = custom_spec("capped", N, 1, 4, 1, C, D, 4, pop, 0)
    a = np.zeros((N, 1, 4), np.int32)
    a[np.arange(N), 0, rng.integers(0, 4, N)] = t
    w = Window(s, t, a)
    ref = oracle_front(w, None, R)
    assert ref["R"] == R
    lays, ok = oracle.seed_trials(w.lengths, ref["seed"], R, C, D, pop, width, s.anneal_seed)
    ctx = load(w, pop=pop, min_rows=R)
    check_front(w, ctx, ref)
    own = rp.rp_seed_population(ctx, width)
    got = rp.rp_debug_dump(ctx, "POPULATION", (pop, N), np.int32)
    assert max(np.bincount(x, weights=t).max() for x in got) <= C
    assert own == int(ok.sum()) and (got == lays).all()
    rp.rp_destroy(ctx)
    if C > 1 << 20:                                              # (selection refuses so large a cap)
        return
    ctx = load(w, pop=8, min_rows=R)
    check_front(w, ctx, ref)
    nd_want, picked_want, lays_want = oracle_init_population(w, ref, None, pop, 8, width, 4, 1 << 16)
    nd, picked = rp.rp_init_population(ctx, pop, width, 4, 1 << 16)
    assert nd == nd_want and (picked == picked_want).all()
    assert (rp.rp_debug_dump(ctx, "POPULATION", (8, N), np.int32) == lays_want).all()
    rp.rp_destroy(ctx)


def pack_only(t, cap, D, min_rows=0):
    """(rows, certified) and the seed of a window of these lengths (None where it does not fit), and the packing's device time in ms."""
    N = len(t)
    a = np.zeros((N, 1, 2), np.int32)
    a[np.arange(N), 0, np.arange(N) % 2] = t
    rp.rp_debug_set_stage_timing(True)
    ctx = rp.rp_window_load(t, a, top_k=1, token_cap=cap, dp_width=D, ep_width=2, pop_size=2, min_rows=min_rows)
    rp.rp_debug_set_stage_timing(False)
    rp.rp_place_experts(ctx)
    try:
        rows, seed = rp.rp_pack_rows(ctx), rp.rp_debug_dump(ctx, "SEED_LAYOUT", (N,), np.int32)
    except rp.RpError as e:
        assert e.status == -4
        rows, seed = None, None
    ms = rp.rp_debug_stage_times(ctx)["pack_rows"]
    rp.rp_destroy(ctx)
    return rows, seed, ms


# Samples of more than half the cap (no row count but the last will do, or none), of half and one more, a third and one more and less, of both
# sides of both; a few long ones among short ones; attempts that fail in the first and in a later warp, and samples in two parts (more than
# 16384 behind the cells).
@pytest.mark.parametrize("N,D,cap,lo,hi,short", [
    (600, 4, 1000, 501, 900, 0), (601, 4, 1000, 501, 900, 0), (600, 4, 1000, 500, 500, 0), (600, 4, 1000, 400, 600, 0), (602, 7, 999, 334, 499, 0),
    (600, 4, 999, 333, 333, 0), (602, 7, 999, 332, 400, 0), (900, 8, 1000, 200, 600, 0), (40, 3, 100, 40, 70, 0), (300, 4, 1000, 501, 900, 300),
    (500, 2, 1 << 16, 22000, 40000, 700), (5000, 8, 1000, 250, 334, 100), (2500, 8, 400, 101, 200, 100), (900, 4, 100000, 30000, 60000, 17500)])
def test_packing_of_long_samples(N, D, cap, lo, hi, short):
    rng = np.random.default_rng(N + cap)
    t = np.concatenate([rng.integers(lo, hi + 1, N), rng.integers(1, max(2, lo // 20), short)])[rng.permutation(N + short)].astype(np.int32)
    R, cert, seed = oracle.pack_ffd(t, cap, D, 0)
    rows, got, _ms = pack_only(t, cap, D)
    if R == 0:
        assert rows is None
    else:
        assert rows == (R, cert) and (got == seed).all()


@pytest.mark.parametrize("cap,lo,hi", [(32768, 17000, 30000), (32768, 12000, 30000)])
def test_packing_does_not_try_every_row_count(cap, lo, hi):
    """Row counts that the long samples rule out take no pass over the samples each: less time than ten windows of as many short samples."""
    rng = np.random.default_rng(5)
    hard, easy = rng.integers(lo, hi + 1, 2000).astype(np.int32), rng.integers(lo // 8, hi // 8, 2000).astype(np.int32)
    times = [sorted(pack_only(t, cap, 8)[2] for _ in range(5))[2] for t in (hard, easy)]
    assert times[0] < 10 * times[1]


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("L,per_level", [(17, 0), (24, 0), (17, 1)])
def test_chains_that_start_beside_the_launch_between_two_levels(L, per_level, extra):
    """Four chains to an SM start beside the launch between two levels, one chain more and they start at its end; with one launch per level that
    launch is not there.  (The number of launches says which of the two ran.)"""
    import torch
    pop = 4 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    w = make_window(custom_spec("beside", 400, L, 32, 2, 4096, 4, 16, pop, 0, data_seed=L))
    ref = oracle_front(w, None, 90)
    ctx = load(w, pop=pop, min_rows=90)
    rp.rp_debug_set_knob(ctx, "LAUNCH_PER_LEVEL", per_level)
    check_front(w, ctx, ref)
    _, stats = check_anneal(w, ctx, ref, None, pop, 5, 40, t_ratio=0.4, check_members=2, t0=3e-3)
    assert rp.rp_debug_chain_kernel(ctx) == "k_anneal_row"
    assert stats.kernel_launches == 2 * 5 + 2 if per_level == 0 else stats.kernel_launches > 2 * 5 + 2
    rp.rp_destroy(ctx)


@pytest.mark.parametrize("name", ["tiny", "medium"])
def test_loading_and_placing_builds_no_population(name):
    """A caller that only places pays for no population: it is rp_pack_rows that launches its set-up and the seed's scoring."""
    w = make_window(name)
    ref = oracle_front(w)
    counts = [rp.rp_debug_launch_count()]
    ctx = load(w)
    pi, _ = rp.rp_place_experts(ctx)
    counts.append(rp.rp_debug_launch_count())
    assert (pi == ref["pi"]).all()
    assert rp.rp_pack_rows(ctx) == (ref["R"], ref["cert"])
    counts.append(rp.rp_debug_launch_count())
    # checks, placement, projection, packing (with the order of 513 and more samples by a launch of its own); set-up, scoring
    assert counts[1] - counts[0] <= 4 + (w.spec.n_samples > 512) and counts[2] - counts[1] >= 2
    rp.rp_destroy(ctx)


# Narrow slices: one chunk with more layers than are worth it (streamed), and fewer; two chunks of many layers, short row-shards (streamed), long
# ones, and few layers with less and more row-shards to a batch than teams.
@pytest.mark.parametrize("N,L,P,D,R,n", [(7100, 30, 4, 4, 3, 210), (7100, 12, 4, 4, 3, 510), (5000, 40, 8, 4, 12, 160), (5000, 40, 8, 2, 2, 160),
                                         (5000, 3, 8, 8, 30, 40), (5000, 3, 8, 8, 30, 400)])
def test_scoring_from_narrow_slices(N, L, P, D, R, n):
    rng = np.random.default_rng(L)
    s = custom_spec("narrow", N, L, P, 1, 1 << 20, D, P, 2, 0)
    t = rng.integers(1, 400, N).astype(np.int32)
    a = np.zeros((N, L, P), np.int32)
    np.put_along_axis(a, rng.integers(0, P, (N, L, 1)), np.broadcast_to(t[:, None, None], (N, L, 1)), 2)
    w = Window(s, t, a)
    ref = oracle_front(w, None, R)
    assert ref["R"] == R
    ctx = load(w, min_rows=R)
    check_front(w, ctx, ref)
    K = R * D
    lays = np.minimum(rng.integers(0, K, (n, N)), rng.integers(0, K, (n, N))).astype(np.int32)      # (row-shards of different lengths)
    lays[-1] = K - 1
    want = oracle.eval_layouts(w.lengths, ref["q"], lays, ref["R"], s.token_cap, D, None, s.alpha, s.beta)["score"]
    fx, _f64 = rp.rp_eval_population(ctx, lays)
    assert (fx == want).all()
    rp.rp_destroy(ctx)


def test_scoring_of_few_long_row_shards_keeps_its_time():
    """Few row-shards of very different lengths, as first fit leaves them, take no more than 1.6 times as long as as many of one length (they took
    more than twice as long)."""
    import torch
    N, L, P, dp, R, n = 3300, 47, 16, 8, 4, 500
    rng = np.random.default_rng(N)
    t = np.clip(rng.lognormal(np.log(0.93 * 65536 * R * dp / N / 1.9), 1.2, N), 16, 16384).astype(np.int32)
    a = torch.zeros((N, L, P), dtype=torch.int32, device="cuda")
    a[torch.arange(N)[:, None], torch.arange(L)[None, :], torch.from_numpy(rng.integers(0, P, (N, L)))] = torch.from_numpy(t).cuda()[:, None]
    ctx = rp.rp_window_load(torch.from_numpy(t).cuda(), a, top_k=1, token_cap=65536, dp_width=dp, ep_width=P, pop_size=2, min_rows=R)
    rp.rp_place_experts(ctx)
    assert rp.rp_pack_rows(ctx)[0] == R
    fx, f64 = torch.empty((n, 3), dtype=torch.int64, device="cuda"), torch.empty((n, 3), dtype=torch.float64, device="cuda")
    times = []
    for seed in (rp.rp_best(ctx)[0], np.arange(N) % (R * dp)):
        lays = torch.from_numpy(np.stack([rng.permutation(R * dp)[seed] for _ in range(n)]).astype(np.int32)).cuda()
        ms = []
        for _ in range(9):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            rp.rp_eval_population(ctx, lays, fx, f64)
            ev[1].record()
            torch.cuda.synchronize()
            ms.append(ev[0].elapsed_time(ev[1]))
        times.append(sorted(ms)[4])
    rp.rp_destroy(ctx)
    assert times[0] < 1.6 * times[1]
