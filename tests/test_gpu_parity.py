"""Parity of the CUDA path (through the C ABI) with the CPU oracle.

Masks, locks and counts must match exactly; norms, GNMR, Delta-GNMR and R to
a relative 1e-5.  The workloads run in lockstep with the oracle (see
trace_driver) so that every rounded decision has margin."""
import math
from types import SimpleNamespace

import numpy as np
import pytest

import oracle
import workloads
from paper_2606_00539_gb300 import Monitor
from paper_2606_00539_gb300 import _native as N
from tests import trace_driver as TD
from tests.golden import hand_traces

pytestmark = pytest.mark.gpu

RTOL = 1e-5


def _monitor(w, **over):
    kw = w.monitor_kwargs()
    kw.update(over)
    return Monitor(w.offsets, w.lengths, device=0, **kw)


def _policy_kwargs(cfg):
    from fractions import Fraction
    return dict(policy=int(cfg.get("policy", 0)), forced_recovery_steps=int(cfg.get("forced", 0)),
                static_warmup_steps=int(cfg.get("static_warmup", 0)),
                static_fraction=float(cfg.get("static_fraction", Fraction(1, 4))))


def _run_lockstep(w, steps=None, every=1):
    tr = TD.LockstepTrace(w, "cuda:0", _monitor)
    try:
        for t in range(steps or w.steps):
            norms, res, got = tr.step(t)
            if t % every == 0 or t == (steps or w.steps) - 1:
                TD.compare(norms, res, got, RTOL)
    finally:
        tr.close()
    return tr


# ---------------------------------------------------------------------------
# The five workloads (small cases: several tiles per unit and ragged tails)
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("config,shrink,steps", [
    ("tiny", 1, None),           # 64 fp32 units, 200 steps
    ("llama2-1.3b", 8, 60),      # 168 bf16 units, dims / 8
    ("llama2-13b", 16, None),    # 280 bf16 units, dims / 16, 20 steps
    ("moe", 16, 30),             # 5454 bf16 units with unrouted experts
    ("aq-stress", 1, 20),        # 100K fp32 units, contended top-64
])
def test_workload_parity(config, shrink, steps, cuda_device):
    w = workloads.make(config, shrink=shrink, steps=steps)
    tr = _run_lockstep(w)
    assert sum(r.attempts for r in tr.records) < 10 * w.steps


@pytest.mark.parametrize("config,group,shrink,steps", [
    ("llama2-13b", "block", 16, None),     # 40 layer units of 7 tensors each
    ("llama2-1.3b", "block", 8, 40),
    ("moe", "expert", 16, 20),             # attention + each expert as one unit
    ("moe", "block", 32, 20),
])
def test_block_level_units_parity(config, group, shrink, steps, cuda_device):
    """Units spanning several tensors (Sec. 3.4): the unit norm covers all of
    its tensors and the whole block shares one decision."""
    w = workloads.make(config, shrink=shrink, steps=steps, group=group)
    assert w.num_units < w.num_segments
    _run_lockstep(w)


def _large_shape_monitor(w, **over):
    return _monitor(w, loop_shape="large", **over)


@pytest.mark.parametrize("config,group,shrink,steps", [
    ("tiny", "tensor", 1, 60),
    ("llama2-13b", "tensor", 16, None),
    ("aq-stress", "tensor", 1, 10),
    ("moe", "expert", 16, 12),
])
def test_large_unit_loop_shape_parity(config, group, shrink, steps, cuda_device):
    """The large-unit loop shape (twice the loads in flight per warp, half
    the resident warps) forced on the small cases, which would otherwise run
    the small-unit shape: same bar against the oracle."""
    w = workloads.make(config, shrink=shrink, steps=steps, group=group)
    tr = TD.LockstepTrace(w, "cuda:0", _large_shape_monitor)
    try:
        assert tr.mon.info()["loop_shape"] == N.GNMR_LOOP_LARGE_UNITS
        for t in range(w.steps):
            norms, res, got = tr.step(t)
            TD.compare(norms, res, got, RTOL)
    finally:
        tr.close()


def test_loop_shape_follows_the_mean_unit_size(cuda_device):
    """GNMR_LOOP_AUTO takes the large-unit shape at >= 1 MiB per unit."""
    for config, want in (("tiny", N.GNMR_LOOP_SMALL_UNITS), ("aq-stress", N.GNMR_LOOP_SMALL_UNITS),
                         ("llama2-1.3b", N.GNMR_LOOP_LARGE_UNITS), ("llama2-13b", N.GNMR_LOOP_LARGE_UNITS),
                         ("moe", N.GNMR_LOOP_LARGE_UNITS)):
        w = workloads.make(config)
        with _monitor(w) as mon:
            assert mon.info()["loop_shape"] == want, config
        for shape, code in (("small", N.GNMR_LOOP_SMALL_UNITS), ("large", N.GNMR_LOOP_LARGE_UNITS)):
            with _monitor(w, loop_shape=shape) as mon:
                assert mon.info()["loop_shape"] == code


def test_large_unit_loop_takes_runs_dynamically(cuda_device):
    """The large-unit loop plans about 16 runs per warp (64-256 KiB each); the
    small-unit loop reports the warps that start on a block as its runs."""
    for config in ("llama2-1.3b", "llama2-13b", "moe", "tiny", "aq-stress"):
        w = workloads.make(config)
        with _monitor(w) as mon:
            info = mon.info()
            cost = w.grad_bytes + 4096 * w.num_units
            if info["loop_shape"] == N.GNMR_LOOP_LARGE_UNITS:
                assert info["num_runs"] > 4 * info["num_warps"], config
                assert (64 << 10) * 0.99 <= cost / info["num_runs"] <= (256 << 10) * 1.01, config
                assert info["num_partials"] >= info["num_runs"]
            else:
                assert info["num_runs"] == info["num_warps"], config
            assert info["num_ctas"] * info["threads_per_cta"] // 32 >= info["num_warps"]


def test_two_handles_stepping_concurrently_do_not_interfere(cuda_device):
    """Two handles of the same large-unit layout (dynamic runs: each handle
    has its own run counter) stepping on two streams at once, with no host
    synchronisation between them, give bit-identical outputs to a third
    handle stepping alone."""
    import torch
    w = workloads.make("llama2-1.3b", shrink=2, steps=6)
    filler = workloads.Filler(w, cuda_device)
    arenas = []
    for t in range(w.steps):
        a = filler.new_arena()
        filler.fill(a, t)
        arenas.append(a)
    torch.cuda.synchronize()
    mons = [_monitor(w) for _ in range(3)]
    try:
        assert mons[0].info()["num_runs"] > mons[0].info()["num_warps"]
        streams = [torch.cuda.Stream(cuda_device) for _ in range(2)]
        stats = [m.new_stats() for m in mons]
        masks = [torch.empty(w.num_units, dtype=torch.uint8, device=cuda_device) for _ in mons]
        history = [[] for _ in mons]
        for t in range(w.steps):
            for k in range(2):                                   # concurrent, no sync between
                mons[k].step(arenas[t], mask=masks[k], stats=stats[k], stream=streams[k])
            torch.cuda.synchronize()
            mons[2].step(arenas[t], mask=masks[2], stats=stats[2])   # alone
            torch.cuda.synchronize()
            for k in range(3):
                history[k].append({n: v.clone() for n, v in stats[k].items()} | {"mask": masks[k].clone()})
        for t in range(w.steps):
            for k in range(2):
                for name, v in history[2][t].items():
                    assert torch.equal(history[k][t][name], v), (t, k, name)
    finally:
        for m in mons:
            m.close()


def test_segments_in_any_order_and_units_without_segments(cuda_device):
    import torch
    rng = np.random.default_rng(21)
    n = 400_000
    off = np.array([5000, 0, 123_457, 300_001, 77, 200_000, 350_000], np.int64)
    ln = np.array([100_000, 77, 3, 99_999, 4_923, 0, 50_000], np.int64)
    unit = np.array([3, 0, 3, 1, 0, 1, 4], np.int32)                # unit 2 has no segment
    U = 5
    base = _random_arena(rng, n, "bf16").to(cuda_device)
    mon = Monitor(off, ln, dtype="bf16", segment_unit=unit, num_units=U, window=2, max_o=2,
                  lock_len=1, device=0)
    ctl = oracle.Controller(U, window=2, max_o=2, lock_len=1, alpha=(1.5, 1.1), beta=(1.5, 1.5))
    stats = mon.new_stats()
    try:
        for t in range(4):
            dev = (base.float() * float(1.0 + 0.37 * t)).to(torch.bfloat16)
            norms = oracle.unit_norms_segmented(_host_view(dev), off, ln, unit, U)
            assert norms[2] == 0.0
            res = ctl.step(norms)
            mask = mon.step(dev, stats=stats)
            got = {k: v.cpu().numpy() for k, v in stats.items()}
            got["mask"] = mask.cpu().numpy()
            np.testing.assert_allclose(got["norm"], norms, rtol=RTOL, atol=0)
            np.testing.assert_allclose(got["gnmr"], res.gnmr, rtol=RTOL, atol=0)
    finally:
        mon.close()
        ctl.close()


@pytest.mark.parametrize("seed", [1, 2])
def test_tiny_more_seeds(seed, cuda_device):
    _run_lockstep(workloads.make("tiny", seed=seed, steps=120))


# ---------------------------------------------------------------------------
# Hand-derived traces replayed on the GPU (exact norms: one fp32 element each)
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("trace", hand_traces.all_traces(), ids=lambda t: t.name)
def test_hand_trace_on_gpu(trace, cuda_device):
    import torch
    cfg = trace.cfg
    U = int(cfg["units"])
    off = np.arange(U, dtype=np.int64) * 4            # one element per unit, 16 B apart
    ln = np.ones(U, np.int64)
    mon = Monitor(off, ln, dtype="f32", recoverable=[int(x) for x in cfg["recoverable"]],
                  window=int(cfg["window"]), max_o=int(cfg["max_o"]),
                  lock_len=int(cfg["lock_len"]),
                  alpha=(float(cfg["alpha_init"]), float(cfg["alpha_main"])),
                  beta=(float(cfg["beta_init"]), float(cfg["beta_main"])),
                  warmup_steps=int(cfg["warmup"]), eps=float(cfg["eps"]), device=0,
                  **_policy_kwargs(cfg))
    stats = mon.new_stats()
    arena = torch.zeros(4 * U, dtype=torch.float32, device=cuda_device)
    try:
        for st in trace.steps:
            arena[off] = torch.tensor([float(x) for x in st.n], dtype=torch.float32,
                                      device=cuda_device)
            mask = mon.step(arena, stats=stats).cpu().numpy()
            g = {k: v.cpu().numpy() for k, v in stats.items()}
            for b in range(U):
                for key, want in (("gnmr", st.gnmr[b]), ("dgnmr", st.dgnmr[b]),
                                  ("risk", st.risk[b])):
                    want = float(want)
                    if math.isinf(want):
                        assert g[key][b] == want, (st.t, b, key)
                    else:
                        assert g[key][b] == pytest.approx(want, rel=1e-6, abs=1e-12), (st.t, b, key)
            assert list(np.nonzero(mask)[0]) == st.selected, st.t
            assert list(g["lock"]) == st.lock_after, st.t
            assert list(g["counts"]) == [len(st.candidates), len(st.selected)], st.t
    finally:
        mon.close()


# ---------------------------------------------------------------------------
# Edge cases
# ---------------------------------------------------------------------------

def _random_arena(rng, n, dtype, scale=1.0):
    import torch
    x = torch.from_numpy((rng.standard_normal(n) * scale).astype(np.float32))
    return x.to(torch.bfloat16) if dtype == "bf16" else x


def _host_view(t):
    import torch
    t = t.cpu()
    return t.view(torch.int16).numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.numpy()


def _parity_on_norms(off, ln, dev_arena, make_step, mon_kw, ctl_kw, steps, recoverable=None):
    """Runs `steps` steps.  make_step(t, attempt, bad) writes step t's
    gradients into dev_arena; when the oracle finds a decision without margin
    it is called again with attempt + 1 and the units to redraw (the oracle
    state is rolled back first).  Every output is compared with the oracle."""
    U = len(off)
    rec = np.ones(U, np.uint8) if recoverable is None else np.asarray(recoverable, np.uint8)
    mon = Monitor(off, ln, device=0, recoverable=rec, **mon_kw)
    ctl = oracle.Controller(U, recoverable=rec, **ctl_kw)
    stats = mon.new_stats()
    margin_cfg = SimpleNamespace(recoverable=rec, warmup_steps=0,
                                 **{k: ctl_kw[k] for k in ("alpha", "beta", "window", "max_o")})
    try:
        for t in range(steps):
            attempt, bad = 0, []
            while True:
                make_step(t, attempt, bad)
                norms = oracle.unit_norms(_host_view(dev_arena), off, ln)
                before = ctl.get_state()
                res = ctl.step(norms)
                bad = TD.margin_violations(before, res, margin_cfg, t + 1)
                if not bad:
                    break
                ctl.set_state(before)
                attempt += 1
                assert attempt < 30, f"no decision margin at step {t + 1}: units {bad[:8]}"
            mask = mon.step(dev_arena, stats=stats)
            got = {k: v.cpu().numpy() for k, v in stats.items()}
            got["mask"] = mask.cpu().numpy()
            TD.compare(norms, res, got, RTOL)
    finally:
        mon.close()
        ctl.close()


@pytest.mark.parametrize("shape", ["small", "large"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_unaligned_overlapping_and_empty_units(dtype, shape, cuda_device):
    """Units at odd element offsets, overlapping units, gaps, zero-length and
    one-element units, and a unit spanning many warps."""
    import torch
    rng = np.random.default_rng(11)
    n = 3_000_001
    off = np.array([0, 1, 3, 7, 100, 101, 5, 2_000_000, 17, 999_999, 0, 2_999_990], np.int64)
    ln = np.array([1, 2, 13, 0, 1, 777, 2_000_000, 1_000_001, 0, 3, 3_000_001, 11], np.int64)
    base = _random_arena(rng, n, "f32").to(cuda_device)
    dev = torch.empty(n, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32,
                      device=cuda_device)
    gen = torch.Generator(device=cuda_device)

    def make_step(t, attempt, bad):
        # fresh elementwise noise per step (and per attempt): every unit's
        # norm moves on its own
        gen.manual_seed(1000 * t + attempt)
        noise = torch.randn(n, generator=gen, device=cuda_device)
        x = base * (1.0 + 0.3 * noise)
        if t == 3:
            x[2_000_000:2_000_500] *= 40.0
        dev.copy_(x.to(dev.dtype))

    _parity_on_norms(off, ln, dev, make_step,
                     dict(dtype=dtype, window=2, max_o=3, lock_len=2, alpha=1.2, beta=1.2,
                          loop_shape=shape),
                     dict(window=2, max_o=3, lock_len=2, alpha=(1.2, 1.2), beta=(1.2, 1.2)), 6)


def test_dynamic_runs_with_unaligned_special_and_empty_units(cuda_device):
    """The large-unit loop with many more runs than warps (a 400 MB bf16 arena,
    ~6,000 runs of 64 KiB): units at odd offsets, overlapping units, empty and
    one-element units, a unit over the whole arena, a unit that turns NaN and
    one whose squares overflow fp32 (the exact path) at some steps."""
    import torch
    n = 200_000_003
    rng = np.random.default_rng(31)
    off = [0, 1, 3, 7, 11, 150_000_001, 5, 0, 99_999_999, 123]
    ln = [1, 0, 40_000_001, 13, 60_000_000, 49_999_999, 20_000_003, n, 2, 3_000_000]
    for _ in range(30):                                   # assorted units in [0, 100M), some overlapping
        o = int(rng.integers(0, 88_000_000))
        off.append(o)
        ln.append(int(rng.integers(100_000, 12_000_000)))
    off = np.array(off, np.int64)
    ln = np.array(ln, np.int64)
    gen = torch.Generator(device=cuda_device)
    gen.manual_seed(5)
    base = torch.randn(n, generator=gen, device=cuda_device)
    dev = torch.empty(n, dtype=torch.bfloat16, device=cuda_device)

    def make_step(t, attempt, bad):
        gen.manual_seed(7000 + 100 * t + attempt)
        noise = torch.randn(n, generator=gen, device=cuda_device)
        x = base * (1.0 + 0.3 * noise)
        if t == 2:
            x[199_999_990] = float("nan")                     # units 5 and 7 only
        if t == 4:
            x[11 + 1_000:11 + 2_000] = 3e25                    # unit 4: fp32 squares overflow
        dev.copy_(x.to(torch.bfloat16))

    mon_kw = dict(dtype="bf16", window=3, max_o=4, lock_len=2, alpha=1.2, beta=1.2, loop_shape="large")
    with Monitor(off, ln, device=0, **mon_kw) as mon:
        info = mon.info()
        assert info["loop_shape"] == N.GNMR_LOOP_LARGE_UNITS
        assert info["num_runs"] > 2 * info["num_warps"]
    _parity_on_norms(off, ln, dev, make_step, mon_kw,
                     dict(window=3, max_o=4, lock_len=2, alpha=(1.2, 1.2), beta=(1.2, 1.2)), 7)


def _per_unit_levels_arena(rng, ln, steps, sigma, device, zero_units=()):
    """Packed fp32 units; step t of unit u is base * level[t, u].  Returns
    (offsets, arena, make_step) with per-unit margin repair."""
    import torch
    off = np.concatenate([[0], np.cumsum(ln)[:-1]]).astype(np.int64)
    base = _random_arena(rng, int(ln.sum()), "f32").to(device)
    unit_of = torch.from_numpy(np.repeat(np.arange(len(ln)), ln)).to(device)
    levels = np.exp(sigma * rng.standard_normal((steps, len(ln))))
    for u in zero_units:
        levels[:, u] = 0.0
    dev = base.clone()
    cur = {}

    def make_step(t, attempt, bad):
        if attempt == 0:
            cur["lv"] = levels[t].copy()
        for u in bad:
            cur["lv"][u] *= math.exp(rng.uniform(-0.01, 0.01))
        lv = torch.from_numpy(cur["lv"].astype(np.float32)).to(device)
        dev.copy_(base * lv[unit_of])

    return off, dev, make_step


def test_nonfinite_gradients(cuda_device):
    """NaN/Inf in a unit: R = +inf (selected first, ties by index), and the
    unit's A, Q, k stay as they were -- checked over the following steps."""
    rng = np.random.default_rng(13)
    U, L = 16, 4096
    ln = np.full(U, L, np.int64)
    off, dev, base_step = _per_unit_levels_arena(rng, ln, 9, 0.2, cuda_device)

    def make_step(t, attempt, bad):
        base_step(t, attempt, bad)
        if t == 4:
            dev[5 * L + 17] = float("nan")
            dev[9 * L + 3] = float("inf")
            dev[2 * L + 100] = float("-inf")

    _parity_on_norms(off, ln, dev, make_step,
                     dict(dtype="f32", window=3, max_o=2, lock_len=1, alpha=1.5, beta=1.5),
                     dict(window=3, max_o=2, lock_len=1, alpha=(1.5, 1.5), beta=(1.5, 1.5)), 9)


@pytest.mark.parametrize("window", [1, 9, 13, 24])
def test_window_lengths(window, cuda_device):
    """Delta-GNMR windows outside the standard 5 and 8: a single entry, and
    windows longer than the eight entries the epilogue reads per batch (the
    ring wraps mid-batch and leaves a remainder); enough steps that every
    window fills and wraps."""
    rng = np.random.default_rng(100 + window)
    U = 300
    ln = rng.integers(1, 2000, U).astype(np.int64)
    steps = window + 7
    off, dev, make_step = _per_unit_levels_arena(rng, ln, steps, 0.3, cuda_device)
    _parity_on_norms(off, ln, dev, make_step,
                     dict(dtype="f32", window=window, max_o=6, lock_len=2, alpha=1.3, beta=1.2),
                     dict(window=window, max_o=6, lock_len=2, alpha=(1.3, 1.3), beta=(1.2, 1.2)), steps)


@pytest.mark.parametrize("max_o,lock_len,thr", [(0, 3, 1.05), (10_000, 0, 1.05), (7, 2, 0.9)])
def test_budget_extremes_and_ties(max_o, lock_len, thr, cuda_device):
    """maxO = 0 (never select), maxO >= U (plain threshold), and thresholds
    below 1 so that every unit ties at t = 1 (index order decides); some units
    are not recoverable and some are all zeros."""
    rng = np.random.default_rng(14)
    U = 5000
    ln = rng.integers(1, 300, U).astype(np.int64)
    rec = (rng.random(U) < 0.9).astype(np.uint8)
    off, dev, make_step = _per_unit_levels_arena(rng, ln, 8, 0.5, cuda_device,
                                                 zero_units=range(0, U, 97))
    _parity_on_norms(off, ln, dev, make_step,
                     dict(dtype="f32", window=2, max_o=max_o, lock_len=lock_len, alpha=thr, beta=thr),
                     dict(window=2, max_o=max_o, lock_len=lock_len, alpha=(thr, thr), beta=(thr, thr)),
                     8, recoverable=rec)


@pytest.mark.parametrize("shape", ["small", "large"])
def test_tiny_and_huge_fp32_values_take_the_exact_path(shape, cuda_device):
    """fp32 squares underflow below ~1e-19 and overflow above ~1.8e19; the
    kernel's fp64 fallback keeps the norm within rounding of the oracle."""
    import torch
    rng = np.random.default_rng(12)
    parts = [rng.standard_normal(5000) * 1e-30, rng.standard_normal(5000) * 1e25,
             rng.standard_normal(5000), np.concatenate([np.full(10, 1e-44), np.zeros(90)]),
             rng.standard_normal(70000) * 3e-21]
    host = np.concatenate(parts).astype(np.float32)
    off = np.cumsum([0] + [len(p) for p in parts[:-1]]).astype(np.int64)
    ln = np.array([len(p) for p in parts], np.int64)
    dev = torch.from_numpy(host).to(cuda_device)
    mon = Monitor(off, ln, dtype="f32", device=0, loop_shape=shape)
    stats = mon.new_stats()
    try:
        mon.step(dev, stats=stats)
        got = stats["norm"].cpu().numpy()
    finally:
        mon.close()
    want = oracle.unit_norms(host, off, ln)
    assert np.all(want > 0)
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=0)


def test_all_units_tie_under_contention(cuda_device):
    """100K units, thresholds 0.5: at t = 1 every unit has R = 2; the top-64
    must be units 0..63."""
    import torch
    U = 100_000
    off = np.arange(U, dtype=np.int64) * 4
    ln = np.full(U, 4, np.int64)
    dev = torch.ones(4 * U, dtype=torch.float32, device=cuda_device)
    mon = Monitor(off, ln, dtype="f32", max_o=64, lock_len=3, alpha=0.5, beta=0.5, window=4, device=0)
    stats = mon.new_stats()
    try:
        mask = mon.step(dev, stats=stats).cpu().numpy()
        assert list(np.nonzero(mask)[0]) == list(range(64))
        assert list(stats["counts"].cpu().numpy()) == [U, 64]
        assert np.all(stats["risk"].cpu().numpy() == 2.0)
    finally:
        mon.close()


def test_threshold_override_and_schedule(cuda_device):
    """gnmr_set_thresholds overrides alpha_t/beta_t until reset with NaN."""
    w = workloads.make("tiny", seed=5, steps=40, shrink=8)
    tr = TD.LockstepTrace(w, "cuda:0", _monitor)
    try:
        for t in range(w.steps):
            if t == 20:
                tr.mon.set_thresholds(1.05, 1.2)
            if t == 30:
                tr.mon.set_thresholds(float("nan"), float("nan"))
            a, b = (1.05, 1.2) if 20 <= t < 30 else (math.nan, math.nan)
            norms, res, got = tr.step(t, a, b)
            TD.compare(norms, res, got, RTOL)
    finally:
        tr.close()


@pytest.mark.parametrize("config,shrink", [("llama2-13b", 32), ("tiny", 1), ("moe", 32)])
def test_pinned_host_arena_is_read_in_place(config, shrink, cuda_device):
    """gnmr_step on a pinned host arena (read in place over the host link)
    gives bitwise the outputs of the same arena in device memory, and so do
    the partial sums; an unpinned host tensor is refused."""
    import torch
    w = workloads.make(config, shrink=shrink, steps=4)
    f = workloads.Filler(w, cuda_device)
    arena = f.new_arena()
    host = torch.empty(arena.numel(), dtype=arena.dtype, pin_memory=True)
    m_dev, m_host = _monitor(w), _monitor(w)
    s_dev, s_host = m_dev.new_stats(), m_host.new_stats()

    def bits(x):
        return x.view(torch.int64) if x.dtype == torch.float64 else x

    try:
        for t in range(w.steps):
            f.fill(arena, t)
            host.copy_(arena)
            a = m_dev.step(arena, stats=s_dev)
            b = m_host.step(host, stats=s_host)
            torch.cuda.synchronize()
            assert torch.equal(a, b), f"mask, step {t + 1}"
            for k in s_dev:
                assert torch.equal(bits(s_dev[k]), bits(s_host[k])), f"{k}, step {t + 1}"
        assert torch.equal(bits(m_dev.step_partials(arena)), bits(m_host.step_partials(host)))
        with pytest.raises(ValueError, match="pinned"):
            m_host.step(torch.zeros(8, dtype=arena.dtype))
    finally:
        m_dev.close()
        m_host.close()


def test_prepared_step_matches_step(cuda_device):
    """Monitor.prepare_step: the prepared call gives bitwise the outputs of
    step() on the same arena contents, follows new contents written into the
    same storage, and refuses to run after close()."""
    import torch
    w = workloads.make("aq-stress", shrink=4, steps=5)
    f = workloads.Filler(w, cuda_device)
    arena = f.new_arena()
    m_a, m_b = _monitor(w), _monitor(w)
    s_a, s_b = m_a.new_stats(), m_b.new_stats()
    mask_b = torch.empty(w.num_units, dtype=torch.uint8, device=cuda_device)
    run = m_b.prepare_step(arena, mask=mask_b, stats=s_b)
    try:
        for t in range(w.steps):
            f.fill(arena, t)
            a = m_a.step(arena, stats=s_a)
            b = run()
            torch.cuda.synchronize()
            assert b is mask_b and torch.equal(a, b), f"mask, step {t + 1}"
            for k in s_a:
                x, y = s_a[k], s_b[k]
                if x.dtype == torch.float64:
                    x, y = x.view(torch.int64), y.view(torch.int64)
                assert torch.equal(x, y), f"{k}, step {t + 1}"
    finally:
        m_a.close()
        m_b.close()
    with pytest.raises(ValueError, match="closed"):
        run()


@pytest.mark.parametrize("shape", ["small", "large"])
def test_deterministic_across_handles_and_runs(shape, cuda_device):
    import torch
    w = workloads.make("llama2-13b", shrink=32, steps=4)
    f = workloads.Filler(w, cuda_device)
    arena = f.new_arena()
    outs = []
    for _ in range(2):
        mon = _monitor(w, loop_shape=shape)
        stats = mon.new_stats()
        vals = []
        for t in range(w.steps):
            f.fill(arena, t)
            mon.step(arena, stats=stats)
            vals.append(stats["norm"].cpu().numpy().copy())
        mon.close()
        outs.append(np.stack(vals))
    assert np.array_equal(outs[0].view(np.uint64), outs[1].view(np.uint64))


def test_errors_leave_state_unchanged(cuda_device):
    import torch
    rng = np.random.default_rng(15)
    U, L = 8, 1000
    off = np.arange(U, dtype=np.int64) * L
    ln = np.full(U, L, np.int64)
    dev = _random_arena(rng, U * L, "bf16").to(cuda_device)
    mon = Monitor(off, ln, dtype="bf16", device=0)
    ctl = oracle.Controller(U, window=8, max_o=4, lock_len=1, alpha=(1.5, 1.1), beta=(1.5, 1.5))
    stats = mon.new_stats()
    mask = torch.empty(U, dtype=torch.uint8, device=cuda_device)
    try:
        h = mon._h
        # arena shorter than the layout
        with pytest.raises(N.GnmrError) as ei:
            N.gnmr_step(h, dev.data_ptr(), U * L - 1, 0, mask.data_ptr(), None)
        assert ei.value.status == N.GNMR_ERR_LAYOUT
        # misaligned arena pointer (odd byte address for bf16)
        with pytest.raises(N.GnmrError) as ei:
            N.gnmr_step(h, dev.data_ptr() + 1, U * L, 0, mask.data_ptr(), None)
        assert ei.value.status == N.GNMR_ERR_INVALID_ARG
        with pytest.raises(N.GnmrError) as ei:
            N.gnmr_step(h, dev.data_ptr(), U * L, 0, None, None)
        assert ei.value.status == N.GNMR_ERR_INVALID_ARG
        with pytest.raises(N.GnmrError):
            mon.set_thresholds(-1.0, 1.0)
        assert mon.info()["steps"] == 0
        for t in range(3):
            dev.mul_(1.0 + t)
            norms = oracle.unit_norms(_host_view(dev), off, ln)
            res = ctl.step(norms)
            m = mon.step(dev, stats=stats)
            got = {k: v.cpu().numpy() for k, v in stats.items()}
            got["mask"] = m.cpu().numpy()
            TD.compare(norms, res, got, RTOL)
        assert mon.info()["steps"] == 3
    finally:
        mon.close()
        ctl.close()


def test_mask_only_and_side_stream(cuda_device):
    import torch
    w = workloads.make("tiny", seed=7, steps=12, shrink=4)
    f = workloads.Filler(w, cuda_device)
    arena = f.new_arena()
    a = _monitor(w)
    b = _monitor(w)
    stats = b.new_stats()
    side = torch.cuda.Stream(cuda_device)
    try:
        for t in range(w.steps):
            f.fill(arena, t)
            torch.cuda.synchronize()
            with torch.cuda.stream(side):
                m1 = a.step(arena, stream=side)
            m2 = b.step(arena, stats=stats)
            side.synchronize()
            torch.cuda.synchronize()
            assert torch.equal(m1, m2)
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("config,shrink,steps", [("tiny", 4, 30),
                                                 ("llama2-1.3b", 2, 10)])   # dynamic runs
def test_cuda_graph_replay_advances_steps(config, shrink, steps, cuda_device):
    """The step is one launch with no host synchronisation: captured once in a
    CUDA graph and replayed, it matches the oracle step by step (the step
    counter, the thresholds and the large-unit loop's run counter live on the
    device and are reset by the kernel)."""
    import torch
    w = workloads.make(config, seed=9, steps=steps, shrink=shrink)
    tr = TD.LockstepTrace(w, "cuda:0", _monitor)
    mask = torch.empty(w.num_units, dtype=torch.uint8, device=cuda_device)
    s = torch.cuda.Stream(cuda_device)
    g = torch.cuda.CUDAGraph()
    try:
        with torch.cuda.graph(g, stream=s):
            tr.mon.step(tr.arena, mask=mask, stats=tr.stats, stream=s)
        # capturing does not run the kernel: the device state is still at t = 0

        def replay():
            g.replay()
            return mask

        for t in range(w.steps):
            norms, res, got = tr.step(t, gpu_step=replay)
            TD.compare(norms, res, got, RTOL)
    finally:
        tr.close()


@pytest.mark.parametrize("config,shrink", [("aq-stress", 8), ("llama2-13b", 16)])
def test_steps_wait_for_the_kernel_that_writes_the_arena(config, shrink, cuda_device):
    """Steps enqueued right behind the kernel that writes their arena, with no
    host synchronisation in between: fill, step, fill, step, ... on one
    stream.  Each step must see its own step's gradients (its norms equal the
    oracle's on that step's bytes, regenerated separately afterwards), so a
    step never starts reading before the writer has finished."""
    import torch
    import oracle
    w = workloads.make(config, shrink=shrink, steps=6)
    filler = workloads.Filler(w, cuda_device)
    arena = filler.new_arena()
    mon = _monitor(w)
    norms = torch.empty((w.steps, w.num_units), dtype=torch.float64, device=cuda_device)
    stats = mon.new_stats()
    try:
        torch.cuda.synchronize()
        for t in range(w.steps):
            filler.fill(arena, t)                    # torch's current stream, then the step on it
            mon.step(arena, stats=dict(stats, norm=norms[t]))
        torch.cuda.synchronize()
        got = norms.cpu().numpy()
        check = filler.new_arena()
        for t in range(w.steps):
            filler.fill(check, t)
            host = check.cpu()
            view = host.view(torch.int16).numpy().view(np.uint16) if w.dtype == "bf16" else host.numpy()
            want = oracle.unit_norms_threaded(view, w.offsets, w.lengths, 8)
            np.testing.assert_allclose(got[t], want, rtol=RTOL, atol=0, err_msg=f"step {t + 1}")
    finally:
        mon.close()


@pytest.mark.parametrize("units_per_sm,extra", [(1, 0), (6, 1), (16, 0), (16, 1), (32, 1), (133, 3), (520, 0)])
def test_small_unit_batches_update_every_unit_once(units_per_sm, extra, cuda_device):
    """The small-unit loop runs the epilogues in batches of 32 units of a CTA,
    by whichever warp completes one.  The controller half runs them unit by
    unit, so both must leave the same state, masks and statistics, bit for
    bit, on the same sums."""
    import torch
    U = units_per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    rng = np.random.default_rng(U)
    lengths = rng.integers(0, 300, U).astype(np.int64)
    offsets = np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64)
    kw = dict(dtype="f32", window=3, max_o=7, lock_len=2, alpha=1.1, beta=1.2)
    one, two = Monitor(offsets, lengths, **kw), Monitor(offsets, lengths, **kw)
    try:
        for step in range(5):
            g = torch.Generator(cuda_device).manual_seed(step)
            arena = torch.randn(int(lengths.sum()), device=cuda_device, generator=g) * (1.0 + (step == 4))
            s1, s2 = one.new_stats(), two.new_stats()
            m1 = one.step(arena, stats=s1)
            m2 = two.finish(two.step_partials(arena), stats=s2)
            assert torch.equal(m1, m2)
            for key in s1:
                assert torch.equal(s1[key], s2[key]), key
        assert one.get_state() == two.get_state()
    finally:
        one.close()
        two.close()


@pytest.mark.parametrize("mib,extra,want", [(512, 0, "large"), (512, -1, "small"), (100, 0, "small")])
def test_loop_shape_of_small_arenas(mib, extra, want, cuda_device):
    """Units of 1 MiB and more take the large-unit shape from 512 MiB on."""
    lengths = np.full(mib // 4, 1 << 20, np.int64)
    lengths[0] += extra
    with Monitor(np.cumsum(lengths) - lengths, lengths, dtype="f32") as mon:
        assert mon.info()["loop_shape"] == (N.GNMR_LOOP_LARGE_UNITS if want == "large" else N.GNMR_LOOP_SMALL_UNITS)


def test_device_memory_of_a_small_unit_handle(cuda_device):
    """Per unit: state, window, candidate, ticket, flag, one partial sum, one
    block and its place; nothing of the large-unit loop's tables."""
    U, window = 50_000, 2
    lengths = np.full(U, 1000, np.int64)                  # 4 KB, one block of a whole warp
    with Monitor(np.cumsum(lengths) - lengths, lengths, dtype="f32", window=window) as mon:
        info = mon.info()
    assert info["loop_shape"] == N.GNMR_LOOP_SMALL_UNITS
    unit = 40 + 8 * window + 16 + 4 + 1 + 8 + 16 + 4
    cta = 64 + 2 * 8 + 2 * 16                             # table, and the parts of the units it cuts
    fixed = 16 * 8192 + 4 * 2048 + 256 + 12 * 256         # hot list, histogram, control, alignment
    assert info["device_bytes"] <= unit * U + cta * info["num_ctas"] + fixed


def _block_layout(name):
    if name == "block-edges":                             # around one and two blocks of 8 KiB
        return np.repeat([0, 1, 2047, 2048, 2049, 4095, 4096, 4097, 6145], 40)
    if name == "whole-units":                             # around the 128 KiB up to which a small arena's stay whole
        return np.array([1, 31_742, 31_743, 31_744, 31_745, 32_769, 0, 63_489, 63_487, 5, 100_003, 300] * 3)
    if name == "cta-spans":                               # units over two, three and more CTAs' parts
        return np.array([5_000, 300_001, 12_000, 20_000, 7, 990_003, 1, 0, 50_000, 64_001] * 8)
    if name == "more-than-resident":                      # more units than the resident CTAs' blocks
        return np.arange(700_001) % 4
    return np.array([70_000_001, 3, 0, 12_345])           # "one-giant": blocks larger than 8 KiB


@pytest.mark.parametrize("name", ["block-edges", "whole-units", "cta-spans", "more-than-resident", "one-giant"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_block_loop_layouts(name, dtype, cuda_device):
    """Norms of the small-unit loop at the edges of its plan, at odd offsets,
    against 64-bit sums, twice (the second step reuses every slot)."""
    import torch
    lengths = _block_layout(name).astype(np.int64)
    offsets = np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64) + 1
    n = int(lengths.sum()) + 1
    ids = torch.repeat_interleave(torch.arange(len(lengths), device=cuda_device),
                                  torch.from_numpy(lengths).to(cuda_device))
    with Monitor(offsets, lengths, dtype=dtype, loop_shape="small", window=2) as mon:
        stats = mon.new_stats()
        for seed in (1, 2):
            g = torch.Generator(cuda_device).manual_seed(seed)
            arena = torch.randn(n, device=cuda_device, generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
            mon.step(arena, stats=stats)
            want = torch.zeros(len(lengths), dtype=torch.float64, device=cuda_device)
            want.index_add_(0, ids, arena[1:].double().square())
            # a piece's fp32 sum: at most about 27 roundings of 2^-24 per block
            # of 16 iterations and 5 over the lanes, halved by the square root
            torch.testing.assert_close(stats["norm"], want.sqrt(), rtol=1e-6, atol=0)


@pytest.mark.parametrize("units,segments,most", [(1, 3000, 0), (1, 20_001, 2), (2, 100_000, 1), (300, 400_000, 3)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_block_loop_of_many_tiny_segments(units, segments, most, dtype, cuda_device):
    """Units of more tiny segments than a CTA has slots for block sums, in
    arenas small enough to be cut between units: the plan cuts inside them."""
    import torch
    rng = np.random.default_rng(segments)
    lengths = rng.integers(0, most + 1, segments)
    unit = np.arange(segments) * units // segments
    offsets = np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64) + 1
    n = int(lengths.sum()) + 1
    ids = torch.from_numpy(np.repeat(unit, lengths)).to(cuda_device)
    with Monitor(offsets, lengths, dtype=dtype, segment_unit=unit.astype(np.int32), num_units=units,
                 loop_shape="small", window=2) as mon:
        stats = mon.new_stats()
        for seed in (1, 2):
            g = torch.Generator(cuda_device).manual_seed(seed)
            arena = torch.randn(n, device=cuda_device, generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
            mon.step(arena, stats=stats)
            want = torch.zeros(units, dtype=torch.float64, device=cuda_device)
            want.index_add_(0, ids, arena[1:].double().square())
            # two roundings of 2^-24 or fewer per segment of up to three elements
            torch.testing.assert_close(stats["norm"], want.sqrt(), rtol=2.0 ** -23, atol=0)


@pytest.mark.parametrize("tiny,large,where", [(2500, 400, 0), (5000, 400, 200), (100_000, 300, 300)])
def test_block_loop_of_tiny_segments_among_large_units(tiny, large, where, cuda_device):
    """A unit of more one-element segments than a CTA has slots for block sums,
    before, between or after ordinary units: it alone is cut shorter."""
    import torch
    lengths = np.concatenate([np.full(where, 100_001), np.ones(tiny, np.int64), np.full(large - where, 100_001)])
    unit = np.concatenate([np.arange(where), np.full(tiny, where), np.arange(where + 1, large + 1)])
    offsets = np.cumsum(lengths) - lengths
    ids = torch.from_numpy(np.repeat(unit, lengths)).to(cuda_device)
    with Monitor(offsets, lengths, dtype="f32", segment_unit=unit.astype(np.int32), num_units=large + 1,
                 loop_shape="small", window=2) as mon:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert mon.info()["num_ctas"] <= (2 if tiny <= 5000 else 4) * sms
        stats = mon.new_stats()
        g = torch.Generator(cuda_device).manual_seed(tiny)
        arena = torch.randn(int(lengths.sum()), device=cuda_device, generator=g)
        mon.step(arena, stats=stats)
        want = torch.zeros(large + 1, dtype=torch.float64, device=cuda_device).index_add_(0, ids, arena.double().square())
        # at most 27 fp32 roundings per block of 16 iterations, and 2^-26 per lane
        torch.testing.assert_close(stats["norm"], want.sqrt(), rtol=1e-6, atol=0)
        assert torch.equal(mon.step_partials(arena).sqrt(), stats["norm"])


@pytest.mark.parametrize("shape", ["small", "large"])
@pytest.mark.parametrize("power", [-75, -51, -50, -49, -3, 0, 40, 48, 49, 50, 51, 62])
def test_lane_totals_of_any_size(power, shape, cuda_device):
    """The warp's sum over lanes whose totals differ by up to 2^60, around the
    ends of the range beyond which squares are taken in fp64."""
    import torch
    lengths = np.array([1, 31, 128, 129, 1000, 4096, 20_000, 300_001], np.int64)
    offsets = np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64)
    n = int(lengths.sum())
    g = torch.Generator(cuda_device).manual_seed(5)
    for spread in (0, 4, 30):
        x = torch.randn(n, device=cuda_device, generator=g, dtype=torch.float64)
        x = x * torch.exp2(-spread * torch.rand(n, device=cuda_device, generator=g, dtype=torch.float64)) * 2.0 ** power
        arena = x.float()
        with Monitor(offsets, lengths, dtype="f32", loop_shape=shape) as mon:
            stats = mon.new_stats()
            mon.step(arena, stats=stats)
            got = stats["norm"].cpu().numpy()
        want = [float(arena[o:o + m].double().square().sum().sqrt()) for o, m in zip(offsets.tolist(), lengths.tolist())]
        # in a block of 16 iterations of up to 16 vectors at most 27 fp32 roundings
        # of non-negative terms, and 2^-26 of the largest lane 32 times; the root
        # halves it: 27 / 2 * 2^-24 + 16 * 2^-26 < 1.1e-6
        np.testing.assert_allclose(got, want, rtol=1.1e-6, atol=0)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("start", [0, 1, 3])
def test_short_units_share_a_warp(dtype, start, cuda_device):
    """20,000 units at the edges of what 4, 8, 16 and 32 lanes stream, packed
    without padding, some of zeros, some whose fp32 squares underflow or
    overflow, some with a NaN or an Inf."""
    import torch
    eb = 4 if dtype == "f32" else 2
    sizes = [b // eb + d for b in (16, 128, 512, 1024, 2048, 4096) for d in (-1, 0, 1)] + [0, 1, 2, 9]
    rng = np.random.default_rng(start)
    U = 20_000
    lengths = rng.choice(np.array(sizes, np.int64), U)
    offsets = start + np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64)
    scale = rng.choice([1.0, 1.0, 1.0, 1e-3, 0.0, 1e-25, 1e25], U)
    n = int(offsets[-1] + lengths[-1])
    ids = torch.repeat_interleave(torch.arange(U, device=cuda_device), torch.from_numpy(lengths).to(cuda_device))
    g = torch.Generator(cuda_device).manual_seed(start)
    x = torch.zeros(n, dtype=torch.float64, device=cuda_device)
    x[start:] = torch.randn(n - start, device=cuda_device, generator=g, dtype=torch.float64) * torch.from_numpy(scale).to(cuda_device)[ids]
    for u, bad in ((77, float("nan")), (78, float("inf")), (4001, float("-inf"))):
        if lengths[u]:
            x[int(offsets[u] + lengths[u] // 2)] = bad
    arena = x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    want = torch.zeros(U, dtype=torch.float64, device=cuda_device).index_add_(0, ids, arena[start:].double().square()).sqrt()
    with Monitor(offsets, lengths, dtype=dtype, window=2) as mon:
        stats = mon.new_stats()
        mon.step(arena, stats=stats)
        # at most 64 fp32 roundings per lane of non-negative terms, mostly of partial
        # sums far below the total, and 2^-26 per lane; measured below 1e-7
        torch.testing.assert_close(stats["norm"], want, rtol=1e-6, atol=0, equal_nan=True)
        sums = mon.step_partials(arena)
        assert torch.equal(sums.sqrt().nan_to_num(7.0), stats["norm"].nan_to_num(7.0))


@pytest.mark.parametrize("shape", ["small", "large", "grouped"])
def test_lanes_are_joined_without_rounding(shape, cuda_device):
    """One element in each lane's first vector, squares of 24 bits in [1, 2) and
    [1/4, 1/2): the lanes' totals and their sum fit the 26-bit fractions exactly,
    where fp32 additions over the lanes would round (1e-8)."""
    import torch
    rng = np.random.default_rng(3)
    if shape == "grouped":                                # 4, 8 and 16 lanes to a unit
        lengths = np.tile([16, 136, 264], 7000)
        lanes = np.tile([4, 8, 16], 7000)
    else:
        lengths = np.full(64, 128)
        lanes = np.full(64, 32)
    offsets = np.cumsum(lengths) - lengths                # multiples of 8 elements: no head
    lane = np.arange(lanes.sum()) - np.repeat(np.cumsum(lanes) - lanes, lanes)
    x = (1 + rng.integers(1, 800, len(lane)) * 2.0 ** -11) * rng.choice([1.0, 0.5], len(lane))
    host = np.zeros(int(lengths.sum()), np.float32)
    host[np.repeat(offsets, lanes) + 4 * lane] = x        # exact in 12 bits
    want = np.sqrt(np.add.reduceat(x * x, np.cumsum(lanes) - lanes))      # exact sums, one rounding
    with Monitor(offsets, lengths, dtype="f32", window=2, loop_shape="large" if shape == "large" else "small") as mon:
        stats = mon.new_stats()
        arena = torch.from_numpy(host).to(cuda_device)
        mon.step(arena, stats=stats)
        # a unit that two CTAs share is cut where fewer lanes may hold more of it
        cut = mon.info()["num_ctas"] - 1 if shape == "grouped" else 0
        for got in (stats["norm"].cpu().numpy(), np.sqrt(mon.step_partials(arena).cpu().numpy())):
            assert (got != want).sum() <= cut
            np.testing.assert_allclose(got, want, rtol=2.0 ** -22, atol=0)


@pytest.mark.parametrize("shape", ["small", "large"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("start", [0, 1])
def test_ends_of_pieces(dtype, shape, start, cuda_device):
    """Units that end around every length of the last round of loads: whole
    numbers, whose sums of squares no rounding touches, come out exact."""
    import torch
    per = 4 if dtype == "f32" else 8
    vecs = [v + d for v in (0, 32, 64, 96, 128, 160, 192, 224, 256, 384, 448, 512, 768, 1024) for d in (-1, 0, 1) if v + d >= 0]
    lengths = np.array([v * per + e for v in vecs for e in (0, 1, per - 1)], np.int64)
    offsets = start + np.cumsum(lengths) - lengths
    n = int(offsets[-1] + lengths[-1])
    g = torch.Generator(cuda_device).manual_seed(11)
    x = torch.randint(-3, 4, (n,), device=cuda_device, generator=g)
    ids = torch.repeat_interleave(torch.arange(len(lengths), device=cuda_device), torch.from_numpy(lengths).to(cuda_device))
    want = torch.zeros(len(lengths), dtype=torch.float64, device=cuda_device).index_add_(0, ids, x[start:].double().square())
    arena = x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    with Monitor(offsets, lengths, dtype=dtype, window=2, loop_shape=shape) as mon:
        stats = mon.new_stats()
        mon.step(arena, stats=stats)
        assert torch.equal(stats["norm"], want.sqrt())
        assert torch.equal(mon.step_partials(arena), want)
