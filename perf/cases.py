"""Performance cases of the GNMR monitor: what a training program has it do,
through its public entry points.

Four kinds of call, each one pass of ``run``:

* ``step``     one ``Monitor.prepare_step`` call: the whole monitor step on a
               gradient arena, with every statistic written;
* ``shard``    one rank's part of a sharded step: ``step_partials`` on its
               slice, then ``finish`` (the all-reduce in between is the
               caller's and is left out);
* ``norms``    ``gnmr_unit_norms_static``, the allocation-free norms;
* ``act``      ``gnmr_actuator_apply`` over every unit's saved activations.

A ``step`` or ``shard`` state holds a monitor that has already observed
``window + 3`` steps, so that queues are full and means have settled, and
several arenas that consecutive passes take in turn, as consecutive training
steps bring other gradients: units that spike in one arena only keep
triggering, so the candidate pools stay those of a live trace.
"""
import math

import numpy as np
import torch

from paper_2606_00539_gb300 import Monitor, sharding
from paper_2606_00539_gb300 import _native as N

DEV = "cuda:0"
EPS = 1e-8
ALPHA, BETA = 1.1, 1.3
FORMATS = {1: (N.GNMR_FQ_E2M1, 6.0), 2: (N.GNMR_FQ_E3M2, 28.0), 3: (N.GNMR_FQ_E4M3, 448.0),
           4: (N.GNMR_FQ_E5M2, 57344.0)}
# mantissa bits and smallest normal exponent of the OCP minifloats above
GRID = {1: (1, 0), 2: (2, -2), 3: (3, -6), 4: (2, -14)}


def listed():
    return [
        # A small model's tensors: a few MB of fp32 gradients, where launches
        # and latency count.  The `tiny` workload's layout.
        dict(name="step-tiny", op="step", layout="loguniform", units=64, lo=1024, hi=65536, dtype="f32",
             align=16, window=8, max_o=4, lock_len=5, spike=0.05, arenas=4, policy=0, layout_seed=1),
        # Low-rank adapter gradients of a 40-layer model (rank 16, seven
        # linears a layer, two factors each): 560 small tensors, 125 MB.
        dict(name="step-adapters", op="step", layout="adapters", layers=40, hidden=5120, ffn=13824, rank=16,
             dtype="bf16", align=16, window=5, max_o=16, lock_len=10, spike=0.02, arenas=4, policy=0, layout_seed=2),
        # The 24-layer 1.3B layout, one unit per linear: an ordinary full-training step.
        dict(name="step-1.3b", op="step", layout="linears", layers=24, hidden=2048, ffn=5504, dtype="bf16",
             align=16, window=8, max_o=8, lock_len=10, spike=0.02, arenas=3, policy=0, layout_seed=3),
        # The 40-layer 13B layout: the largest step.
        dict(name="step-13b", op="step", layout="linears", layers=40, hidden=5120, ffn=13824, dtype="bf16",
             align=16, window=5, max_o=16, lock_len=10, spike=0.02, arenas=2, policy=0, layout_seed=4),
        # Mixture of experts, four layers of the `moe` workload with one unit
        # per expert (three tensors each), 30 % of the experts unrouted,
        # the admission cap, and the memory cost statistic.
        dict(name="step-moe-experts", op="step", layout="experts", layers=4, hidden=2048, ffn=1408, experts=66,
             dtype="bf16", align=16, window=8, max_o=16, lock_len=8, spike=0.02, unrouted=0.3, arenas=3, policy=1,
             layout_seed=5),
        # 100K units under contention: the `aq-stress` workload's layout.
        dict(name="step-100k", op="step", layout="loguniform", units=100000, lo=256, hi=16384, dtype="f32",
             align=16, window=8, max_o=64, lock_len=3, spike=0.05, arenas=4, policy=0, layout_seed=6),
        # Biases, norm gains and other short tensors of a bf16 flat buffer
        # packed without padding: odd lengths, odd starts.
        dict(name="step-short-packed", op="step", layout="loguniform", units=30000, lo=48, hi=4096, dtype="bf16",
             align=2, window=8, max_o=32, lock_len=3, spike=0.05, arenas=4, policy=0, layout_seed=7),
        # One of eight ranks holding a contiguous slice of the 1.3B gradients.
        dict(name="shard-1.3b", op="shard", layout="linears", layers=24, hidden=2048, ffn=5504, dtype="bf16",
             align=2, window=8, max_o=8, lock_len=10, spike=0.02, arenas=4, policy=0, world=8, rank=3, layout_seed=8),
        # The allocation-free norms over a few thousand mid-sized fp32 units.
        dict(name="norms-static", op="norms", layout="loguniform", units=3000, lo=512, hi=262144, dtype="f32",
             align=16, spike=0.05, layout_seed=9),
        # The actuator over the inputs of every linear of the 13B layout, 1024 tokens.
        dict(name="act-13b", op="act", layout="linears", layers=40, hidden=5120, ffn=13824, tokens=1024,
             dtype="bf16", low=1, rec=3, active=0.06, layout_seed=10),
        # The same for a 130M model (hidden 768), 2048 tokens: short rows.
        dict(name="act-130m", op="act", layout="linears", layers=12, hidden=768, ffn=2048, tokens=2048,
             dtype="bf16", low=1, rec=3, active=0.06, layout_seed=11),
        # One layer's experts, each with its own share of the tokens, in fp32:
        # few and uneven rows, a call of a few microseconds.
        dict(name="act-experts", op="act", layout="routed", experts=64, hidden=1408, tokens=1024,
             dtype="f32", low=2, rec=4, active=0.1, layout_seed=12),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = dict(layout_seed=rng.randrange(1 << 30), dtype=rng.choice(["bf16", "f32"]))
    kind = rng.choice(["units", "units", "linears", "adapters", "experts", "shard", "norms", "act", "act", "routed"])
    eb = 2 if c["dtype"] == "bf16" else 4
    step = dict(op="step", align=rng.choice([eb, 16]), window=rng.choice([3, 5, 8, 13]), max_o=_log(rng, 2, 64),
                lock_len=rng.randint(1, 10), spike=rng.choice([0.01, 0.02, 0.05]), arenas=3, policy=rng.choice([0, 0, 1]))
    if kind in ("units", "norms"):
        lo = _log(rng, 48, 2048)
        c.update(layout="loguniform", lo=lo, hi=lo * rng.choice([8, 64]))
        mean = (c["hi"] - lo) / math.log(c["hi"] / lo)
        c.update(units=_log(rng, 33, min(100000, 4e8 / mean)))
        c.update(step if kind == "units" else dict(op="norms", align=step["align"], spike=step["spike"]))
    elif kind in ("linears", "shard"):
        hidden = 64 * _log(rng, 4, 64)
        c.update(step, layout="linears", layers=rng.randint(4, 24), hidden=hidden, ffn=hidden * 8 // 3 + rng.randint(0, 9))
        if kind == "shard":
            world = rng.choice([2, 4, 8])
            c.update(op="shard", world=world, rank=rng.randrange(world), policy=0)
    elif kind == "adapters":
        hidden = 64 * _log(rng, 8, 80)
        c.update(step, layout="adapters", layers=rng.randint(8, 40), hidden=hidden, ffn=hidden * 8 // 3 // 2 * 2,
                 rank=rng.choice([4, 8, 16, 32]))
    elif kind == "experts":
        c.update(step, layout="experts", layers=rng.randint(1, 4), hidden=64 * _log(rng, 4, 32), ffn=64 * _log(rng, 4, 22),
                 experts=rng.randint(8, 66), unrouted=0.3)
    elif kind == "act":
        hidden = 32 * _log(rng, 4, 160)
        c.update(op="act", layout="linears", layers=rng.randint(1, 24), hidden=hidden, ffn=hidden * 8 // 3 + rng.randint(0, 9),
                 tokens=_log(rng, 16, 1024), low=rng.choice([1, 2]), rec=rng.choice([3, 4]), active=0.06)
    else:
        c.update(op="act", layout="routed", experts=rng.randint(8, 128), hidden=_log(rng, 96, 6000), tokens=_log(rng, 64, 8192),
                 low=rng.choice([1, 2]), rec=rng.choice([3, 4]), active=0.1)
    return c


# -- layouts ------------------------------------------------------------------

def _elem(case):
    return 2 if case["dtype"] == "bf16" else 4


def _torch_dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _lengths(case):
    """(segment lengths, unit of each segment or None)."""
    if case["layout"] == "loguniform":
        rng = np.random.default_rng([case["layout_seed"], 1])
        u = rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["units"])
        return np.round(np.exp(u)).astype(np.int64), None
    d, f = case["hidden"], case["ffn"]
    if case["layout"] == "experts":
        lens, unit = [], []
        for layer in range(case["layers"]):
            u = layer * (case["experts"] + 1)
            lens += [d * d] * 4 + [f * d] * (3 * case["experts"])
            unit += [u] * 4 + [u + 1 + e for e in range(case["experts"]) for _ in range(3)]
        return np.array(lens, np.int64), np.array(unit, np.int32)
    shapes = [(d, d)] * 4 + [(f, d), (f, d), (d, f)]
    if case["layout"] == "adapters":
        one = [n for o, i in shapes for n in (case["rank"] * i, o * case["rank"])]
    else:
        one = [o * i for o, i in shapes]
    return np.array(one * case["layers"], np.int64), None


def _offsets(lens, align):
    step = -(-lens // align) * align
    return np.concatenate([[0], np.cumsum(step)[:-1]]).astype(np.int64), int(step.sum())


def _layout(case):
    """(offsets, lengths, unit of each segment or None, units, arena elements)
    of the arena that the call reads: for a shard, the rank's slice."""
    lens, unit = _lengths(case)
    off, total = _offsets(lens, case["align"] // _elem(case))
    if case["op"] == "shard":
        start, count = sharding.even_shards(total, case["world"])[case["rank"]]
        off, lens = sharding.shard_layout(off, lens, start, count)
        total = count
    return off, lens, unit, len(lens) if unit is None else int(unit.max()) + 1, total


def _gradients(off, lens, scale, total, dtype, g):
    """A flat arena whose segment s holds scale[s] * N(0, 1)."""
    if len(lens) <= 2048:
        arena = torch.zeros(total, dtype=dtype, device=DEV)
        for o, n, s in zip(off.tolist(), lens.tolist(), scale.tolist()):
            if n:
                arena[o:o + n].normal_(0.0, s, generator=g)
        return arena
    ends = np.append(off[1:], total)
    per = torch.repeat_interleave(torch.from_numpy(scale.astype(np.float32)).to(DEV),
                                  torch.from_numpy(ends - off).to(DEV), output_size=total)
    return per.mul_(torch.randn(total, device=DEV, generator=g)).to(dtype)


def _trace(case, seed, lens, unit, units):
    """What the training run brings: the units' sums of squares at the steps
    already observed [window + 3, U], and the segments' scales in each arena."""
    rng = np.random.default_rng([seed, case["layout_seed"]])
    of = np.arange(len(lens)) if unit is None else unit
    level = np.exp(rng.standard_normal(units))
    steps, arenas = case.get("window", 1) + 3, case.get("arenas", 1)
    walk = np.exp(np.cumsum(0.01 * rng.standard_normal((steps + arenas, units)), axis=0))
    hit = rng.random((steps + arenas, units)) < case["spike"]
    factor = np.exp(rng.uniform(math.log(4.0), math.log(1000.0), (steps + arenas, units)))
    s = level * walk * np.where(hit, factor, 1.0)
    if case.get("unrouted"):
        s[(rng.random(s.shape) < case["unrouted"]) & (np.arange(units) % (case["experts"] + 1) != 0)] = 0.0
    count = np.bincount(of, weights=lens, minlength=units)
    return s[:steps] ** 2 * count, s[steps:][:, of]


def _costs(case, units):
    return np.linspace(1.0, 2.0, units) if case["policy"] == 1 else None


def _act_layout(case):
    """(offsets, rows, cols, total elements) of the saved activations."""
    if case["layout"] == "routed":
        rng = np.random.default_rng([case["layout_seed"], 2])
        rows = rng.multinomial(case["tokens"] * 2, rng.dirichlet(np.ones(case["experts"]))).astype(np.int64)
        cols = np.full(case["experts"], case["hidden"], np.int64)
    else:
        one = [case["hidden"]] * 6 + [case["ffn"]]
        cols = np.array(one * case["layers"], np.int64)
        rows = np.full(len(cols), case["tokens"], np.int64)
    off, total = _offsets(rows * cols, 16 // _elem(case))
    return off, rows, cols, total


def _act_inputs(case, seed, units, total):
    g = torch.Generator(DEV).manual_seed(seed)
    x = torch.empty(total, dtype=_torch_dtype(case), device=DEV).normal_(0.0, 1.0, generator=g)
    # a few channels far above the rest, as activations have them
    x[torch.randint(0, total, (max(1, total // 5000),), device=DEV, generator=g)] *= 20.0
    mask = (torch.rand(units, device=DEV, generator=g) < case["active"]).to(torch.uint8)
    return x, mask


# -- the passes -----------------------------------------------------------------

class _Actuator:
    def __init__(self, off, rows, cols, dtype):
        self.h = N.gnmr_actuator_create(off, rows, cols, dtype, 0)

    def __del__(self):
        N.gnmr_actuator_destroy(self.h)


def prepare(case, seed):
    code = N.GNMR_DTYPE_BF16 if case["dtype"] == "bf16" else N.GNMR_DTYPE_F32
    if case["op"] == "act":
        off, rows, cols, total = _act_layout(case)
        x, mask = _act_inputs(case, seed, len(off), total)
        return dict(op="act", act=_Actuator(off, rows, cols, code), x=x, mask=mask, out=torch.zeros_like(x),
                    low=FORMATS[case["low"]][0], rec=FORMATS[case["rec"]][0])
    off, lens, unit, units, total = _layout(case)
    sums, scales = _trace(case, seed, lens, unit, units)
    g = torch.Generator(DEV).manual_seed(seed)
    arenas = [_gradients(off, lens, s, total, _torch_dtype(case), g) for s in scales]
    if case["op"] == "norms":
        return dict(op="norms", arena=arenas[0], code=code, off=off, lens=lens,
                    out=torch.zeros(units, dtype=torch.float64, device=DEV))
    more = {} if unit is None else dict(segment_unit=unit, num_units=units)
    mon = Monitor(off, lens, dtype=case["dtype"], window=case["window"], max_o=case["max_o"],
                  lock_len=case["lock_len"], alpha=ALPHA, beta=BETA, eps=EPS, policy=case["policy"],
                  unit_cost=_costs(case, units), **more)
    for row in sums:
        mon.finish(torch.from_numpy(row).to(DEV))
    stats = mon.new_stats()
    mask = torch.zeros(units, dtype=torch.uint8, device=DEV)
    state = dict(op=case["op"], mon=mon, stats=stats, mask=mask, arenas=arenas, at=0)
    if case["op"] == "step":
        state["steps"] = [mon.prepare_step(a, mask=mask, stats=stats) for a in arenas]
    else:
        state["sumsq"] = torch.zeros(units, dtype=torch.float64, device=DEV)
    return state


def run(state):
    if state["op"] == "act":
        x = state["x"]
        N.gnmr_actuator_apply(state["act"].h, x.data_ptr(), state["out"].data_ptr(), x.numel(),
                              state["mask"].data_ptr(), state["low"], state["rec"],
                              torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if state["op"] == "norms":
        status = N.load().gnmr_unit_norms_static(
            state["arena"].data_ptr(), state["arena"].numel(), state["code"], len(state["off"]),
            state["off"].ctypes.data, state["lens"].ctypes.data, state["out"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        if status != N.GNMR_OK:
            raise RuntimeError(N.last_error(None))
        return state["out"]
    at = state["at"]
    state["at"] = (at + 1) % len(state["arenas"])
    if state["op"] == "step":
        mask = state["steps"][at]()
        return {"mask": mask, **state["stats"]}
    sums = state["mon"].step_partials(state["arenas"][at], sumsq=state["sumsq"])
    mask = state["mon"].finish(sums, mask=state["mask"], stats=state["stats"])
    return {"sumsq": sums, "mask": mask, **state["stats"]}


# -- what a pass cannot do without ------------------------------------------------

def work(case):
    if case["op"] == "act":
        _, rows, cols, _ = _act_layout(case)
        n = int((rows * cols).sum())
        return {"bytes": 2 * n * _elem(case), "flops": 4 * n}
    off, lens, unit, units, total = _layout(case)
    n = int(lens.sum())
    if case["op"] == "norms":
        return {"bytes": n * _elem(case) + 8 * units, "flops": 2 * n}
    # per unit: 40 bytes of controller state read and written, the window read
    # and one entry of it written, the mask, four fp64 statistics and the lock
    per = 80 + 8 * case["window"] + 8 + 1 + 4 * 8 + 4
    per += 16 if case["op"] == "shard" else 0
    return {"bytes": n * _elem(case) + per * units, "flops": 2 * n + 12 * units}


def tolerance(case):
    # The actuator's arithmetic is fixed to fp32 element by element, and every
    # bit of it with it.  (Against 64 bits it is up to 1e-2 off: bf16 values
    # often lie on the midpoint of two codes, and the rounding of the row's
    # scale factor to fp32 decides to which side they go.)
    if case["op"] == "act":
        return "exact"
    # fp32 sums of squares, joined without loss per lane and in fp32 over the
    # lanes: measured up to 3e-8 against 64 bits over all units of a case;
    # a single unit's few roundings in another order are up to 3e-7.
    return {"rel": 2e-7, "max": 2e-6, "differ": 0.0}


# -- the same in 64 bits ----------------------------------------------------------

def _sums_exact(arena, off, lens):
    if len(lens) <= 2048:
        out = torch.zeros(len(lens), dtype=torch.float64, device=DEV)
        for s, (o, n) in enumerate(zip(off.tolist(), lens.tolist())):
            if n:
                out[s] = arena[o:o + n].double().square().sum()
        return out.cpu().numpy()
    sq = arena.double().square_()
    ends = np.append(off[1:], arena.numel())
    parts = np.stack([lens, ends - off - lens], axis=1).reshape(-1)      # segment, gap, segment, gap, ...
    got = torch.segment_reduce(sq, "sum", lengths=torch.from_numpy(parts).to(DEV), initial=0.0)
    return got[::2].cpu().numpy()


class _Controller:
    """Algorithms 1 and 2 on arrays, in 64 bits."""

    def __init__(self, case, units):
        self.c, self.k = case, 0
        self.mean = np.zeros(units)
        self.queue = np.zeros((0, units))
        self.lock = np.zeros(units, np.int32)
        self.active = np.zeros(units, bool)
        self.cost = _costs(case, units)

    def step(self, sums):
        c, n = self.c, np.sqrt(sums)
        first = (self.mean == 0.0) | (self.k == 0)
        g = np.where(first, 1.0, n / np.where(first, 1.0, self.mean + EPS))
        d = g / (self.queue.mean(axis=0) + EPS) if len(self.queue) == c["window"] else np.ones_like(g)
        self.k += 1
        self.mean = self.mean + (n - self.mean) / self.k
        self.queue = np.concatenate([self.queue, g[None]])[-c["window"]:]
        r = np.maximum(g / ALPHA, d / BETA)
        cand = np.flatnonzero((r > 1.0) | (self.lock > 0))
        kept = cand[self.active[cand]] if c["policy"] == 1 else cand[:0]
        pool = np.setdiff1d(cand, kept)
        new = pool[np.lexsort((pool, -r[pool]))][:c["max_o"]]
        chosen = np.concatenate([kept, new])
        lock = np.zeros_like(self.lock)
        lock[chosen] = np.where(r[chosen] > 1.0, c["lock_len"], np.maximum(self.lock[chosen] - 1, 0))
        self.lock = lock
        self.active = np.zeros_like(self.active)
        self.active[chosen] = True
        cost = self.cost[self.active].sum() if self.cost is not None else 0.0
        return {"mask": self.active.astype(np.uint8), "norm": n, "gnmr": g, "dgnmr": d, "risk": r, "lock": lock,
                "counts": np.array([len(cand), len(chosen)], np.int32), "delta_mem": np.array([cost])}


def _quantize_exact(x, code):
    """Per-token fake quantization of the rows of x (64 bits)."""
    top, (bits, low) = FORMATS[code][1], GRID[code]
    amax = x.abs().amax(dim=1, keepdim=True)
    inv = torch.where(amax > 0, top / amax, torch.zeros_like(amax))
    y = x * inv
    e = torch.frexp(y)[1].sub_(1).clamp_(min=low).sub_(bits).to(torch.float64)
    ulp = torch.exp2(e)
    return (y.div_(ulp).round_().mul_(ulp).clamp_(-top, top)).mul_(amax / top)


def exact(case, seed):
    if case["op"] == "act":
        off, rows, cols, total = _act_layout(case)
        x, mask = _act_inputs(case, seed, len(off), total)
        out = torch.zeros(total, dtype=torch.float64, device=DEV)
        for o, r, n, m in zip(off.tolist(), rows.tolist(), cols.tolist(), mask.tolist()):
            if r:
                part = x[o:o + r * n].view(r, n).double()
                out[o:o + r * n] = _quantize_exact(part, case["rec"] if m else case["low"]).view(-1)
        return out
    off, lens, unit, units, total = _layout(case)
    sums, scales = _trace(case, seed, lens, unit, units)
    g = torch.Generator(DEV).manual_seed(seed)
    arena = _gradients(off, lens, scales[0], total, _torch_dtype(case), g)
    got = _sums_exact(arena, off, lens)
    if case["op"] == "norms":
        return np.sqrt(got)
    if unit is not None:
        got = np.bincount(unit, weights=got, minlength=units)
    ctl = _Controller(case, units)
    for row in sums:
        ctl.step(row)
    res = ctl.step(got)
    return {"sumsq": got, **res} if case["op"] == "shard" else res
