"""The small-unit loop's work partition (plan_blocks, host code): run here as the
step kernel reads it.  Every element of every segment in exactly one block, every
block's sum in a slot of its own in unit order, the blocks a batch waits for equal
to the blocks that count down on it, a unit's parts numbered without a gap, and a
CTA never with more blocks than its shared memory has sums for."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_00539_gb300", "csrc")
CTAS = 304                      # two to each of 152 SMs
CAP, BATCH, WARPS = 2048, 32, 16
MAX_BYTES = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2606_00539_gb300.build import _cuda_home
    so = str(tmp_path_factory.mktemp("plan") / "plan_query.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC,
                    "-I" + os.path.join(_cuda_home(), "include"),
                    os.path.join(ROOT, "tests", "plan_query.cpp"), os.path.join(CSRC, "gnmr_plan.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def _pointer(a):
    return a.ctypes.data_as(ctypes.c_void_p)


class Plan:
    def __init__(self, lib, off, lens, unit=None, eb=2, ctas=CTAS):
        self.off = np.ascontiguousarray(off, np.int64)
        self.lens = np.ascontiguousarray(lens, np.int64)
        self.unit = np.arange(len(lens), dtype=np.int32) if unit is None else np.ascontiguousarray(unit, np.int32)
        self.units, self.eb, self.asked = int(self.unit[-1]) + 1, eb, ctas
        sizes = np.zeros(5, np.int64)
        ok = lib.plan_query(ctypes.c_int64(len(lens)), _pointer(self.off), _pointer(self.lens), _pointer(self.unit),
                            ctypes.c_int32(self.units), ctypes.c_int(eb), ctypes.c_int32(ctas), _pointer(sizes))
        assert ok == 1
        self.cta = np.zeros((sizes[0], 12), np.int64)
        self.block = np.zeros((sizes[1], 5), np.int64)
        self.unit_block = np.zeros(self.units + 1, np.int32)
        lib.plan_tables(_pointer(self.cta), _pointer(self.block), _pointer(self.unit_block))
        self.grouped, self.partials, self.entries = bool(sizes[2]), int(sizes[3]), int(sizes[4])

    @property
    def block_bytes(self):
        return int(self.block[:, 1].max()) * self.eb


def _packed(lens, pad=0):
    return np.concatenate([[0], np.cumsum(np.asarray(lens, np.int64) + pad)[:-1]])


def check(p):
    """Walks the tables as the kernel does."""
    parts = [[] for _ in range(p.units)]
    pieces = []                                           # unit, start, elements
    turn = 0
    for first, count, unit, units, t0, turns, pa0, pa1, sl0, sl1, ba0, ba1 in p.cta.tolist():
        assert 1 <= count <= CAP and 1 <= units <= count and t0 == turn
        turn += turns
        assert p.grouped or turns == count
        b = p.block[t0 * p.entries:(t0 + turns) * p.entries]
        if p.grouped:                                     # a turn's blocks: one batch, one width, enough lanes
            rows = b.reshape(turns, p.entries, 5)
            real = rows[:, :, 1] >= 0
            assert (rows[:, 0, 1] >= 0).all()
            assert ((rows[:, :, 2] == rows[:, :1, 2]) | ~real).all()
            lanes = 1 << rows[:, 0, 4]
            assert (rows[:, :, 4] == rows[:, :1, 4]).all()
            assert (real.sum(1) * lanes <= 32).all()
            assert ((rows[:, :, 1] * p.eb <= 16 * 8 * lanes[:, None]) | (lanes[:, None] == 32) | ~real).all()
            b = b[b[:, 1] >= 0]
        else:
            assert (b[:, 1] >= 0).all() and (b[:, 4] == 5).all()
        assert len(b) == count
        b = b[np.argsort(b[:, 3], kind="stable")]
        assert np.array_equal(b[:, 3], np.arange(count)), "one slot each"
        ends = np.minimum(p.unit_block[unit + 1:unit + units + 1] - first, count)
        begins = np.concatenate([[0], ends[:-1]])
        assert (ends > begins).all() and ends[-1] == count
        owner = np.repeat(np.arange(units), ends - begins)
        assert np.array_equal(b[:, 2], owner // BATCH), "a block counts down its own unit's batch"
        for k in range(0, units, BATCH):                  # the kernel's count of a batch's blocks
            u0, n = unit + k, min(BATCH, units - k)
            lo, hi = p.unit_block[u0] - first, min(p.unit_block[u0 + n] - first, count)
            assert hi - max(lo, 0) == (b[:, 2] == k // BATCH).sum()
        pieces.append(np.stack([owner + unit, b[:, 0], b[:, 1]], 1))
        for i in range(units):
            if i == 0:
                parts[unit].append((pa0, sl0, ba0))
            elif i == units - 1:
                parts[unit + i].append((pa1, sl1, ba1))
            else:
                parts[unit + i].append((1, 0, None))
        if units == 1:
            assert (pa0, sl0, ba0) == (pa1, sl1, ba1)
    used = set()
    for q in parts:
        assert [s for _, s, _ in q] == list(range(len(q))) and all(n == len(q) for n, _, _ in q)
        if len(q) > 1:
            base = q[0][2]
            assert all(x[2] == base for x in q) and 0 <= base and base + len(q) <= p.partials
            assert not used & set(range(base, base + len(q)))
            used |= set(range(base, base + len(q)))
    # every element once: a unit's blocks, in order, are its segments, in order
    got = np.concatenate(pieces)
    got = got[got[:, 2] > 0]
    assert (np.diff(got[:, 0]) >= 0).all()
    full = p.lens > 0
    want = np.stack([p.unit[full], p.off[full], p.lens[full]], 1)
    starts = np.cumsum(got[:, 2]) - got[:, 2]             # places in the stream
    seg0 = np.cumsum(want[:, 2]) - want[:, 2]
    seg = np.searchsorted(seg0, starts, side="right") - 1
    assert got[:, 2].sum() == want[:, 2].sum()
    assert np.array_equal(got[:, 0], want[seg, 0])
    assert np.array_equal(got[:, 1] - want[seg, 1], starts - seg0[seg])
    assert (starts + got[:, 2] <= seg0[seg] + want[seg, 2]).all()
    assert ((got[:, 1] - want[seg, 1]) * p.eb % 512 == 0).all(), "cuts keep the segment's alignment"


def _random_layout(seed):
    rng = np.random.default_rng(seed)
    n = int(rng.integers(1, 4000))
    kind = seed % 6
    if kind == 0:
        lens = rng.integers(0, 5000, n)
    elif kind == 1:
        lens = np.exp(rng.uniform(0, 15, n)).astype(np.int64)
    elif kind == 2:
        lens = np.zeros(n, np.int64)
    elif kind == 3:
        lens = rng.integers(0, 3, n) * rng.integers(1, 10**6, n)
    elif kind == 4:                                       # few large units
        lens = rng.integers(1, 4 * 10**7, max(n // 100, 1))
    else:                                                 # a cluster of tiny segments among large ones
        lens = np.concatenate([rng.integers(0, 4, int(rng.integers(1, 9000))), rng.integers(10**5, 10**6, max(n // 10, 1))])
    unit = None
    if seed % 4 >= 2:                                     # several segments a unit
        unit = np.cumsum(rng.random(len(lens)) < 0.2)
        unit -= unit[0]
    return _packed(lens, seed % 3), lens, unit


@pytest.mark.parametrize("seed", range(36))
def test_plan_of_random_layouts(lib, seed):
    off, lens, unit = _random_layout(seed)
    for eb in (2, 4):
        for ctas in (1, 7, CTAS):
            check(Plan(lib, off, lens, unit, eb, ctas))


@pytest.mark.parametrize("config", [1, 2, 5])
def test_plan_of_workloads(lib, config):
    import workloads
    w = workloads.make(config)
    p = Plan(lib, _packed(w.lengths), w.lengths, None, 2 if w.dtype == "bf16" else 4)
    check(p)
    assert len(p.cta) <= CTAS


def _dense_cluster(tiny, large, length, one_unit=True, where=0):
    """`tiny` segments of one element, in one unit or a unit each, before the
    `where`-th of `large` units of `length` elements."""
    lens = np.concatenate([np.full(where, length), np.ones(tiny, np.int64), np.full(large - where, length)])
    tiny_units = np.zeros(tiny, np.int64) if one_unit else np.arange(tiny)
    unit = np.concatenate([np.arange(where), where + tiny_units, where + tiny_units[-1] + 1 + np.arange(large - where)])
    return _packed(lens), lens, unit


@pytest.mark.parametrize("tiny,large,length,where", [
    (2000, 560, 112_000, 0), (2500, 560, 112_000, 0), (2500, 560, 112_000, 560), (5000, 5000, 400_000, 0),
    (5000, 5000, 400_000, 2500), (20_000, 5000, 400_000, 1)])
def test_a_cluster_of_tiny_segments_leaves_the_rest_as_it_is(lib, tiny, large, length, where):
    """A unit of thousands of one-element segments fills its own CTAs' block
    tables; the ordinary units beside it keep about the parts and the blocks that
    they have without it."""
    p = Plan(lib, *_dense_cluster(tiny, large, length, where=where))
    check(p)
    alone = Plan(lib, _packed(np.full(large, length)), np.full(large, length))
    assert len(alone.cta) <= CTAS
    assert len(p.cta) <= len(alone.cta) + (0 if tiny <= 5000 else CTAS)
    assert p.block_bytes <= 2 * alone.block_bytes
    if tiny <= 5000:                                      # the longest part: a little longer
        def longest(q):
            return max(int(b[:, 1].sum()) for b in np.split(q.block, q.cta[1:, 0]))
        assert longest(p) <= longest(alone) * 17 / 16 + 512


def test_many_tiny_units_beside_few_large_ones(lib):
    """640,000 units of two elements (more than 304 CTAs have block sums for) and
    eight of 64 MiB: the large ones' blocks stay small enough for a CTA's 16 warps."""
    lens = np.concatenate([np.full(640_000, 2), np.full(8, 1 << 25)])
    p = Plan(lib, _packed(lens), lens)
    check(p)
    assert len(p.cta) <= 2 * CTAS
    assert p.block_bytes <= 64 << 10


def test_more_units_than_one_wave_of_ctas_holds(lib):
    lens = np.full(700_000, 7)
    p = Plan(lib, _packed(lens), lens)
    check(p)
    assert len(p.cta) <= 2 * CTAS


def test_plan_refuses_what_it_cannot_number(lib):
    lens = np.full(1, np.iinfo(np.int64).max // 8)
    sizes = np.zeros(5, np.int64)
    off, unit = np.zeros(1, np.int64), np.zeros(1, np.int32)
    assert lib.plan_query(ctypes.c_int64(1), _pointer(off), _pointer(lens), _pointer(unit), ctypes.c_int32(1),
                          ctypes.c_int(2), ctypes.c_int32(CTAS), _pointer(sizes)) == 0


@pytest.mark.parametrize("units,top,eb", [(3000, 60_000, 2), (100_000, 3000, 4), (600, 200_000, 2)])
def test_the_public_query_gives_the_ctas_of_larger_arenas(lib, units, top, eb):
    """gnmr_plan_partition, asked for as many runs as there are resident CTAs,
    lists the CTAs' parts of arenas above 48 KiB of cost per CTA."""
    from paper_2606_00539_gb300 import _native as N
    lens = np.random.default_rng(units).integers(0, top, units).astype(np.int64)
    assert (lens * eb + 4096).sum() > CTAS * (48 << 10)
    p = Plan(lib, _packed(lens), lens, None, eb)
    run_unit, _, first, parts = N.gnmr_plan_partition(lens, N.GNMR_DTYPE_BF16 if eb == 2 else N.GNMR_DTYPE_F32, CTAS)
    assert np.array_equal(run_unit[:-1], p.cta[:, 2])
    for ends, col in ((p.cta[:, 2], 6), (p.cta[:, 2] + p.cta[:, 3] - 1, 7)):
        assert np.array_equal(parts[ends], p.cta[:, col])
        assert np.array_equal(np.arange(len(ends)) - first[ends], p.cta[:, col + 2])


@pytest.mark.parametrize("units,eb,seed", [(300, 2, 1), (300, 4, 2), (500, 2, 3), (40, 4, 4)])
def test_small_arenas_give_no_cta_two_rounds(lib, units, eb, seed):
    """Arenas cut between units: no CTA gets more than 128 KiB, units of that and
    more get CTAs of their own, and there is one wave of CTAs."""
    lens = np.minimum(np.exp(np.random.default_rng(seed).normal(8, 1.8, units)).astype(np.int64), 100_000)
    cost = lens * eb + 4096
    assert cost.sum() <= CTAS * (48 << 10)
    p = Plan(lib, _packed(lens), lens, None, eb)
    check(p)
    assert len(p.cta) <= CTAS
    for c in p.cta:
        b = p.block[c[4] * p.entries:(c[4] + c[5]) * p.entries]
        assert b[b[:, 1] > 0, 1].sum() * eb + 4096 * (c[3] - (c[8] > 0)) <= (128 << 10) + 512
