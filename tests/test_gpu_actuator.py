"""The recovery actuator on the GPU against the oracle's fake quantization
(App. E.2): every output bit must match, for both dtypes, every format,
mixed per-unit formats chosen by a mask, unaligned rows, special rows, in
place, and with the mask written by gnmr_step."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2606_00539_gb300 import Monitor
from paper_2606_00539_gb300 import _native as N

pytestmark = pytest.mark.gpu

FORMATS = [N.GNMR_FQ_E2M1, N.GNMR_FQ_E3M2, N.GNMR_FQ_E4M3, N.GNMR_FQ_E5M2, N.GNMR_FQ_NONE]


def _layout(rng, U, max_rows=40, max_cols=700, gap=True):
    rows = rng.integers(0, max_rows, U).astype(np.int64)
    cols = rng.integers(1, max_cols, U).astype(np.int64)
    off, pos = [], 0
    for r, c in zip(rows, cols):
        pos += int(rng.integers(0, 5)) if gap else 0          # odd starts on purpose
        off.append(pos)
        pos += int(r * c)
    return np.array(off, np.int64), rows, cols, pos + 3


def _host_bits(t):
    import torch
    t = t.cpu()
    return t.view(torch.int16).numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.numpy()


def _oracle_apply(host_in, off, rows, cols, fmt_of_unit):
    out = host_in.copy()
    for b in range(len(off)):
        n = int(rows[b] * cols[b])
        if n == 0:
            continue
        blk = host_in[off[b]:off[b] + n].reshape(rows[b], cols[b])
        out[off[b]:off[b] + n] = oracle.fake_quant(blk, fmt_of_unit[b]).reshape(-1)
    return out


def _special_rows(x, off, rows, cols):
    """Plant zero, NaN, Inf, -0, huge-range and tiny rows in the first units
    (the tiny row's amax, 1e-37, makes fmax / amax overflow fp32 for E4M3
    and E5M2: that row must come back unchanged, with no NaN)."""
    import torch
    for b, kind in enumerate(["zero", "nan", "inf", "negzero", "wide", "tiny"]):
        if b >= len(off) or rows[b] == 0:
            continue
        s, c = int(off[b]), int(cols[b])
        if kind == "zero":
            x[s:s + c] = 0
        elif kind == "nan":
            x[s + c // 2] = float("nan")
        elif kind == "inf":
            x[s] = float("-inf")
        elif kind == "negzero":
            x[s:s + c] = -0.0
        elif kind == "wide":
            x[s:s + c] = torch.logspace(-30, 30, c, dtype=torch.float32).to(x.dtype) * \
                torch.sign(torch.randn(c)).to(x.dtype)
        else:
            row = torch.randn(c, dtype=torch.float32) * 1e-37
            row[::4] = 0.0
            row[0] = 1e-37
            x[s:s + c] = row.to(x.dtype)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("low,rec", [(N.GNMR_FQ_E2M1, N.GNMR_FQ_E4M3), (N.GNMR_FQ_E3M2, N.GNMR_FQ_E5M2),
                                     (N.GNMR_FQ_E4M3, N.GNMR_FQ_NONE)])
def test_actuator_bit_exact(dtype, low, rec, cuda_device):
    import torch
    rng = np.random.default_rng(low * 10 + rec)
    U = 60
    off, rows, cols, total = _layout(rng, U)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = (torch.randn(total, generator=torch.Generator().manual_seed(3)) *
         torch.exp(torch.randn(total, generator=torch.Generator().manual_seed(4)))).to(tdt)
    _special_rows(x, off, rows, cols)
    d_in = x.to(cuda_device)
    d_out = torch.full_like(d_in, 7.0)
    mask = (rng.random(U) < 0.4).astype(np.uint8)
    d_mask = torch.from_numpy(mask).to(cuda_device)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_BF16 if dtype == "bf16" else N.GNMR_DTYPE_F32, 0)
    try:
        N.gnmr_actuator_apply(h, d_in.data_ptr(), d_out.data_ptr(), total, d_mask.data_ptr(), low, rec)
        torch.cuda.synchronize()
        got = _host_bits(d_out)
        want = _oracle_apply(_host_bits(x), off, rows, cols, [rec if m else low for m in mask])
        covered = np.zeros(total, bool)
        for b in range(U):
            covered[off[b]:off[b] + rows[b] * cols[b]] = True
        g, w_ = got[covered], want[covered]
        same = (g.view(np.uint16 if dtype == "bf16" else np.uint32) ==
                w_.view(np.uint16 if dtype == "bf16" else np.uint32))
        assert same.all(), f"{(~same).sum()} of {same.size} elements differ"
        # bytes outside every unit are untouched
        seven = _host_bits(torch.full((1,), 7.0, dtype=tdt))[0]
        assert np.all(_host_bits(d_out)[~covered] == seven)
        # in place, mask NULL = low-cost everywhere
        N.gnmr_actuator_apply(h, d_in.data_ptr(), d_in.data_ptr(), total, None, low, rec)
        torch.cuda.synchronize()
        want2 = _oracle_apply(_host_bits(x), off, rows, cols, [low] * U)
        g2 = _host_bits(d_in)[covered]
        w2 = want2[covered]
        assert np.array_equal(g2.view(np.uint16 if dtype == "bf16" else np.uint32),
                              w2.view(np.uint16 if dtype == "bf16" else np.uint32))
    finally:
        N.gnmr_actuator_destroy(h)


# Row lengths (in 16-byte vectors) at the edges of every thread group that can
# hold a row (4 to 256 threads of 8 vectors), and past the widest.
GROUP_EDGES = [1, 31, 32, 33, 64, 65, 127, 129, 256, 257, 511, 513, 1023, 1025, 2047, 2048, 2049]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_row_groups_bit_exact(dtype, many, shift, cuda_device):
    """One unit per row length around each group's edge, in tiles that are
    full, one row short and one row long; `many` adds so many rows of 513
    vectors that rows wider than two warps are read twice; `shift` moves the
    output against the input by that many elements (1, 3: rows element by
    element).  Every row is compared, of the many ones a random 64."""
    import torch
    rng = np.random.default_rng(shift)
    per = 8 if dtype == "bf16" else 4
    rows, cols = [], []
    for v in GROUP_EDGES:
        group = max(4, 1 << (-(-v // 8) - 1).bit_length())
        tile = max(1, 256 // group)
        for k, n in enumerate((v * per, v * per + per - 1, v * per + 1)):
            rows.append(min(9, tile) + k - 1)
            cols.append(n)
    if many:
        rows.append(8 * 2 * 8 * torch.cuda.get_device_properties(0).multi_processor_count)
        cols.append(513 * per + 1)
    rows, cols = np.array(rows, np.int64), np.array(cols, np.int64)
    off = np.concatenate([[0], np.cumsum(rows * cols + rng.integers(0, 5, len(rows)))[:-1]]).astype(np.int64)
    total = int(off[-1] + rows[-1] * cols[-1]) + 8
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(cuda_device).manual_seed(7 + shift)
    d_in = torch.empty(total, dtype=tdt, device=cuda_device).normal_(0.0, 1.0, generator=g)
    for b in range(0, len(rows), 4):                       # kept rows among the others
        if rows[b] > 1:
            d_in[off[b]:off[b] + cols[b]] = 0
            d_in[off[b] + cols[b] + cols[b] // 2] = float("nan")
    whole = torch.full((total + 16,), 7.0, dtype=tdt, device=cuda_device)
    d_out = whole[shift:shift + total]
    mask = (np.arange(len(rows)) % 3 == 0).astype(np.uint8)
    d_mask = torch.from_numpy(mask).to(cuda_device)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_BF16 if dtype == "bf16" else N.GNMR_DTYPE_F32, 0)
    try:
        N.gnmr_actuator_apply(h, d_in.data_ptr(), d_out.data_ptr(), total, d_mask.data_ptr(), N.GNMR_FQ_E2M1,
                              N.GNMR_FQ_E5M2)
        torch.cuda.synchronize()
    finally:
        N.gnmr_actuator_destroy(h)
    covered = torch.zeros(total, dtype=torch.bool, device=cuda_device)
    for b in range(len(rows)):
        at, n = int(off[b]), int(cols[b])
        covered[at:at + int(rows[b]) * n] = True
        pick = np.arange(rows[b]) if rows[b] <= 64 else np.sort(rng.choice(rows[b], 64, replace=False))
        if not len(pick):
            continue
        idx = torch.from_numpy((at + pick[:, None] * n + np.arange(n)[None]).reshape(-1)).to(cuda_device)
        x = _host_bits(d_in[idx]).reshape(len(pick), n)
        want = oracle.fake_quant(x, N.GNMR_FQ_E5M2 if mask[b] else N.GNMR_FQ_E2M1)
        got = _host_bits(d_out[idx]).reshape(len(pick), n)
        bits = np.uint16 if dtype == "bf16" else np.uint32
        assert np.array_equal(got.view(bits), want.view(bits)), (b, n, int(rows[b]))
    assert bool((d_out[~covered] == 7.0).all()) and bool((whole[total + shift:] == 7.0).all())


def test_actuator_driven_by_gnmr_step(cuda_device):
    """The mask gnmr_step writes selects each unit's activation format."""
    import torch
    w = workloads.make("llama2-13b", shrink=64, steps=8)
    f = workloads.Filler(w, cuda_device)
    arena = f.new_arena()
    mon = Monitor(w.offsets, w.lengths, device=0, **w.monitor_kwargs())
    rng = np.random.default_rng(1)
    rows = np.full(w.num_units, 32, np.int64)
    cols = (w.lengths // 64).clip(1)
    off = np.concatenate([[0], np.cumsum(rows * cols)[:-1]]).astype(np.int64)
    total = int((rows * cols).sum())
    acts = torch.randn(total, device=cuda_device).to(torch.bfloat16)
    out = torch.empty_like(acts)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_BF16, 0)
    try:
        for t in range(w.steps):
            f.fill(arena, t)
            mask = mon.step(arena)
            N.gnmr_actuator_apply(h, acts.data_ptr(), out.data_ptr(), total, mask.data_ptr(),
                                  N.GNMR_FQ_E2M1, N.GNMR_FQ_E4M3,
                                  torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            m = mask.cpu().numpy()
            want = _oracle_apply(_host_bits(acts), off, rows, cols,
                                 [N.GNMR_FQ_E4M3 if v else N.GNMR_FQ_E2M1 for v in m])
            assert np.array_equal(_host_bits(out), want)
        del rng
    finally:
        N.gnmr_actuator_destroy(h)
        mon.close()


@pytest.mark.parametrize("where", [0, 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_rows_without_elements_take_no_time(where, shift, cuda_device):
    """A unit of 2^58 rows of no columns has nothing to quantize: its rows are
    not walked, and the unit beside it comes out as if it were alone."""
    import torch
    rows, cols = np.array([5, 5], np.int64), np.array([70, 70], np.int64)
    rows[where], cols[where] = 1 << 58, 0
    x = torch.randn(350, device=cuda_device)
    out = torch.zeros(366, device=cuda_device)[shift:shift + 350]
    for counts in (rows, np.where(cols > 0, 0, rows)):    # then nothing at all
        h = N.gnmr_actuator_create(np.zeros(2, np.int64), counts, cols, N.GNMR_DTYPE_F32, 0)
        try:
            N.gnmr_actuator_apply(h, x.data_ptr(), out.data_ptr(), 350, None, N.GNMR_FQ_E2M1, N.GNMR_FQ_E4M3)
            torch.cuda.synchronize()
        finally:
            N.gnmr_actuator_destroy(h)
    want = _oracle_apply(_host_bits(x), np.zeros(1, np.int64), np.array([5]), np.array([70]), [N.GNMR_FQ_E2M1])
    assert np.array_equal(_host_bits(out), want)


def test_actuator_errors(cuda_device):
    import torch
    off = np.array([0, 10], np.int64)
    rows = np.array([2, 3], np.int64)
    cols = np.array([5, 4], np.int64)
    with pytest.raises(N.GnmrError):
        N.gnmr_actuator_create(np.array([-1, 0]), rows, cols, N.GNMR_DTYPE_F32, 0)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_F32, 0)
    x = torch.zeros(22, device=cuda_device)
    try:
        with pytest.raises(N.GnmrError) as ei:
            N.gnmr_actuator_apply(h, x.data_ptr(), x.data_ptr(), 21, None, 1, 3)
        assert ei.value.status == N.GNMR_ERR_LAYOUT
        with pytest.raises(N.GnmrError) as ei:
            N.gnmr_actuator_apply(h, x.data_ptr(), x.data_ptr(), 22, None, 9, 3)
        assert ei.value.status == N.GNMR_ERR_INVALID_ARG
        N.gnmr_actuator_apply(h, x.data_ptr(), x.data_ptr(), 22, None, 1, 3)
    finally:
        N.gnmr_actuator_destroy(h)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_units_kept_in_place(dtype, cuda_device):
    """In place, a unit without a format keeps its bytes, held rows and rows
    read twice alike, between units that are rounded; a second launch right
    behind the first finds the same groups in step."""
    import torch
    cols = np.array([64, 1000, 3000, 8000, 17_000, 257, 9000, 40_000], np.int64)
    rows = np.array([70, 9, 17, 5, 3, 33, 4, 2], np.int64)
    off = np.concatenate([[0], np.cumsum(rows * cols + 3)[:-1]]).astype(np.int64)
    total = int(off[-1] + rows[-1] * cols[-1])
    g = torch.Generator(cuda_device).manual_seed(3)
    x = torch.randn(total, device=cuda_device, generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    x[off[1]:off[1] + cols[1]] = 0
    x[off[3] + 5] = float("inf")
    host = _host_bits(x.clone())
    mask = (np.arange(len(rows)) % 2).astype(np.uint8)
    d_mask = torch.from_numpy(mask).to(cuda_device)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_BF16 if dtype == "bf16" else N.GNMR_DTYPE_F32, 0)
    try:
        for low, rec in ((N.GNMR_FQ_NONE, N.GNMR_FQ_E4M3), (N.GNMR_FQ_E2M1, N.GNMR_FQ_NONE)):
            N.gnmr_actuator_apply(h, x.data_ptr(), x.data_ptr(), total, d_mask.data_ptr(), low, rec)
            host = _oracle_apply(host, off, rows, cols, [rec if m else low for m in mask])
        torch.cuda.synchronize()
        word = np.uint16 if dtype == "bf16" else np.uint32
        assert np.array_equal(_host_bits(x).view(word), host.view(word))
    finally:
        N.gnmr_actuator_destroy(h)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("most_rows", [1, 3])
@pytest.mark.parametrize("shift", [0, 1])
def test_units_of_few_rows(dtype, most_rows, shift, cuda_device):
    """Units of a few short rows, which warps take one by one: rows of up to a
    warp's 256 vectors, empty units among them, against the oracle."""
    import torch
    rng = np.random.default_rng(most_rows)
    per = 8 if dtype == "bf16" else 4
    cols = np.array([1, per, 33 * per, 64 * per - 1, 129 * per, 256 * per + per - 1, 31] * 40, np.int64)
    rows = rng.integers(0, most_rows + 1, len(cols)).astype(np.int64)
    rows[0] = 1
    off = np.concatenate([[0], np.cumsum(rows * cols + 1)[:-1]]).astype(np.int64)
    total = int(off[-1] + rows[-1] * cols[-1]) + 1
    g = torch.Generator(cuda_device).manual_seed(most_rows)
    x = torch.randn(total, device=cuda_device, generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    x[off[14]:off[14] + rows[14] * cols[14]] = 0
    whole = torch.full((total + 16,), 3.0, dtype=x.dtype, device=cuda_device)
    out = whole[shift:shift + total]
    mask = (np.arange(len(rows)) % 3 == 0).astype(np.uint8)
    d_mask = torch.from_numpy(mask).to(cuda_device)
    h = N.gnmr_actuator_create(off, rows, cols, N.GNMR_DTYPE_BF16 if dtype == "bf16" else N.GNMR_DTYPE_F32, 0)
    try:
        low, rec = N.GNMR_FQ_E2M1, N.GNMR_FQ_E4M3
        N.gnmr_actuator_apply(h, x.data_ptr(), out.data_ptr(), total, d_mask.data_ptr(), low, rec)
        torch.cuda.synchronize()
        want = _oracle_apply(_host_bits(x), off, rows, cols, [rec if m else low for m in mask])
        got = _host_bits(out)
        word = np.uint16 if dtype == "bf16" else np.uint32
        for b in range(len(rows)):
            part = slice(off[b], off[b] + rows[b] * cols[b])
            assert np.array_equal(got[part].view(word), want[part].view(word)), (b, rows[b], cols[b])
        # nothing else is written: not between the units, nor before and behind the buffer
        covered = np.zeros(total + 16, bool)
        for b in range(len(rows)):
            covered[shift + off[b]:shift + off[b] + rows[b] * cols[b]] = True
        assert (whole.float().cpu().numpy()[~covered] == 3.0).all()
    finally:
        N.gnmr_actuator_destroy(h)
