// Work partition of the step kernel (host only).
//
// The gradient of a unit is one or more segments of the arena (a transformer
// block spans several weight tensors).  Segments are ordered by unit, and the
// segments of all units are concatenated into one stream of "points": a
// segment of L elements contributes max(L, 1) points (a unit with no element
// still needs one warp to run its Algorithm 1 update).  A unit costs
// kUnitCostBytes plus the bytes of its segments.  The stream is cut into runs
// of about equal cost, so skewed sizes (a 256-element unit next to a
// 70M-element one) balance across the grid: large segments are split over
// many runs, small ones are packed many to a run.  The small-unit loop gives
// every warp one run; the large-unit loop plans several runs per warp, which
// the warps take in turn.
//
// Cuts inside a segment fall on multiples of kSplitBytes from its start, so
// the body of every piece keeps the segment's 16-byte alignment.  Runs are
// strictly increasing and never empty, and a unit's segments are contiguous in
// the stream, so the runs that touch a unit are a contiguous range
// first_run[b] .. first_run[b] + num_parts[b] - 1; the kernel stores the
// partial sum of run r for unit b in slot part_base[b] + (r - first_run[b]),
// so the reduction order of a unit is fixed by the plan (whichever warp
// streams a run) and results are bitwise reproducible run to run.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "gnmr_internal.h"

namespace gnmr {

namespace {

struct Point {
    int64_t seg;
    int64_t pos;
    bool operator<(const Point &o) const { return seg != o.seg ? seg < o.seg : pos < o.pos; }
};

}  // namespace

bool plan_partition(int64_t num_segments, const int64_t *seg_lengths, const int32_t *seg_unit,
                    int32_t num_units, int elem_bytes, int32_t max_runs, Plan &out, const std::vector<int64_t> *targets)
{
    if (num_segments < 1 || num_units < 1 || !seg_lengths || !seg_unit ||
        (elem_bytes != 2 && elem_bytes != 4) || max_runs < 1)
        return false;
    const int64_t S = num_segments, U = num_units;
    // segments must be grouped by unit, every unit present
    for (int64_t g = 0; g < S; ++g) {
        const int64_t u = seg_unit[g];
        if (u < 0 || u >= U || (g > 0 && u < seg_unit[g - 1]) || (g > 0 && u > seg_unit[g - 1] + 1) ||
            (g == 0 && u != 0))
            return false;
    }
    if (seg_unit[S - 1] != U - 1)
        return false;

    std::vector<int64_t> cstart(S + 1, 0);     // cost at the start of segment g
    for (int64_t g = 0; g < S; ++g) {
        const int64_t L = seg_lengths[g];
        if (L < 0 || L > (INT64_MAX / 8) / elem_bytes)
            return false;
        const bool first = g == 0 || seg_unit[g] != seg_unit[g - 1];
        const int64_t cost = (first ? kUnitCostBytes : 0) + std::max<int64_t>(L, 1) * elem_bytes;
        if (cstart[g] > INT64_MAX / 2 - cost)
            return false;
        cstart[g + 1] = cstart[g] + cost;
    }
    const int64_t total = cstart[S];
    const int64_t want = (total + kMinRunBytes - 1) / kMinRunBytes;
    const int64_t W = targets ? int64_t(targets->size()) + 1 : std::max<int64_t>(1, std::min<int64_t>(want, max_runs));
    const int64_t align = std::max<int64_t>(1, kSplitBytes / elem_bytes);

    std::vector<Point> cuts;
    cuts.reserve(W + 1);
    cuts.push_back({0, 0});
    for (int64_t w = 1; w < W; ++w) {
        const int64_t target = targets ? (*targets)[w - 1] : (int64_t)((__int128)total * w / W);
        // segment g with cstart[g] <= target < cstart[g + 1]
        int64_t g = (int64_t)(std::upper_bound(cstart.begin(), cstart.end(), target) - cstart.begin()) - 1;
        g = std::min<int64_t>(std::max<int64_t>(g, 0), S - 1);
        const bool first = g == 0 || seg_unit[g] != seg_unit[g - 1];
        const int64_t local = target - cstart[g] - (first ? kUnitCostBytes : 0);
        int64_t pos = local <= 0 ? 0 : (local + elem_bytes - 1) / elem_bytes;
        pos = (pos + align - 1) / align * align;
        Point p{g, pos};
        if (pos >= std::max<int64_t>(seg_lengths[g], 1))
            p = {g + 1, 0};
        if (cuts.back() < p)
            cuts.push_back(p);
    }
    const Point end{S, 0};
    while (!(cuts.back() < end) && cuts.size() > 1)
        cuts.pop_back();
    cuts.push_back(end);

    const int64_t nw = (int64_t)cuts.size() - 1;
    out.num_runs = (int32_t)nw;
    out.run_seg.resize(nw + 1);
    out.run_pos.resize(nw + 1);
    for (int64_t w = 0; w <= nw; ++w) {
        out.run_seg[w] = cuts[w].seg;
        out.run_pos[w] = cuts[w].pos;
    }
    out.first_run.assign(U, -1);
    out.num_parts.assign(U, 0);
    for (int64_t w = 0; w < nw; ++w) {
        const int64_t g0 = cuts[w].seg;
        const int64_t last = cuts[w + 1].pos > 0 ? cuts[w + 1].seg : cuts[w + 1].seg - 1;
        int64_t prev_unit = -1;
        for (int64_t g = g0; g <= last; ++g) {
            const int64_t b = seg_unit[g];
            if (b == prev_unit)
                continue;
            prev_unit = b;
            if (out.first_run[b] < 0)
                out.first_run[b] = (int32_t)w;
            out.num_parts[b] += 1;
        }
    }
    out.part_base.resize(U);
    int64_t acc = 0;
    for (int64_t b = 0; b < U; ++b) {
        if (out.num_parts[b] < 1)
            return false;  // unreachable: every unit holds at least one point
        out.part_base[b] = acc;
        acc += out.num_parts[b];
    }
    out.num_partials = acc;
    return true;
}

// Cost at which each run of a small arena ends, whole units wherever they are
// at most kWholeUnitBytes: a run ends with the unit that takes it to `run`.
static std::vector<int64_t> whole_unit_targets(int64_t num_segments, const int64_t *seg_lengths, const int32_t *seg_unit,
                                               int elem_bytes, int64_t run)
{
    std::vector<int64_t> targets;
    int64_t cost = 0, begin = 0;                             // of the stream so far; of the current run
    for (int64_t g = 0; g < num_segments;) {
        const int32_t u = seg_unit[g];
        int64_t unit = kUnitCostBytes;
        for (; g < num_segments && seg_unit[g] == u; ++g)
            unit += std::max<int64_t>(seg_lengths[g], 1) * elem_bytes;
        const int64_t pieces = (unit + kWholeUnitBytes - 1) / kWholeUnitBytes;
        for (int64_t k = 1; k < pieces; ++k)
            targets.push_back(cost + unit * k / pieces);
        if (pieces > 1)
            begin = targets.back();
        cost += unit;
        if (cost - begin >= run && g < num_segments) {
            targets.push_back(cost);
            begin = cost;
        }
    }
    return targets;
}

// Packs the blocks of each CTA into turns of several short ones, if that saves
// enough turns.  A turn holds blocks of one batch: the longest not yet taken
// sets the lanes per block, and the next longest fill the rest of the warp.
static void group_blocks(BlockPlan &plan, int elem_bytes)
{
    const auto log2_lanes = [&](int32_t elems) {
        int l = 2;
        while (l < 5 && int64_t(elems) * elem_bytes > (int64_t(16) * kGroupVecs << l))
            ++l;
        return l;
    };
    if (plan.block.size() <= 2 * kWarpsPerCta * plan.cta.size())
        return;                                           // at most two turns a warp as it is
    int64_t lanes = 0;                                    // if every turn were full
    for (const Block &b : plan.block)
        lanes += int64_t(1) << log2_lanes(b.elems);
    if (lanes > 32 * kGroupedShare * plan.block.size())
        return;
    std::vector<Block> turns;
    std::vector<CtaBlocks> cta = plan.cta;
    turns.reserve(static_cast<size_t>(kGroupedShare * plan.block.size()) * kItemBlocks);
    std::vector<Block> batch;
    for (CtaBlocks &c : cta) {
        c.turn = static_cast<int32_t>(turns.size() / kItemBlocks);
        for (int32_t i = 0; i < c.count;) {
            batch.clear();
            const uint32_t k = plan.block[c.first + i].where % (1u << kSlotShift);
            for (; i < c.count && plan.block[c.first + i].where % (1u << kSlotShift) == k; ++i)
                batch.push_back(plan.block[c.first + i]);
            // (equal lengths in the order of their slots: the plan is a function of the layout)
            std::sort(batch.begin(), batch.end(), [](const Block &x, const Block &y) {
                return x.elems != y.elems ? x.elems > y.elems : x.where < y.where;
            });
            for (size_t j = 0; j < batch.size();) {
                const int l = log2_lanes(batch[j].elems);
                const size_t n = std::min<size_t>(batch.size() - j, size_t(32) >> l);
                for (size_t m = 0; m < size_t(kItemBlocks); ++m) {
                    Block b = m < n ? batch[j + m] : Block{0, -1, 0};
                    b.where = b.where % (1u << kLanesShift) | static_cast<uint32_t>(l) << kLanesShift;
                    turns.push_back(b);
                }
                j += n;
            }
        }
        c.turns = static_cast<int32_t>(turns.size() / kItemBlocks) - c.turn;
    }
    if (turns.size() / kItemBlocks > kGroupedShare * plan.block.size() || turns.size() > size_t(INT32_MAX / 2))
        return;
    plan.cta = std::move(cta);
    plan.block = std::move(turns);
    plan.grouped = true;
}

// Blocks: the pieces of one segment that a CTA's warps take in turn.  The sums
// of a CTA's blocks live in its shared memory, kBlocksPerCta of them at most:
// larger blocks first, then more CTAs than are resident, make room.
bool plan_blocks(int64_t num_segments, const int64_t *seg_offsets, const int64_t *seg_lengths,
                 const int32_t *seg_unit, int32_t num_units, int elem_bytes, int32_t max_ctas, Plan &out,
                 BlockPlan &blocks)
{
    if (num_segments < 1 || !seg_offsets || !seg_lengths || !seg_unit || max_ctas < 1)
        return false;
    int64_t cost = int64_t(num_units) * kUnitCostBytes;
    for (int64_t g = 0; g < num_segments; ++g) {
        if (seg_lengths[g] < 0 || seg_lengths[g] > (INT64_MAX / 8) / elem_bytes ||
            cost > INT64_MAX / 2 - seg_lengths[g] * elem_bytes)
            return false;
        cost += seg_lengths[g] * elem_bytes;
    }
    int64_t ctas = std::min<int64_t>(max_ctas, std::max<int64_t>(1, cost / kMinCtaBytes));
    std::vector<int64_t> targets;
    bool cut_at = cost <= max_ctas * kSmallArenaCtaBytes;    // the runs end at `targets`
    if (cut_at)
        targets = whole_unit_targets(num_segments, seg_lengths, seg_unit, elem_bytes, std::max(kMinCtaBytes, cost / max_ctas));
    const int64_t granule = kSplitBytes / elem_bytes;
    // Few long units per CTA: blocks that make whole turns of its warps.
    const int64_t share = cost / ctas / kWarpsPerCta;
    const bool even = !cut_at && cost / num_units >= kEvenUnitBytes && share >= kMinBlockBytes;
    const int64_t rounds = (share + kEvenBlockBytes - 1) / kEvenBlockBytes;
    for (int64_t bytes = even ? (share + rounds - 1) / rounds : kMinBlockBytes;;) {
        if (ctas > INT32_MAX / 2 || !plan_partition(num_segments, seg_lengths, seg_unit, num_units, elem_bytes,
                                                    static_cast<int32_t>(ctas), out, cut_at ? &targets : nullptr))
            return false;
        blocks.cta.clear();
        blocks.block.clear();
        blocks.block.reserve(static_cast<size_t>(std::min(num_segments + cost / bytes + out.num_runs,
                                                          int64_t(kBlocksPerCta) * out.num_runs)));
        blocks.unit_block.assign(num_units + 1, 0);
        bool fits = true;
        int32_t prev_unit = -1;
        for (int32_t r = 0; r < out.num_runs && fits; ++r) {
            CtaBlocks c{};
            c.first = static_cast<int32_t>(blocks.block.size());
            c.unit = seg_unit[out.run_seg[r]];
            int64_t pos = out.run_pos[r];
            for (int64_t g = out.run_seg[r]; g < out.run_seg[r + 1] || (g == out.run_seg[r + 1] && pos < out.run_pos[r + 1]);
                 ++g, pos = 0) {
                const int64_t stop = g == out.run_seg[r + 1] ? std::min(out.run_pos[r + 1], seg_lengths[g]) : seg_lengths[g];
                const int64_t n = std::max<int64_t>(stop - pos, 0);
                const int32_t u = seg_unit[g];
                if (u != prev_unit)
                    blocks.unit_block[u] = static_cast<int32_t>(blocks.block.size());
                prev_unit = u;
                // equal pieces of whole granules; an empty segment is one empty piece
                const int64_t pieces = n * elem_bytes <= bytes ? 1 : (n * elem_bytes + (even ? bytes / 2 : bytes - 1)) / bytes;
                const int64_t per = pieces == 1 ? n : ((n + pieces - 1) / pieces + granule - 1) / granule * granule;
                int64_t at = 0;
                do {
                    const int64_t m = std::min(std::max<int64_t>(per, 1), n - at);
                    const uint32_t slot = static_cast<uint32_t>(blocks.block.size() - c.first) % (1u << (kLanesShift - kSlotShift));
                    blocks.block.push_back({seg_offsets[g] + pos + at, static_cast<int32_t>(m),
                                            static_cast<uint32_t>((u - c.unit) / kBatch) % (1u << kSlotShift) |
                                                slot << kSlotShift | 5u << kLanesShift});
                    at += m;
                } while (at < n);
                c.units = u - c.unit + 1;
                if (blocks.block.size() - c.first > size_t(kBlocksPerCta) || blocks.block.size() > size_t(INT32_MAX / 2)) {
                    fits = false;
                    break;
                }
            }
            c.count = static_cast<int32_t>(blocks.block.size()) - c.first;
            c.turn = c.first;
            c.turns = c.count;
            for (int e = 0; e < 2; ++e) {
                const int32_t u = e == 0 ? c.unit : c.unit + c.units - 1;
                c.parts[e] = out.num_parts[u];
                c.slot[e] = r - out.first_run[u];
                c.base[e] = out.part_base[u];
            }
            blocks.cta.push_back(c);
        }
        if (fits) {
            blocks.unit_block[num_units] = static_cast<int32_t>(blocks.block.size());
            group_blocks(blocks, elem_bytes);
            return true;
        }
        if (bytes < kMaxBlockBytes) {
            bytes *= 2;
        } else {
            // Equal parts, ever smaller: a block costs two bytes and more, so parts of
            // 4 KB hold few enough however many the segments of a unit.
            ctas = std::max<int64_t>(2 * ctas, out.num_runs + 1);
            int64_t points = int64_t(num_units) * kUnitCostBytes;
            for (int64_t g = 0; g < num_segments; ++g)
                points += std::max<int64_t>(seg_lengths[g], 1) * elem_bytes;
            if (ctas > points)
                return false;                            // unreachable: a run for each byte
            targets.resize(ctas - 1);
            for (int64_t w = 1; w < ctas; ++w)
                targets[w - 1] = static_cast<int64_t>(static_cast<__int128>(points) * w / ctas);
            cut_at = true;
        }
    }
}

}  // namespace gnmr
