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
// every CTA one run, which its warps share in blocks (plan_blocks); the
// large-unit loop plans several runs per warp, which the warps take in turn.
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
// at most kWholeUnitBytes: a run ends with the unit that takes it to `run`, or
// before one with which it would pass kWholeUnitBytes, a block for each warp (so
// at most a run for each `run` of cost, if that is half of kWholeUnitBytes or less:
// two such runs hold more than kWholeUnitBytes).  300 log-normal bf16 units, 5 MB,
// whose runs ended with the unit only: 11.7 us, so 10.7; their sums alone 7.4 and
// 5.8, log-normal fp32 ones 6.9 and 5.7.
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
        if (cost > begin && cost - begin + unit / pieces > kWholeUnitBytes) {
            targets.push_back(cost);
            begin = cost;
        }
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

// Blocks of one segment's n elements in a run: equal pieces of whole granules of
// about `bytes`, at most of that size, or with `nearest` as close to it as a whole
// number of them can be.  An empty segment is one empty block.
namespace {
struct BlockRule {
    int64_t bytes, granule;
    int elem_bytes;
    bool nearest;
    int64_t elems(int64_t n) const                       // of each block but the last
    {
        const int64_t size = n * elem_bytes;
        const int64_t pieces = size <= bytes ? 1 : (size + (nearest ? bytes / 2 : bytes - 1)) / bytes;
        return pieces == 1 ? n : ((n + pieces - 1) / pieces + granule - 1) / granule * granule;
    }
    int64_t count(int64_t n) const { return n <= 0 ? 1 : (n + elems(n) - 1) / elems(n); }
};
}  // namespace

// Calls f(segment, first element, elements) for every piece of a segment in run r.
template <typename F>
static void for_run(const Plan &plan, const int64_t *seg_lengths, int32_t r, const F &f)
{
    const int64_t last = plan.run_seg[r + 1], end = plan.run_pos[r + 1];
    int64_t pos = plan.run_pos[r];
    for (int64_t g = plan.run_seg[r]; g < last || (g == last && pos < end); ++g, pos = 0) {
        const int64_t stop = g == last ? std::min(end, seg_lengths[g]) : seg_lengths[g];
        f(g, pos, std::max<int64_t>(stop - pos, 0));
    }
}

static bool every_run_fits(const Plan &plan, const int64_t *seg_lengths, const BlockRule &rule)
{
    for (int32_t r = 0; r < plan.num_runs; ++r) {
        int64_t n = 0;
        for_run(plan, seg_lengths, r, [&](int64_t, int64_t, int64_t elems) { n += rule.count(elems); });
        if (n > kBlocksPerCta)
            return false;
    }
    return true;
}

// Cost at which each run ends if none may cost more than `run` or hold more than
// kBlocksPerCta blocks; at most `limit` targets (one too many: no such runs).
static void bounded_targets(int64_t num_segments, const int64_t *seg_lengths, const int32_t *seg_unit, int elem_bytes,
                            int64_t run, int64_t bytes, int64_t limit, std::vector<int64_t> &targets)
{
    // (the cut falls on a granule, up to one block further on than the target)
    constexpr int64_t kCap = kBlocksPerCta - 2;
    targets.clear();
    int64_t at = 0, begin = 0, held = 0;                     // the stream's cost so far, the run's begin and blocks
    const auto cut = [&](int64_t cost) {
        targets.push_back(cost);
        begin = at = cost;
        held = 0;
    };
    for (int64_t g = 0; g < num_segments && static_cast<int64_t>(targets.size()) < limit; ++g) {
        const bool first = g == 0 || seg_unit[g] != seg_unit[g - 1];
        const int64_t data = at + (first ? kUnitCostBytes : 0);
        const int64_t end = data + std::max<int64_t>(seg_lengths[g], 1) * elem_bytes;
        if (held >= kCap)
            cut(at);
        while (static_cast<int64_t>(targets.size()) < limit) {
            const int64_t room = std::min(begin + run - at, std::max<int64_t>(data - at, 0) + (kCap - held) * bytes);
            if (end - at <= room)
                break;
            cut(at + std::max(room, int64_t(elem_bytes)));
        }
        held += (end - std::max(data, at) + bytes - 1) / bytes;
        at = end;
    }
}

// Cuts the stream into one run per CTA.  The sums of a CTA's blocks live in its
// shared memory, kBlocksPerCta of them at most.  Where equal runs of a large arena
// need more, the blocks get larger, up to those of which half as many would do for
// the bytes alone.  What then still does not fit has too many segments: the runs
// around those are cut shorter and all the others get longer, by at most a quarter;
// only if that does not do there are two runs to a CTA, four, ... (no CTA waits for
// another).  5,000 one-element segments beside 5,000 bf16 units of 400,000 leave 304
// CTAs with parts 1 % longer: 589 us, 555 without those segments.
static bool cut_runs(int64_t num_segments, const int64_t *seg_lengths, const int32_t *seg_unit, int32_t num_units,
                     int64_t cost, int64_t ctas, const std::vector<int64_t> *targets, BlockRule &rule, Plan &out)
{
    const auto plan = [&](int64_t runs, const std::vector<int64_t> *at) {
        return plan_partition(num_segments, seg_lengths, seg_unit, num_units, rule.elem_bytes,
                              static_cast<int32_t>(runs), out, at);
    };
    if (!plan(ctas, targets))
        return false;
    const int64_t least = rule.bytes;
    int64_t most = least;
    while (most < kMaxBlockBytes && (most == least || most / 2 * kBlocksPerCta < cost / ctas))
        most *= 2;
    for (; rule.bytes <= most; rule.bytes *= 2)
        if (every_run_fits(out, seg_lengths, rule))
            return true;
    if (cost / most > INT32_MAX / 2)
        return false;

    int64_t points = int64_t(num_units) * kUnitCostBytes;
    for (int64_t g = 0; g < num_segments; ++g)
        points += std::max<int64_t>(seg_lengths[g], 1) * rule.elem_bytes;
    std::vector<int64_t> cuts;
    for (int64_t runs = ctas; runs <= INT32_MAX / 2; runs *= 2) {
        // the longest run at most a quarter above the mean, and in one round of CTAs the
        // smallest blocks that allow it
        const int64_t mean = (points + runs - 1) / runs;
        const auto cuts_at = [&](int64_t run) {
            bounded_targets(num_segments, seg_lengths, seg_unit, rule.elem_bytes, run, rule.bytes, runs, cuts);
            return static_cast<int64_t>(cuts.size()) < runs;
        };
        rule.bytes = most;
        if (!cuts_at(mean + mean / 4))
            continue;
        if (runs == ctas)
            for (rule.bytes = least; rule.bytes < most && !cuts_at(mean + mean / 4); rule.bytes *= 2) {
            }
        int64_t lo = mean - 1, hi = mean + mean / 4;        // hi will do
        while (hi - lo > 1 + mean / 256) {
            const int64_t mid = lo + (hi - lo) / 2;
            (cuts_at(mid) ? hi : lo) = mid;
        }
        cuts_at(hi);
        if (!plan(static_cast<int64_t>(cuts.size()) + 1, &cuts))
            return false;
        if (every_run_fits(out, seg_lengths, rule))
            return true;
    }
    return false;                                            // unreachable: a block costs two bytes and more
}

// Blocks: the pieces of one segment that a CTA's warps take in turn.
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
    const int64_t ctas = std::min<int64_t>(max_ctas, std::max<int64_t>(1, cost / kMinCtaBytes));
    std::vector<int64_t> targets;
    const bool cut_at = cost <= max_ctas * kSmallArenaCtaBytes;    // the runs end at `targets`
    if (cut_at)
        targets = whole_unit_targets(num_segments, seg_lengths, seg_unit, elem_bytes, std::max(kMinCtaBytes, cost / max_ctas));
    // Few long units per CTA: blocks that make whole turns of its warps.
    const int64_t share = cost / ctas / kWarpsPerCta;
    const bool even = !cut_at && cost / num_units >= kEvenUnitBytes && share >= kMinBlockBytes;
    const int64_t rounds = (share + kEvenBlockBytes - 1) / kEvenBlockBytes;
    BlockRule rule{even ? (share + rounds - 1) / rounds : kMinBlockBytes, kSplitBytes / elem_bytes, elem_bytes, even};
    if (!cut_runs(num_segments, seg_lengths, seg_unit, num_units, cost, ctas, cut_at ? &targets : nullptr, rule, out))
        return false;

    blocks.cta.clear();
    blocks.block.clear();
    blocks.block.reserve(static_cast<size_t>(std::min(num_segments + cost / rule.bytes + out.num_runs,
                                                      int64_t(kBlocksPerCta) * out.num_runs)));
    blocks.unit_block.assign(num_units + 1, 0);
    int32_t prev_unit = -1;
    for (int32_t r = 0; r < out.num_runs; ++r) {
        CtaBlocks c{};
        c.first = static_cast<int32_t>(blocks.block.size());
        c.unit = seg_unit[out.run_seg[r]];
        for_run(out, seg_lengths, r, [&](int64_t g, int64_t pos, int64_t n) {
            const int32_t u = seg_unit[g];
            if (u != prev_unit)
                blocks.unit_block[u] = static_cast<int32_t>(blocks.block.size());
            prev_unit = u;
            const int64_t per = rule.elems(n);
            int64_t at = 0;
            do {
                const int64_t m = std::min(std::max<int64_t>(per, 1), n - at);
                const uint32_t slot = static_cast<uint32_t>(blocks.block.size() - c.first);
                blocks.block.push_back({seg_offsets[g] + pos + at, static_cast<int32_t>(m),
                                        static_cast<uint32_t>((u - c.unit) / kBatch) | slot << kSlotShift | 5u << kLanesShift});
                at += m;
            } while (at < n);
            c.units = u - c.unit + 1;
        });
        if (blocks.block.size() > size_t(INT32_MAX / 2))
            return false;
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
    blocks.unit_block[num_units] = static_cast<int32_t>(blocks.block.size());
    group_blocks(blocks, elem_bytes);
    return true;
}

}  // namespace gnmr
