// The small-unit loop's work partition (plan_blocks) behind a C interface, for
// the CPU tests: compiled together with gnmr_plan.cpp into a library of its own.
#include <cstdint>
#include <cstring>

#include "gnmr_internal.h"

static gnmr::Plan g_plan;
static gnmr::BlockPlan g_blocks;

extern "C" {

// Plans a layout; sizes[5]: CTAs, table entries, 1 if grouped, partial slots, entries a turn.
int plan_query(int64_t segments, const int64_t *offsets, const int64_t *lengths, const int32_t *seg_unit,
               int32_t units, int elem_bytes, int32_t max_ctas, int64_t *sizes)
{
    g_plan = gnmr::Plan{};
    g_blocks = gnmr::BlockPlan{};
    if (!gnmr::plan_blocks(segments, offsets, lengths, seg_unit, units, elem_bytes, max_ctas, g_plan, g_blocks))
        return 0;
    sizes[0] = static_cast<int64_t>(g_blocks.cta.size());
    sizes[1] = static_cast<int64_t>(g_blocks.block.size());
    sizes[2] = g_blocks.grouped ? 1 : 0;
    sizes[3] = g_plan.num_partials;
    sizes[4] = g_blocks.grouped ? gnmr::kItemBlocks : 1;
    return 1;
}

// The tables of the last plan.  cta[12] per CTA: first, count, unit, units, turn,
// turns, parts[2], slot[2], base[2]; block[5] per entry: start, elements (-1: none),
// batch, slot and log2 of the lanes; unit_block[units + 1].
void plan_tables(int64_t *cta, int64_t *block, int32_t *unit_block)
{
    for (const gnmr::CtaBlocks &c : g_blocks.cta) {
        const int64_t row[12] = {c.first, c.count, c.unit, c.units, c.turn, c.turns, c.parts[0], c.parts[1],
                                 c.slot[0], c.slot[1], c.base[0], c.base[1]};
        std::memcpy(cta, row, sizeof row);
        cta += 12;
    }
    for (const gnmr::Block &b : g_blocks.block) {
        const int64_t row[5] = {b.start, b.elems, b.where % (1u << gnmr::kSlotShift),
                                (b.where >> gnmr::kSlotShift) % (1u << (gnmr::kLanesShift - gnmr::kSlotShift)),
                                b.where >> gnmr::kLanesShift};
        std::memcpy(block, row, sizeof row);
        block += 5;
    }
    std::memcpy(unit_block, g_blocks.unit_block.data(), sizeof(int32_t) * g_blocks.unit_block.size());
}

}  // extern "C"
