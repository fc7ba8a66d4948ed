// Internal declarations shared by the host API (gnmr_api.cpp, gnmr_plan.cpp)
// and the device code (gnmr_kernels.cu).  Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime_api.h>

namespace gnmr {

// Launch shape of the step kernel: 512 threads = 16 warps per CTA.  Two
// compiled variants of the streaming loop (gnmr_kernels.cu): kVariantSmall
// (two resident CTAs per SM, each with a part of its own that its warps take
// block by block) for layouts of small and mid-sized units and for small
// arenas (kVariantGroups: the same where short blocks dominate, several of them
// to a warp at a time), kVariantBulk (one CTA per SM, deeper per-warp streams, runs
// taken from a shared counter) for layouts whose mean unit holds at least
// kBulkUnitBytes.
constexpr int kThreads = 512;
constexpr int kWarpsPerCta = kThreads / 32;
constexpr int kVariantSmall = 0;
constexpr int kVariantBulk = 1;
constexpr int kVariantGroups = 2;
constexpr int64_t kBulkUnitBytes = int64_t(1) << 20;
// Below this many gradient bytes the large-unit loop's 64 KiB runs are too few
// to balance: 168 units in 303 MB took 60.7 us with it, 57.9 with blocks; 84 in
// 170 MB 56.3 and 54.4, 84 in 95 MB 43.0 and 37.0.  (607 MB: 100.4 and 98.4; 1.2
// GB: 179.2 and 180.8; 2.4 GB: 333.4 and 336.0.)
constexpr int64_t kBulkArenaBytes = int64_t(512) << 20;
// Controller half: up to 2 kFewUnits units per SM a warp takes kFewUnits units
// (four lanes each in the epilogue), else 32; warps go one to a CTA first, as an
// SM's fp64 pipe serves all of its warps.  From full warps, 16 to a CTA: 168 units
// 8.6 -> 7.2 us, 560 15.3 -> 7.1, 20,000 16.4 -> 8.2, 100,000 28.7 -> 20.6.
constexpr int kFewUnits = 8;

// Work partition: a unit costs its element bytes plus this many bytes of
// equivalent fixed work (reduction, Algorithm 1 update, bookkeeping); runs
// are cut at multiples of kSplitBytes inside a unit, and no run is planned
// smaller than kMinRunBytes unless the whole problem is.
constexpr int64_t kUnitCostBytes = 4096;
constexpr int64_t kSplitBytes = 512;
constexpr int64_t kMinRunBytes = 4096;   // one 4 KiB load round per warp
// Large-unit loop: the stream is cut into about kRunsPerWarp runs per warp of
// kBulkRunMin..kBulkRunMax bytes each.  Each warp starts on its own run and
// then takes the next untaken one, so warps that stream faster take more runs
// and all finish together (static equal runs left the slowest warps ~8 % of
// the step behind the median one).
constexpr int64_t kRunsPerWarp = 16;
constexpr int64_t kBulkRunMin = int64_t(64) << 10;
constexpr int64_t kBulkRunMax = int64_t(256) << 10;

// Small-unit loop: every CTA owns a contiguous part of the segment stream of
// at least kMinCtaBytes of cost, cut into blocks of at most kMinBlockBytes (or
// that doubled, up to kMaxBlockBytes, if a CTA would have more than kBlocksPerCta
// for its bytes alone), which its warps take in turn.  kBatch units are one batch of the unit epilogue.  8 KiB blocks, two
// load rounds of a warp: 4 KiB took 246.8 us on 100K units, 8 KiB 242.9, 16
// KiB 244.2 (560 units of 224 KB: 34.1, 32.7, 31.6).  24 KiB per CTA: 3.7 MB
// over 64 units took 11.9 us with 64 KiB, 11.4 with 24.
constexpr int kBatch = 32;
constexpr int kBlocksPerCta = 2048;
constexpr int64_t kMinCtaBytes = int64_t(24) << 10;
constexpr int64_t kMinBlockBytes = int64_t(8) << 10;
constexpr int64_t kMaxBlockBytes = int64_t(1) << 20;
// Layouts of units of kEvenUnitBytes and more on average: a CTA's part divided
// by its warps, in as many equal rounds as keep a block within kEvenBlockBytes
// or a little above (560 units of 224 KB, 26 KB a warp: one 26 KB round 27.5 us,
// two of 13 KB 27.8, 8 KiB blocks 29.3, 24 KB blocks, 18 to a CTA, 31.3; a rank's
// 303 MB of 168 units 56.9 -> 55.3; 84 units in 95 MB 36.6 -> 35.0).
constexpr int64_t kEvenUnitBytes = int64_t(128) << 10;
constexpr int64_t kEvenBlockBytes = int64_t(16) << 10;
// Arenas of at most kSmallArenaCtaBytes of cost per resident CTA are cut between
// units: joining the parts of a split unit takes longer than streaming a unit of
// up to kWholeUnitBytes, 8 KiB a warp (64 units in 3.7 MB: 11.4 -> 10.1 us).
constexpr int64_t kSmallArenaCtaBytes = int64_t(48) << 10;
constexpr int64_t kWholeUnitBytes = int64_t(128) << 10;

// A piece of one segment.  `where`: its epilogue batch, counted from the CTA's
// first unit (8 bits), the slot of its sum (12 bits: its place in the CTA's
// blocks in unit order) and log2 of the lanes that stream it (3 bits).
struct alignas(16) Block {
    int64_t start;    // first element, in the arena
    int32_t elems;    // -1: no block
    uint32_t where;
};
constexpr uint32_t kSlotShift = 8, kLanesShift = 20;
static_assert(kBlocksPerCta / kBatch < (1 << kSlotShift) && kBlocksPerCta <= (1 << (kLanesShift - kSlotShift)), "Block::where");
// What a warp takes at a time with kVariantGroups: up to kItemBlocks blocks of
// one batch, each streamed by 32, 16, 8 or 4 lanes with kGroupVecs 16-byte
// vectors a lane; kVariantSmall takes one block, streamed by the whole warp.
// Planned where it makes at most kGroupedShare of the turns: a turn is about 2 us
// of a warp, whatever its size, mostly the latency of its loads.  100,000 bf16
// units of 55-440 elements 55.7 -> 34.2 us, of 64-512 fp32 elements 52.2 -> 36.6,
// 30,000 of 48-4,096 bf16 elements 31.0 -> 28.1.
constexpr int kItemBlocks = 8;
constexpr int kGroupVecs = 8;
constexpr double kGroupedShare = 0.75;
struct alignas(16) CtaBlocks {
    int32_t first, count;         // blocks
    int32_t unit, units;          // first unit touched, and how many
    int32_t turn, turns;          // what the warps take: entries of `block`, in kItemBlocks with kVariantGroups
    // the first and the last unit (one and the same if units == 1), which
    // other CTAs may have parts of: number of parts (1: none), the unit's
    // first partial slot, and this CTA's slot from there
    int32_t parts[2], slot[2];
    int32_t pad[2];
    int64_t base[2];
};

// Persistent per-unit controller state (Algorithm 1 and 2), 40 bytes.
struct UnitState {
    double mean;      // A_b, historical mean of n_b
    int64_t count;    // k_b, steps at which b was observed
    int32_t fill;     // |Q_b|, valid entries of the GNMR queue (<= window)
    int32_t head;     // ring position of the oldest queue entry once full
    int32_t lock;     // Lock_b
    int32_t active;   // 1 if b was on the recovery path at the previous step
    double gsum;      // GNMR summed over the static policy's warm-up
};
// lock and active are written together as one 8-byte store
static_assert(offsetof(UnitState, lock) % 8 == 0 && offsetof(UnitState, active) == offsetof(UnitState, lock) + 4,
              "UnitState lock/active pair");

// Bit pattern of an empty partial slot (a NaN that no partial sum takes:
// partials are non-negative, +inf or the canonical NaN).  The first slot of
// every unit split in two holds it between steps.
constexpr unsigned long long kEmptyPartial = ~0ull;

// Candidate-pool entry written by the unit epilogue, read by the selection
// (one 16-byte load).
struct Candidate {
    double risk;      // R_{b,t} (the static policy ranks by the GNMR sum)
    int32_t unit;
    uint32_t lock;    // Lock_b before this step, bit 31: active at the previous step
};
constexpr uint32_t kCandActive = 0x80000000u;

// Risk histogram of the candidate pool, built by the unit epilogues with one
// atomic per pool member and read (and cleared) by the selecting CTA.  Bin 0
// holds R < 1 (lock-only candidates); the bins above 1.0 get wider with R
// (risk_bin); the last one also holds everything larger (+inf included).
constexpr int kRiskBins = 2048;
// Hot list: the candidates a step appends because their bin is at or above a
// bin predicted from the previous step's cut (plus, under the admission cap,
// every retained unit).  When the prediction holds, the selecting CTA reads
// this short list instead of the whole candidate list.
constexpr uint32_t kHotCapMax = 8192;
constexpr uint32_t kNoHot = kRiskBins;   // hot_bin: no prediction, no pool member is hot

// Up to this many units (four a thread of the selecting CTA) a step keeps no
// lists and no histogram: reading every unit's entry costs the selection one
// round trip, where appending cost each epilogue two (64 units: tail of the
// step after the last epilogue 3.7 -> 2.8 us, the epilogue itself 4.4 -> 3.1
// us with the four-lane divisions).
constexpr int32_t kDenseUnits = 2048;

// Device-resident step control block.
struct Control {
    uint32_t ctas_done;   // CTA completion ticket of the current launch
    uint32_t n_cand;      // |C_t| appended so far
    int64_t steps;        // completed steps (t of the last step)
    uint32_t n_hot;       // hot-list entries appended so far (may exceed the capacity)
    uint32_t hot_bin;     // lowest bin whose pool members go to the hot list this step
    uint32_t pad[26];     // the run counters below on a 128-byte line of their own
    uint32_t next_run;    // runs taken beyond the warps' first ones (large-unit loop)
    uint32_t warps_done;  // partial-sums half: warps that have taken their last run
                          // (both zero between launches)
};
static_assert(offsetof(Control, next_run) == 128, "run counters on their own line");

// Checkpoint blob: this header, then UnitState[num_units], then the GNMR ring
// buffers double[num_units * window] (little-endian, as on the device).
struct StateHeader {
    char magic[4];        // "GNMR"
    uint32_t version;     // 2
    int32_t num_units;
    int32_t window;
    int64_t steps;
    int64_t reserved;
};

// A divisor fixed for many divisions, with its reciprocal rounded to nearest; 0
// where the device has to divide (see divide_by).
struct Divisor {
    double value;
    double inverse;
};
inline Divisor make_divisor(double v)
{
    return {v, v >= 0x1p-200 && v <= 0x1p+200 ? 1.0 / v : 0.0};
}

struct StepParams {
    const void *arena;
    // large-unit loop only (first_run, num_parts and part_base too)
    const int64_t *offset;       // [S] segment offsets, segments grouped by unit
    const int64_t *length;       // [S] segment lengths
    const int32_t *seg_unit;     // [S] unit of each segment (non-decreasing)
    const uint8_t *recoverable;  // [U]
    const int64_t *run_seg;      // [R + 1] first segment of each run
    const int64_t *run_pos;      // [R + 1]
    const CtaBlocks *cta_blocks; // [num_ctas] small-unit loop: each CTA's part,
    const Block *block;          // the blocks of all CTAs, in the order the warps take them
    const int32_t *unit_block;   // [U + 1] and the first block of each unit
    const int32_t *first_run;    // [U] first run touching unit b
    const int32_t *num_parts;    // [U]
    const int64_t *part_base;    // [U] first partial slot of unit b
    double *partial;             // [num_partials]
    uint32_t *unit_ticket;       // [U]
    UnitState *state;            // [U]
    double *queue;               // [U * window] GNMR ring buffers
    Candidate *cand;             // [U]
    Candidate *hot;              // [hot_cap] the hot list
    uint32_t *risk_hist;         // [kRiskBins], zero between steps
    Control *ctl;
    uint8_t *mask;               // [U], caller
    double *out_norm, *out_gnmr, *out_dgnmr, *out_risk;  // caller, optional
    int32_t *out_lock, *out_counts;                       // caller, optional
    double *out_sumsq;                                    // kStepPartials output [U]
    const double *in_sumsq;                               // kStepFinish input [U]
    double *out_delta_mem;                                // caller, optional [1]
    const double *unit_cost;                              // [U] or null
    int32_t policy;
    int32_t num_recoverable;
    int64_t forced_steps;
    int64_t static_warmup;
    int32_t static_keep;                                  // ceil(static_fraction * |B_rec|)
    uint32_t hot_cap;                                     // min(U, kHotCapMax)
    int32_t num_units;
    int32_t num_warps;           // large-unit loop: warps with a first run, 0 .. num_warps - 1
    int32_t window;
    int32_t max_o;
    int32_t lock_len;
    int32_t finish_units;        // controller half: units per warp, kFewUnits or 32
    int32_t dense;               // 1: at most kDenseUnits units, selected from one entry each
    int32_t num_runs;            // R; runs num_warps .. R - 1 are taken dynamically
    int64_t warmup_steps;
    Divisor alpha_init, alpha_main, beta_init, beta_main;
    Divisor alpha_override, beta_override;  // NaN = two-stage schedule
    Divisor window_length;
    double eps;
};

// Step kernel modes: the full step, its gradient half (per-unit sums of
// squares only) and its controller half (Algorithms 1-2 on given sums).
constexpr int kStepFull = 0;
constexpr int kStepPartials = 1;
constexpr int kStepFinish = 2;

// Enqueues one launch of the step kernel in `mode`; returns the launch status.
cudaError_t launch_step(const StepParams &p, int dtype, int num_ctas, cudaStream_t stream,
                        int mode = kStepFull, int variant = kVariantSmall);

// Resident CTAs per SM of the step kernel for `dtype`, `variant` and `dense`.
cudaError_t step_occupancy(int dtype, int variant, bool dense, int *ctas_per_sm);

// Records the failure detail that gnmr_last_error(NULL) reports on the
// calling thread (used by calls that have no handle).
void record_thread_error(const char *why);

// Host-side work partition (gnmr_plan.cpp).
struct Plan {
    int32_t num_runs = 0;
    std::vector<int64_t> run_seg;     // [num_runs + 1]
    std::vector<int64_t> run_pos;     // [num_runs + 1]
    std::vector<int32_t> first_run;   // [U]
    std::vector<int32_t> num_parts;   // [U]
    std::vector<int64_t> part_base;   // [U]
    int64_t num_partials = 0;
};

// Segments must be grouped by unit (seg_unit non-decreasing, every unit
// 0..num_units-1 present).  Cuts the stream into at most max_runs runs, none
// smaller than kMinRunBytes unless the whole problem is; or at the given costs
// (increasing).  Returns false if the inputs are out of range.
bool plan_partition(int64_t num_segments, const int64_t *seg_lengths, const int32_t *seg_unit,
                    int32_t num_units, int elem_bytes, int32_t max_runs, Plan &out,
                    const std::vector<int64_t> *targets = nullptr);

// The blocks of a plan with one run per CTA (small-unit loop).
struct BlockPlan {
    std::vector<CtaBlocks> cta;       // [num_runs]
    std::vector<Block> block;         // kItemBlocks entries a turn if grouped
    std::vector<int32_t> unit_block;  // [U + 1]
    bool grouped = false;
};

// Cuts the stream into one run per CTA (about max_ctas of them, more where their
// kBlocksPerCta blocks each do not do) and the runs into blocks.
// Same input rules as plan_partition; seg_offsets in elements.
bool plan_blocks(int64_t num_segments, const int64_t *seg_offsets, const int64_t *seg_lengths,
                 const int32_t *seg_unit, int32_t num_units, int elem_bytes, int32_t max_ctas, Plan &out,
                 BlockPlan &blocks);

}  // namespace gnmr
