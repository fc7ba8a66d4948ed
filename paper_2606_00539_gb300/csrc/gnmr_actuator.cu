// Recovery actuator: per-token fake quantization of every unit's saved
// activations, in the low-cost or the recovery format as the unit's mask bit
// says (App. E.2; the activation-quantization stress bench of Sec. 5.1).  For
// each token row: amax = max |x|; inv = fmax / amax; scale = amax / fmax;
// y = round_to_format(x * inv) * scale, rounding to the nearest representable
// value with ties to the even code and saturating at fmax.  All arithmetic is
// fp32, so the quantized codes are the same on any IEEE machine.  Rows whose
// max is 0, that hold a NaN or Inf, or whose scale factor fmax / amax
// overflows fp32 (amax below fmax / FLT_MAX) are copied unchanged.
//
// The rounding is the hardware minifloat conversion (cvt.rn.satfinite to
// e2m1x2 / e3m2x2 / e4m3x2 / e5m2x2, then back to f16x2, where every value of
// these formats is exact): round to nearest even, saturating -- the format
// definition itself, two values per instruction.
//
// Rows of up to 2,048 16-byte vectors are read once: a group of 4 to 256
// threads holds the row in registers, 8 vectors a thread, takes amax (shuffles,
// over several warps a named barrier and shared memory) and writes the
// registers out rounded.  A CTA takes a tile of 256 / group rows of one unit
// at a time, so whatever the row length all its threads have about 8 loads in
// flight and the work per row is shared by the rows of a warp.  HBM-bound from
// 512-byte rows on.  Measured on one GB300 (read + write bytes / time), from
// one row per warp, read twice, to held rows:
//     256-element bf16 rows (with 683)   1.66 -> 6.0 TB/s
//     768 (with 2048)                    3.1  -> 6.5 TB/s
//     2048 (with 5504)                   5.3  -> 6.6 TB/s
//     1408 fp32 (with 3755)              5.1  -> 6.5 TB/s
// 24 warps per SM: 32 (64 registers, a few spills) were 0-10 % slower, 16
// 10-20 %.  Streaming stores: plain ones 2 % slower, evict-first policies 3 %.
//
// A longer row, and in layouts of many rows every row of more than 512
// vectors, is read twice by one warp: pass 1 for amax (integer max over the
// magnitude bits), pass 2 from L2 to write the result, so HBM still sees one
// read and one write per element.  That grid holds 16 warps per SM, whose rows
// (about 30 MB in all) stay resident in the 129 MB L2 between the two passes:
// pass 1 loads them with an L2 evict-last policy, pass 2 reads and the output
// stores use evict-first, so the write stream does not push the waiting rows
// out.  (32 warps per SM left a fifth of the pass-2 reads missing L2; 8 cannot
// keep enough loads in flight.)
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "gnmr.h"
#include "gnmr_internal.h"

struct gnmr_actuator {
    int32_t num_units = 0;
    int32_t dtype = 0;
    int32_t device = 0;
    int32_t sms = 1;
    bool any_long = false;                // some row is too long to be held
    bool any_held = false;                // and some is not
    bool by_warp = false;                 // tiles of a warp, not of a CTA
    int32_t most = 0;                     // widest group that holds a row
    int64_t tiles = 0;
    int64_t tiles_plain = 0;              // one row each
    int64_t max_end = 0;
    void *dmem = nullptr;
    const int64_t *offset = nullptr;      // [U]
    const int64_t *rows = nullptr;        // [U]
    const int64_t *cols = nullptr;        // [U]
    const int64_t *start = nullptr;       // [U + 1] first tile of each unit
    const int64_t *start_plain = nullptr; // [U + 1]
};

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kLongCtas = 2;            // 16 warps per SM: the rows read twice stay in L2
constexpr int kShortCtas = 3;           // 24 warps per SM, 80 registers per thread
constexpr int kPass1Loads = 16;         // 16-byte loads in flight per lane in pass 1 (from HBM)
constexpr int kPass2Loads = 8;          // in pass 2 (from L2)

struct FqFmt {
    float fmax;
    int code;      // gnmr_fq_format; 0 = copy
};

bool fmt_of(int code, FqFmt &f)
{
    switch (code) {
    case GNMR_FQ_NONE: f = {1.0f, 0}; return true;
    case GNMR_FQ_E2M1: f = {6.0f, 1}; return true;
    case GNMR_FQ_E3M2: f = {28.0f, 2}; return true;
    case GNMR_FQ_E4M3: f = {448.0f, 3}; return true;
    case GNMR_FQ_E5M2: f = {57344.0f, 4}; return true;
    default: return false;
    }
}

// Two fp32 products in one instruction (each rounded as the scalar one is).
__device__ __forceinline__ float2 mul2(float2 a, float b)
{
    float2 r;
    asm("{ .reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %4}; mul.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z; }"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b));
    return r;
}

// Rounds (a0, a1) to format CODE and returns them as fp32 (exact).
template <int CODE>
__device__ __forceinline__ float2 fq_round2(float a0, float a1)
{
    uint32_t h2;
    if (CODE == 1)
        asm("{ .reg .b8 t; cvt.rn.satfinite.e2m1x2.f32 t, %2, %1; cvt.rn.f16x2.e2m1x2 %0, t; }"
            : "=r"(h2) : "f"(a0), "f"(a1));
    else if (CODE == 2)
        asm("{ .reg .b16 t; cvt.rn.satfinite.e3m2x2.f32 t, %2, %1; cvt.rn.f16x2.e3m2x2 %0, t; }"
            : "=r"(h2) : "f"(a0), "f"(a1));
    else if (CODE == 3)
        asm("{ .reg .b16 t; cvt.rn.satfinite.e4m3x2.f32 t, %2, %1; cvt.rn.f16x2.e4m3x2 %0, t; }"
            : "=r"(h2) : "f"(a0), "f"(a1));
    else
        asm("{ .reg .b16 t; cvt.rn.satfinite.e5m2x2.f32 t, %2, %1; cvt.rn.f16x2.e5m2x2 %0, t; }"
            : "=r"(h2) : "f"(a0), "f"(a1));
    __half2 h;
    memcpy(&h, &h2, sizeof h);
    return make_float2(__low2float(h), __high2float(h));
}

// Scalar loads are plain ones, not the read-only path: the kernel may start
// before the kernel that writes its input has ended, and works in place.
template <int DT> struct Act;
template <> struct Act<0> {                     // fp32: 4 per vector
    static constexpr int kBytes = 4;
    static constexpr int kN = 4;
    __device__ static float load(const void *p, int64_t i) { return static_cast<const float *>(p)[i]; }
    __device__ static void store(void *p, int64_t i, float y) { static_cast<float *>(p)[i] = y; }
    using Bits = unsigned int;
    __device__ static Bits bits(const void *s, int64_t i) { return static_cast<const Bits *>(s)[i]; }
    __device__ static void put(void *d, int64_t i, Bits x) { static_cast<Bits *>(d)[i] = x; }
    __device__ static void copy(const void *s, void *d, int64_t i) { put(d, i, bits(s, i)); }
    __device__ static void unpack(const uint4 v, float *x)
    {
        x[0] = __uint_as_float(v.x); x[1] = __uint_as_float(v.y);
        x[2] = __uint_as_float(v.z); x[3] = __uint_as_float(v.w);
    }
    __device__ static uint4 pack(const float *y)
    {
        return make_uint4(__float_as_uint(y[0]), __float_as_uint(y[1]), __float_as_uint(y[2]), __float_as_uint(y[3]));
    }
};
template <> struct Act<1> {                     // bf16: 8 per vector
    static constexpr int kBytes = 2;
    static constexpr int kN = 8;
    __device__ static float load(const void *p, int64_t i)
    {
        return __uint_as_float(static_cast<uint32_t>(static_cast<const unsigned short *>(p)[i]) << 16);
    }
    __device__ static void store(void *p, int64_t i, float y)
    {
        static_cast<unsigned short *>(p)[i] = __bfloat16_as_ushort(__float2bfloat16_rn(y));
    }
    using Bits = unsigned short;
    __device__ static Bits bits(const void *s, int64_t i) { return static_cast<const Bits *>(s)[i]; }
    __device__ static void put(void *d, int64_t i, Bits x) { static_cast<Bits *>(d)[i] = x; }
    __device__ static void copy(const void *s, void *d, int64_t i) { put(d, i, bits(s, i)); }
    __device__ static void unpack(const uint4 v, float *x)
    {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    __device__ static uint4 pack(const float *y)
    {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(y[2 * i], y[2 * i + 1]);
            memcpy(&w[i], &p, sizeof w[i]);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

template <int DT, int CODE>
__device__ __forceinline__ uint4 quantize_vec(const uint4 v, float inv, float scale)
{
    float x[Act<DT>::kN], y[Act<DT>::kN];
    Act<DT>::unpack(v, x);
#pragma unroll
    for (int k = 0; k < Act<DT>::kN; k += 2) {
        const float2 t = mul2(make_float2(x[k], x[k + 1]), inv);
        const float2 q = mul2(fq_round2<CODE>(t.x, t.y), scale);
        y[k] = q.x;
        y[k + 1] = q.y;
    }
    return Act<DT>::pack(y);
}

// Largest magnitude of a 16-byte vector as an fp32 bit pattern without its
// sign: for non-negative floats the bit patterns order like the values, and
// Inf (0x7f800000) and NaN (above it) order above every finite value.
template <int DT> __device__ __forceinline__ uint32_t vec_max_bits(const uint4 v);
template <> __device__ __forceinline__ uint32_t vec_max_bits<0>(const uint4 v)
{
    return max(max(v.x & 0x7fffffffu, v.y & 0x7fffffffu), max(v.z & 0x7fffffffu, v.w & 0x7fffffffu));
}
template <> __device__ __forceinline__ uint32_t vec_max_bits<1>(const uint4 v)
{
    // two bf16 per word: per-halfword unsigned max of the magnitudes
    const uint32_t m = __vmaxu2(__vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu),
                                __vmaxu2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu));
    return max(m << 16, m & 0xffff0000u);
}
template <int DT> __device__ __forceinline__ uint32_t elem_max_bits(const char *p, int64_t i)
{
    return __float_as_uint(Act<DT>::load(p, i)) & 0x7fffffffu;
}

// The rows of a unit are taken in tiles of rows_of(group); the last tile
// of a unit may hold fewer.  start[b]: first tile of unit b, [U + 1].
struct RowTables {
    const int64_t *offset;
    const int64_t *rows;
    const int64_t *cols;
    const int64_t *start;
    int64_t tiles;
    int32_t num_units;
    int32_t most;                         // widest group: see group_of
};

// The unit a warp is in: tiles [begin, end).
struct UnitCursor {
    int64_t begin = 0, end = 0;
    int32_t unit = -1;
    FqFmt f = {1.0f, 0};
};

// Last unit with start <= r, by the whole warp: each round reads 32 evenly
// spaced starts at once, so 1,000 units take two dependent loads where a
// binary search takes ten.
__device__ __forceinline__ int32_t find_unit(int64_t r, const int64_t *start, int32_t num_units, int lane)
{
    int32_t lo = 0, hi = num_units;              // start[lo] <= r < start[hi]
    while (hi - lo > 1) {
        const int32_t step = (hi - lo - 1) / 32 + 1;
        const int64_t at = lo + static_cast<int64_t>(step) * lane;
        const bool ok = at < hi && start[at] <= r;
        const int last = 31 - __clz(__ballot_sync(kFull, ok));       // lane 0 always holds
        lo += step * last;
        hi = hi - lo > step ? lo + step : hi;
    }
    return lo;
}

// Moves the cursor to the unit of tile r.  Called by the whole warp.
__device__ __forceinline__ void seek(UnitCursor &c, int64_t r, const RowTables &t, int lane)
{
    c.unit = find_unit(r, t.start, t.num_units, lane);
    c.begin = t.start[c.unit];
    c.end = t.start[c.unit + 1];
}

// Where a row lives and how it splits into head / 16-byte body / tail (the
// body is vectorised only when input and output share 16-byte alignment).
struct RowRef {
    const char *src;
    char *dst;
    int64_t n, head, nvec, tail_at;
    FqFmt f;
};

template <int DT>
__device__ __forceinline__ RowRef locate_row(int64_t e0, int64_t n, const FqFmt &f, const void *in, void *out)
{
    constexpr int kEB = Act<DT>::kBytes;
    RowRef q;
    q.f = f;
    q.n = n;
    q.src = static_cast<const char *>(in) + e0 * kEB;
    q.dst = static_cast<char *>(out) + e0 * kEB;
    const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(q.src) & 15u);
    const bool aligned = mis == static_cast<uint32_t>(reinterpret_cast<uintptr_t>(q.dst) & 15u);
    q.head = aligned ? static_cast<int64_t>(((16u - mis) & 15u) / kEB) : q.n;
    q.head = q.head < q.n ? q.head : q.n;
    q.nvec = (q.n - q.head) / Act<DT>::kN;
    q.tail_at = q.head + q.nvec * Act<DT>::kN;
    return q;
}

// L2 eviction policies for a whole access (createpolicy), and 16-byte
// accesses that carry one.
__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint4 ld_policy(const uint4 *q, uint64_t pol)
{
    uint4 r;
    asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(q), "l"(pol));
    return r;
}
__device__ __forceinline__ void st_policy(uint4 *q, uint4 v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;"
                 ::"l"(q), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "l"(pol) : "memory");
}

// Pass 1's load keeps the line in L2 for pass 2; pass 2's load is its last
// use, and the output is written once.
__device__ __forceinline__ uint4 ld_keep(const uint4 *p) { return ld_policy(p, policy_evict_last()); }
__device__ __forceinline__ uint4 ld_last(const uint4 *p) { return ld_policy(p, policy_evict_first()); }
__device__ __forceinline__ void st_once(uint4 *p, uint4 v) { st_policy(p, v, policy_evict_first()); }

// A row that is read once: no reuse, so nothing to keep in L1.
__device__ __forceinline__ uint4 ld_once(const uint4 *q)
{
    uint4 r;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(q));
    return r;
}

// A row kept as it is (bit-for-bit copy): no format, a zero row, a non-finite
// value, or a row so small that its scale factor fmax / amax overflows fp32.
__device__ __forceinline__ bool row_kept(const FqFmt &f, uint32_t mbits)
{
    return f.code == 0 || mbits == 0u || mbits >= 0x7f800000u || isinf(f.fmax / __uint_as_float(mbits));
}

// Elements [from, to) of a row one by one, kElemLoads in flight per lane (the
// compiler does not move a load over the stores before it: 300 rows of 300,000
// fp32 whose output is shifted by an element took 4,460 us with one load a lane,
// 723 with 16).
constexpr int kElemLoads = 16;
template <int DT> __device__ __forceinline__ uint32_t max_elems(const char *src, int64_t from, int64_t to, int lane)
{
    uint32_t m = 0;
    int64_t i = from + lane;
    for (; i + (kElemLoads - 1) * 32 < to; i += kElemLoads * 32) {
        uint32_t x[kElemLoads];
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            x[j] = elem_max_bits<DT>(src, i + j * 32);
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            m = max(m, x[j]);
    }
    for (; i < to; i += 32)
        m = max(m, elem_max_bits<DT>(src, i));
    return m;
}
template <int DT, int CODE>
__device__ __forceinline__ void quantize_elems(const char *src, char *dst, int64_t from, int64_t to, float inv,
                                               float scale, int lane)
{
    int64_t i = from + lane;
    for (; i + (kElemLoads - 1) * 32 < to; i += kElemLoads * 32) {
        float x[kElemLoads];
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            x[j] = Act<DT>::load(src, i + j * 32);
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            Act<DT>::store(dst, i + j * 32, fq_round2<CODE>(x[j] * inv, 0.f).x * scale);
    }
    for (; i < to; i += 32)
        Act<DT>::store(dst, i, fq_round2<CODE>(Act<DT>::load(src, i) * inv, 0.f).x * scale);
}
template <int DT>
__device__ __forceinline__ void copy_elems(const char *src, char *dst, int64_t from, int64_t to, int lane)
{
    int64_t i = from + lane;
    for (; i + (kElemLoads - 1) * 32 < to; i += kElemLoads * 32) {
        typename Act<DT>::Bits x[kElemLoads];
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            x[j] = Act<DT>::bits(src, i + j * 32);
#pragma unroll
        for (int j = 0; j < kElemLoads; ++j)
            Act<DT>::put(dst, i + j * 32, x[j]);
    }
    for (; i < to; i += 32)
        Act<DT>::copy(src, dst, i);
}

// Pass 2 of one row in format CODE (one warp): quantize and write.
template <int DT, int CODE>
__device__ __forceinline__ void quantize_row_warp(const char *src, char *dst, const uint4 *vs, uint4 *vd,
                                                  int64_t head, int64_t nvec, int64_t tail_at, int64_t n,
                                                  float inv, float scale, int lane)
{
    quantize_elems<DT, CODE>(src, dst, 0, head, inv, scale, lane);
    int64_t i = lane;
    for (; i + (kPass2Loads - 1) * 32 < nvec; i += kPass2Loads * 32) {
        uint4 v[kPass2Loads];
#pragma unroll
        for (int j = 0; j < kPass2Loads; ++j)
            v[j] = ld_last(vs + i + j * 32);
#pragma unroll
        for (int j = 0; j < kPass2Loads; ++j)
            st_once(vd + i + j * 32, quantize_vec<DT, CODE>(v[j], inv, scale));
    }
    for (; i < nvec; i += 32)
        st_once(vd + i, quantize_vec<DT, CODE>(ld_last(vs + i), inv, scale));
    quantize_elems<DT, CODE>(src, dst, tail_at, n, inv, scale, lane);
}

// A row too long for registers, or whose input and output lie differently in
// their 16-byte words (then all of it is "head"): pass 1 reads it (16 16-byte
// loads in flight per lane) for amax, pass 2 reads it again -- from L2, the
// resident warps' rows fit there -- and writes the result once.
template <int DT>
__device__ __forceinline__ void row_two_pass(const RowRef &q, int lane)
{
    constexpr int kEB = Act<DT>::kBytes;
    const uint4 *vs = reinterpret_cast<const uint4 *>(q.src + q.head * kEB);
    uint4 *vd = reinterpret_cast<uint4 *>(q.dst + q.head * kEB);
    uint32_t mbits = max_elems<DT>(q.src, 0, q.head, lane);
    int64_t i = lane;
    for (; i + (kPass1Loads - 1) * 32 < q.nvec; i += kPass1Loads * 32) {
        uint4 v[kPass1Loads];
#pragma unroll
        for (int j = 0; j < kPass1Loads; ++j)
            v[j] = ld_keep(vs + i + j * 32);
#pragma unroll
        for (int j = 0; j < kPass1Loads; ++j)
            mbits = max(mbits, vec_max_bits<DT>(v[j]));
    }
    for (; i < q.nvec; i += 32)
        mbits = max(mbits, vec_max_bits<DT>(ld_keep(vs + i)));
    mbits = max(mbits, max_elems<DT>(q.src, q.tail_at, q.n, lane));
    mbits = __reduce_max_sync(kFull, mbits);

    if (row_kept(q.f, mbits)) {
        if (q.src != q.dst) {
            copy_elems<DT>(q.src, q.dst, 0, q.head, lane);
            for (int64_t t = lane; t < q.nvec; t += 32)
                st_once(vd + t, ld_last(vs + t));
            copy_elems<DT>(q.src, q.dst, q.tail_at, q.n, lane);
        }
        return;
    }
    const float amax = __uint_as_float(mbits);
    const float inv = q.f.fmax / amax;
    const float scale = amax / q.f.fmax;
    switch (q.f.code) {                           // one dispatch per row
    case 1: quantize_row_warp<DT, 1>(q.src, q.dst, vs, vd, q.head, q.nvec, q.tail_at, q.n, inv, scale, lane); break;
    case 2: quantize_row_warp<DT, 2>(q.src, q.dst, vs, vd, q.head, q.nvec, q.tail_at, q.n, inv, scale, lane); break;
    case 3: quantize_row_warp<DT, 3>(q.src, q.dst, vs, vd, q.head, q.nvec, q.tail_at, q.n, inv, scale, lane); break;
    default: quantize_row_warp<DT, 4>(q.src, q.dst, vs, vd, q.head, q.nvec, q.tail_at, q.n, inv, scale, lane); break;
    }
}

// Threads that hold a row of n elements in their registers, kHold vectors
// each: the smallest power of two from kMinGroup to `most` that has room for
// it, or 0 if the row is longer (it is then read twice, by one warp).
constexpr int kHold = 8;
constexpr int kMinGroup = 4;
__host__ __device__ constexpr int group_of(int64_t n, int per_vec, int most)
{
    int g = kMinGroup;
    while (g <= most && n / per_vec > int64_t(kHold) * g)
        g *= 2;
    return g <= most ? g : 0;
}
// Rows wider than two warps are held by up to the whole CTA, unless a layout
// has at least kManyRows of them per resident warp of the two-pass kernel.
// Measured on one GB300: 5120 / 13824-element bf16 rows, 3 a warp, 40 us read
// twice against 36 us held; 70 a warp, 679 against 767 us.
constexpr int kWideGroup = 64;
constexpr int64_t kManyRows = 8;
static_assert(kThreads == 256, "a row is held by at most eight warps");
// Rows of one unit that a CTA takes at a time.  With kWarpTiles each warp takes
// rows by itself: where every row is read twice, and in layouts of units of so
// few rows that more than half of the warps of CTA tiles would have none, if no
// row takes more than a warp (1,000 units of one 64-element row 7.9 -> 3.0 us).
template <bool kWarpTiles> __host__ __device__ constexpr int rows_of(int group)
{
    return group ? (kWarpTiles ? 32 : kThreads) / group : kWarpTiles ? 1 : kWarps;
}

// A row of n elements (0: none) held by a group of threads, `gl` the thread's
// place in it: vector gl + group j in v[j], and of the head and the tail (less
// than one vector each) element gl + group e in xh[e], xt[e].
template <int DT>
struct HeldRow {
    static constexpr int kEB = Act<DT>::kBytes;
    static constexpr int kEdge = (Act<DT>::kN - 2) / kMinGroup + 1;
    int head, nvec, tail, tail_at;
    uint4 v[kHold];
    float xh[kEdge], xt[kEdge];

    // Issues the row's loads.
    __device__ __forceinline__ void load(const char *src, int n, int group, int gl)
    {
        const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src)) & 15u;
        head = min(static_cast<int>(((16u - mis) & 15u) / kEB), n);
        nvec = (n - head) / Act<DT>::kN;
        tail_at = head + nvec * Act<DT>::kN;
        tail = n - tail_at;
        const uint4 *vs = reinterpret_cast<const uint4 *>(src + head * kEB);
#pragma unroll
        for (int j = 0; j < kHold; ++j)
            v[j] = gl + group * j < nvec ? ld_once(vs + gl + group * j) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int e = 0; e < kEdge; ++e) {
            xh[e] = gl + group * e < head ? Act<DT>::load(src, gl + group * e) : 0.0f;
            xt[e] = gl + group * e < tail ? Act<DT>::load(src, tail_at + gl + group * e) : 0.0f;
        }
    }

    // Largest magnitude of the thread's part of the row.
    __device__ __forceinline__ uint32_t max_bits() const
    {
        uint32_t m = 0;
#pragma unroll
        for (int e = 0; e < kEdge; ++e)
            m = max(m, max(__float_as_uint(xh[e]) & 0x7fffffffu, __float_as_uint(xt[e]) & 0x7fffffffu));
#pragma unroll
        for (int j = 0; j < kHold; ++j)
            m = max(m, vec_max_bits<DT>(v[j]));
        return m;
    }

    // Rounds the row to format CODE and writes it; mbits: the row's largest
    // magnitude.  `bound` >= nvec for every row of the tile.
    template <int CODE>
    __device__ __forceinline__ void write(const char *src, char *dst, const FqFmt &f, uint32_t mbits, int bound,
                                          int group, int gl) const
    {
        const bool kept = row_kept(f, mbits);
        if (kept && src == dst)
            return;                               // in place: there already
        const float inv = f.fmax / __uint_as_float(mbits);
        const float scale = __uint_as_float(mbits) / f.fmax;
        uint4 *vd = reinterpret_cast<uint4 *>(dst + head * kEB);
#pragma unroll
        for (int j = 0; j < kHold; ++j) {
            if (group * j < bound) {
                const uint4 y = quantize_vec<DT, CODE>(v[j], inv, scale);
                if (gl + group * j < nvec)
                    __stcs(vd + gl + group * j, kept ? v[j] : y);
            }
        }
#pragma unroll
        for (int e = 0; e < kEdge; ++e) {
            const int at = gl + group * e;
            if (at < head) {
                if (kept)
                    Act<DT>::copy(src, dst, at);
                else
                    Act<DT>::store(dst, at, fq_round2<CODE>(xh[e] * inv, 0.0f).x * scale);
            }
            if (at < tail) {
                if (kept)
                    Act<DT>::copy(src, dst, tail_at + at);
                else
                    Act<DT>::store(dst, tail_at + at, fq_round2<CODE>(xt[e] * inv, 0.0f).x * scale);
            }
        }
    }
};

// Where the warps of a row held by two, four or eight warps exchange their
// maxima.  Each width has slots and barriers of its own (groups of another
// width hold other warps), and two sets of slots that its rows use in turn: a
// warp that writes a set has passed the barrier of the other one, which every
// reader of the first has reached after reading.
struct GroupMax {
    uint32_t slot[3][2][kWarps];
};

// One tile of held rows: the CTA's (or warp's) threads in groups, one row each.  `turn`
// has a bit for each width, the set of slots it uses next.
template <int DT, bool kWarpTiles>
__device__ __forceinline__ void held_tile(const char *src, char *dst, int n, int group, int count, const FqFmt &f,
                                          GroupMax &gm, uint32_t &turn)
{
    const int row = (kWarpTiles ? threadIdx.x & 31 : threadIdx.x) >> (__ffs(group) - 1), gl = threadIdx.x & (group - 1);
    const bool there = row < count;
    const int64_t at = there ? static_cast<int64_t>(row) * n * Act<DT>::kBytes : 0;
    src += at;
    dst += at;
    HeldRow<DT> h;
    h.load(src, there ? n : 0, group, gl);
    uint32_t m = h.max_bits();
    if (group >= 32) {
        m = __reduce_max_sync(kFull, m);
        if (!kWarpTiles && group > 32) {
            const int warps = group / 32, first = row * warps;
            const int width = warps == 2 ? 0 : warps == 4 ? 1 : 2;
            const int barrier = (width == 0 ? 1 : width == 1 ? 5 : 7) + row;     // 1-4, 5-6, 7
            volatile uint32_t *slot = gm.slot[width][(turn >> width) & 1u];
            turn ^= 1u << width;
            if ((threadIdx.x & 31) == 0)
                slot[threadIdx.x >> 5] = m;
            asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(group) : "memory");
            for (int i = 0; i < warps; ++i)
                m = max(m, slot[first + i]);
        }
    } else {
        for (int o = group / 2; o > 0; o >>= 1)
            m = max(m, __shfl_xor_sync(kFull, m, o));
    }
    const int bound = n / Act<DT>::kN;
    switch (f.code) {                             // one dispatch per tile
    case 1: h.template write<1>(src, dst, f, m, bound, group, gl); break;
    case 2: h.template write<2>(src, dst, f, m, bound, group, gl); break;
    case 3: h.template write<3>(src, dst, f, m, bound, group, gl); break;
    default: h.template write<4>(src, dst, f, m, bound, group, gl); break;   // 4, and 0: every row kept
    }
}

// kLong = false: every row is held; kLong and kWarpTiles: none.  Held rows need input and output to share
// their 16-byte alignment (the host sees to it: most = 0 where they do not).
template <int DT, bool kLong, bool kWarpTiles>
__global__ void __launch_bounds__(kThreads, kLong ? kLongCtas : kShortCtas) fake_quant_kernel(
    const void *in, void *out, RowTables t, const uint8_t *mask, FqFmt low, FqFmt rec)
{
    constexpr int kEB = Act<DT>::kBytes;
    __shared__ GroupMax s_max;
    uint32_t turn = 0;
    const int lane = threadIdx.x & 31;
    int64_t r = blockIdx.x, stride = gridDim.x;
    if (kWarpTiles) {
        r += stride * (threadIdx.x >> 5);
        stride *= kWarps;
    }
    UnitCursor cur;
    // The tables never change after create: the first unit is looked up while
    // the kernel before this one on the stream is still running.  Its writes
    // (activations, mask) are visible after the wait.
    seek(cur, r, t, lane);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cur.f = (mask != nullptr && mask[cur.unit]) ? rec : low;
    for (; r < t.tiles; r += stride) {
        if (r >= cur.end) {
            seek(cur, r, t, lane);
            cur.f = (mask != nullptr && mask[cur.unit]) ? rec : low;
        }
        if (cur.f.code == 0 && in == out)
            continue;                             // a unit left as it is, in place
        const int64_t n = t.cols[cur.unit];
        const int group = kLong && kWarpTiles ? 0 : group_of(n, Act<DT>::kN, t.most);
        const int rows = rows_of<kWarpTiles>(group);
        const int64_t at = (r - cur.begin) * rows;             // the tile's first row in its unit
        const int64_t e0 = t.offset[cur.unit] + at * n;
        const int64_t left = t.rows[cur.unit] - at;
        const int count = left < rows ? static_cast<int>(left) : rows;
        if (kLong) {
            if (group == 0) {
                const int k = kWarpTiles ? 0 : threadIdx.x >> 5;
                if (k < count)
                    row_two_pass<DT>(locate_row<DT>(e0 + k * n, n, cur.f, in, out), lane);
                continue;
            }
        }
        if (kLong && kWarpTiles)
            continue;
        held_tile<DT, kWarpTiles>(static_cast<const char *>(in) + e0 * kEB, static_cast<char *>(out) + e0 * kEB,
                      static_cast<int>(n), group, count, cur.f, s_max, turn);
    }
}

// Launched as a programmatic dependent of the kernel before it on the stream.
template <int DT, bool kLong, bool kWarpTiles>
cudaError_t launch_shape(const RowTables &t, int sms, const void *in, void *out, const uint8_t *mask, FqFmt low,
                         FqFmt rec, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(std::min<int64_t>(t.tiles, int64_t(sms) * (kLong ? kLongCtas : kShortCtas))));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fake_quant_kernel<DT, kLong, kWarpTiles>, in, out, t, mask, low, rec);
}

template <int DT>
cudaError_t launch(const gnmr_actuator &a, const void *in, void *out, const uint8_t *mask, FqFmt low, FqFmt rec,
                   cudaStream_t stream)
{
    const bool together = ((reinterpret_cast<uintptr_t>(in) ^ reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
    RowTables t{a.offset, a.rows, a.cols, a.start, a.tiles, a.num_units, a.most};
    if (together && a.any_held) {
        if (a.any_long)
            return launch_shape<DT, true, false>(t, a.sms, in, out, mask, low, rec, stream);
        return a.by_warp ? launch_shape<DT, false, true>(t, a.sms, in, out, mask, low, rec, stream)
                         : launch_shape<DT, false, false>(t, a.sms, in, out, mask, low, rec, stream);
    }
    // every row read twice: too long, or no 16-byte vectors in common
    t.start = a.start_plain;
    t.tiles = a.tiles_plain;
    t.most = 0;
    return launch_shape<DT, true, true>(t, a.sms, in, out, mask, low, rec, stream);
}

gnmr_status act_fail(gnmr_status s, const std::string &why)
{
    gnmr::record_thread_error(why.c_str());
    return s;
}

}  // namespace

extern "C" {

gnmr_status gnmr_actuator_create(int32_t num_units, const int64_t *offsets, const int64_t *rows,
                                 const int64_t *cols, int32_t dtype, int32_t device, gnmr_actuator **out)
{
    if (out)
        *out = nullptr;
    if (!out || !offsets || !rows || !cols || num_units < 1)
        return act_fail(GNMR_ERR_INVALID_ARG, "actuator: NULL argument or num_units < 1");
    if (dtype != GNMR_DTYPE_F32 && dtype != GNMR_DTYPE_BF16)
        return act_fail(GNMR_ERR_INVALID_ARG, "actuator: unknown dtype");
    int64_t max_end = 0, total = 0;
    const int64_t limit = INT64_MAX / 8;
    for (int32_t b = 0; b < num_units; ++b) {
        if (offsets[b] < 0 || rows[b] < 0 || cols[b] < 0 || (cols[b] > 0 && rows[b] > limit / cols[b]) ||
            offsets[b] > limit - rows[b] * cols[b] || total > limit - rows[b])
            return act_fail(GNMR_ERR_INVALID_ARG, "actuator: unit " + std::to_string(b) + " out of range");
        total += rows[b];
        max_end = std::max(max_end, offsets[b] + rows[b] * cols[b]);
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
        return act_fail(GNMR_ERR_CUDA, "actuator: device not available");
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(device);
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    gnmr_actuator *a = new (std::nothrow) gnmr_actuator;
    if (!a) {
        cudaSetDevice(prev);
        return act_fail(GNMR_ERR_OOM, "actuator: host allocation failed");
    }
    const size_t U = static_cast<size_t>(num_units);
    const int per_vec = dtype == GNMR_DTYPE_BF16 ? Act<1>::kN : Act<0>::kN;
    int64_t wide = 0;
    for (size_t b = 0; b < U; ++b)
        if (group_of(cols[b], per_vec, kWideGroup) == 0)
            wide += rows[b];
    const int most = wide < kManyRows * sms * kLongCtas * kWarps ? kThreads : kWideGroup;
    bool any_long = false, any_held = false, by_warp = true;
    int64_t cta_tiles = 0, warp_tiles = 0;
    const auto tiles_of = [](int64_t n, int64_t per) { return n / per + (n % per != 0); };
    // rows without elements are no work, however many a unit claims to have
    const auto rows_with = [&](size_t b) { return cols[b] > 0 ? rows[b] : 0; };
    for (size_t b = 0; b < U; ++b) {
        const int group = group_of(cols[b], per_vec, most);
        any_long |= group == 0 && rows_with(b) > 0;
        any_held |= group != 0 && rows_with(b) > 0;
        by_warp &= group != 0 && group <= 32;
        if (by_warp) {
            cta_tiles += tiles_of(rows_with(b), rows_of<false>(group));
            warp_tiles += tiles_of(rows_with(b), rows_of<true>(group));
        }
    }
    by_warp &= cta_tiles * kWarps > 2 * warp_tiles;
    std::vector<int64_t> img;
    try {
        img.resize(5 * U + 2);
    } catch (const std::bad_alloc &) {
        cudaSetDevice(prev);
        delete a;
        return act_fail(GNMR_ERR_OOM, "actuator: host allocation failed");
    }
    std::memcpy(img.data(), offsets, 8 * U);
    std::memcpy(img.data() + U, rows, 8 * U);
    std::memcpy(img.data() + 2 * U, cols, 8 * U);
    int64_t *start = img.data() + 3 * U, *start_plain = start + U + 1;
    start[0] = start_plain[0] = 0;
    for (size_t b = 0; b < U; ++b) {
        const int group = group_of(cols[b], per_vec, most);
        start[b + 1] = start[b] + tiles_of(rows_with(b), by_warp ? rows_of<true>(group) : rows_of<false>(group));
        start_plain[b + 1] = start_plain[b] + rows_with(b);
    }
    cudaError_t e = cudaMalloc(&a->dmem, 8 * img.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(a->dmem, img.data(), 8 * img.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(nullptr);       // the tables are in place whatever stream reads them
    cudaSetDevice(prev);
    if (e != cudaSuccess) {
        if (a->dmem)
            cudaFree(a->dmem);
        delete a;
        return act_fail(e == cudaErrorMemoryAllocation ? GNMR_ERR_OOM : GNMR_ERR_CUDA,
                        std::string("actuator: ") + cudaGetErrorString(e));
    }
    const int64_t *base = static_cast<const int64_t *>(a->dmem);
    a->offset = base;
    a->rows = base + U;
    a->cols = base + 2 * U;
    a->start = base + 3 * U;
    a->start_plain = base + 4 * U + 1;
    a->num_units = num_units;
    a->dtype = dtype;
    a->device = device;
    a->most = most;
    a->tiles = start[U];
    a->tiles_plain = start_plain[U];
    a->max_end = max_end;
    a->any_long = any_long;
    a->any_held = any_held;
    a->by_warp = by_warp;
    a->sms = sms;
    *out = a;
    return GNMR_OK;
}

gnmr_status gnmr_actuator_apply(gnmr_actuator *a, const void *d_in, void *d_out, int64_t arena_elems,
                                const uint8_t *d_mask, int32_t lowcost_format, int32_t recovery_format,
                                void *stream)
{
    FqFmt low, rec;
    if (!a)
        return GNMR_ERR_INVALID_ARG;
    if (!fmt_of(lowcost_format, low) || !fmt_of(recovery_format, rec))
        return act_fail(GNMR_ERR_INVALID_ARG, "actuator: unknown format");
    if ((!d_in || !d_out) && a->max_end > 0)
        return act_fail(GNMR_ERR_INVALID_ARG, "actuator: NULL activation buffer");
    const int eb = a->dtype == GNMR_DTYPE_BF16 ? 2 : 4;
    if (reinterpret_cast<uintptr_t>(d_in) % eb || reinterpret_cast<uintptr_t>(d_out) % eb)
        return act_fail(GNMR_ERR_INVALID_ARG, "actuator: buffers not aligned to the element size");
    if (arena_elems < a->max_end)
        return act_fail(GNMR_ERR_LAYOUT, "actuator: buffer shorter than the layout");
    if (a->tiles == 0)
        return GNMR_OK;
    int prev = a->device;
    cudaGetDevice(&prev);
    if (prev != a->device)                        // switching costs as much as a tenth of a small launch
        cudaSetDevice(a->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const cudaError_t e = a->dtype == GNMR_DTYPE_BF16 ? launch<1>(*a, d_in, d_out, d_mask, low, rec, st)
                                                      : launch<0>(*a, d_in, d_out, d_mask, low, rec, st);
    if (e != cudaSuccess)
        cudaGetLastError();                       // reported here, not by the caller's next call
    if (prev != a->device)
        cudaSetDevice(prev);
    if (e != cudaSuccess)
        return act_fail(GNMR_ERR_CUDA, std::string("actuator launch: ") + cudaGetErrorString(e));
    return GNMR_OK;
}

gnmr_status gnmr_actuator_destroy(gnmr_actuator *a)
{
    if (!a)
        return GNMR_OK;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(a->device);
    const cudaError_t e = a->dmem ? cudaFree(a->dmem) : cudaSuccess;
    cudaSetDevice(prev);
    delete a;
    return e == cudaSuccess ? GNMR_OK : GNMR_ERR_CUDA;
}

}  // extern "C"
