// Streaming sum of squares over a gradient segment and the completion
// ticket, shared by the step kernel and the allocation-free norms entry point
// (device code only).
//
// A warp reads a segment with 16-byte loads (no L1 allocation, 256-byte L2
// prefetch), squares in fp32, sums short blocks in
// fp32 and the blocks as an unevaluated pair of floats (hi + lo, about 48
// significant bits), then adds the 32 lanes' totals in fixed point (exact from
// the lanes' rounding to 26 bits on; a five-level fp32 tree over the lanes may be
// 3e-7 off) and forms the fp64 result once per segment.  It flags segments whose
// fp32 squares may have lost accuracy (denormal or overflowing squares), which
// the caller recomputes with exact fp64 squares.  Any element alignment: a scalar
// head and tail around the 16-byte body.
//
// Error of a unit's norm against 64 bits, root mean square over the units of a
// layout (normal values): fp32 units of 8 KB 3.7e-9, of 120 KB 9.5e-10, of 1.2 MB
// 4.3e-10, of 12 MB 3.3e-10; with an fp32 tree over the lanes (and one run per warp
// in the small-unit loop) 1.9e-8, 1.2e-8, 3.7e-9 and 1.5e-9.  bf16 units: 5.7e-9 to
// 6.6e-9 at every size, with the tree 6.1e-9 (units of 6 MB) to 2.0e-8 (4 KB).  What
// is left there is a common offset of about -5.8e-9, the same as with the tree,
// whose scatter lay around it: a bf16 square ends in the bits 001 or in zeros, so
// rounding the first sums of a few to fp32 drops more than it adds.
//
// Why float pairs: on GB300 an fp64 add has a 64-cycle dependent latency and
// the SM retires one fp64 warp-instruction every 20 cycles, shared by all its
// warps.  A five-round fp64 shuffle reduction per segment held that pipe 40 %
// of the time on layouts of many small units and stalled the streams; the
// fp32 error-free additions run on the fp32 pipe.  The pairs keep a long run
// of blocks accurate.  The lanes' sum is three warp reductions of integers
// (redux), with no fp64 instruction at all.
#ifndef GNMR_STREAM_CUH
#define GNMR_STREAM_CUH

#include <cstdint>

namespace gnmr {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kFlush = 16;   // main-loop iterations summed in fp32 before the pair add

template <int DT> struct Elem;
template <> struct Elem<0> {             // fp32
    static constexpr int kBytes = 4;
    static constexpr uint32_t kMagnitude = 0x7fffffffu;
};
template <> struct Elem<1> {             // bf16, two per 32-bit word
    static constexpr int kBytes = 2;
    static constexpr uint32_t kMagnitude = 0x7fff7fffu;
};

// 16-byte streaming load: no L1 allocation, 256-byte L2 prefetch granularity.
// A coherent load, and volatile like the element loads below: a kernel that
// was started early (griddepcontrol) knows its addresses before the data is
// written, so no load may move up over the wait.
constexpr int kVecWords = 4;
constexpr int kVecBytes = 16;
struct alignas(kVecBytes) Vec {
    uint32_t w[kVecWords];
};

__device__ __forceinline__ Vec ld_stream(const Vec *p)
{
    Vec r;
    asm volatile("ld.global.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]) : "l"(p));
    return r;
}

__device__ __forceinline__ Vec zero_vec()
{
    Vec r;
#pragma unroll
    for (int i = 0; i < kVecWords; ++i)
        r.w[i] = 0u;
    return r;
}

__device__ __forceinline__ uint32_t vec_or(const Vec &v)
{
    uint32_t o = 0;
#pragma unroll
    for (int i = 0; i < kVecWords; ++i)
        o |= v.w[i];
    return o;
}

// One element as an fp32 bit pattern (bf16 is the upper half of an fp32).
template <int DT> __device__ __forceinline__ uint32_t ld_elem_bits(const char *p);
template <> __device__ __forceinline__ uint32_t ld_elem_bits<0>(const char *p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
template <> __device__ __forceinline__ uint32_t ld_elem_bits<1>(const char *p)
{
    uint16_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return static_cast<uint32_t>(v) << 16;
}

// Sum of squares of the elements packed in one vector, in fp32 (two
// independent chains per vector).
template <int DT> __device__ __forceinline__ float vec_sumsq(const Vec &v);
template <> __device__ __forceinline__ float vec_sumsq<0>(const Vec &v)
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int i = 0; i < kVecWords; i += 2) {
        const float a = __uint_as_float(v.w[i]), b = __uint_as_float(v.w[i + 1]);
        s0 = fmaf(a, a, s0);
        s1 = fmaf(b, b, s1);
    }
    return s0 + s1;
}
template <> __device__ __forceinline__ float vec_sumsq<1>(const Vec &v)
{
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int i = 0; i < kVecWords; ++i) {
        const float lo = __uint_as_float(v.w[i] << 16);
        const float hi = __uint_as_float(v.w[i] & 0xffff0000u);
        s0 = fmaf(lo, lo, s0);
        s1 = fmaf(hi, hi, s1);
    }
    return s0 + s1;
}

__device__ __forceinline__ double warp_allreduce_sum(double v)
{
    // xor butterfly: both partners add the same two operands, so every lane
    // ends with the same bits.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Knuth's TwoSum: s + e == a + b exactly, s = fl(a + b), in any operand
// order (fl(a + b) == fl(b + a), and e is the exact rounding error).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fadd_rn(s, -a);
    e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb));
}

// (hi, lo) += x for an unevaluated pair hi + lo.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float x)
{
    float s, e;
    two_sum(hi, x, s, e);
    hi = s;
    lo = __fadd_rn(lo, e);
}

// Sum of squares of kN vectors, their fp32 sums added pairwise; bits: or of all of
// their words.
template <int DT, int kN> __device__ __forceinline__ float vecs_sumsq(const Vec (&r)[kN], uint32_t &bits)
{
    float a[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
        a[j] = vec_sumsq<DT>(r[j]);
        bits |= vec_or(r[j]);
    }
#pragma unroll
    for (int n = kN; n > 1; n = (n + 1) / 2)
#pragma unroll
        for (int j = 0; j < n / 2; ++j)
            a[j] += a[j + (n + 1) / 2];
    return a[0];
}

// The same of vectors q[0], q[32], ... as far as their places are below `rest`, at
// most kN of them.
template <int DT, int kN> __device__ __forceinline__ float rest_sumsq(const Vec *q, int32_t rest, uint32_t &bits)
{
    Vec r[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j)
        r[j] = j * 32 < rest ? ld_stream(q + j * 32) : zero_vec();
    return vecs_sumsq<DT, kN>(r, bits);
}

// Sum of squares of n elements at seg, by the whole warp.  Returns the sum
// in every lane and sets `suspect` when fp32 squaring may have lost accuracy:
// a nonzero segment whose largest lane total is below 2^-100 (denormal squares),
// at least 2^100 (possible fp32 overflow), or NaN or Inf.
template <int DT, int kUnroll>
__device__ __forceinline__ double warp_segment_sumsq(const char *seg, int64_t n, int lane,
                                                     bool &suspect)
{
    constexpr int kEB = Elem<DT>::kBytes;
    constexpr int kVE = kVecBytes / kEB;
    constexpr uint32_t kAlign = kVecBytes - 1;
    const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(seg) & kAlign);
    int64_t head = static_cast<int64_t>(((kVecBytes - mis) & kAlign) / kEB);
    head = head < n ? head : n;
    const int64_t nvec = (n - head) / kVE;
    const int64_t tail = n - head - nvec * kVE;

    uint32_t bits = 0;
    float blk = 0.f;
    if (lane < head) {
        const uint32_t w = ld_elem_bits<DT>(seg + lane * kEB);
        const float x = __uint_as_float(w);
        bits |= w;
        blk = fmaf(x, x, blk);
    }
    if (lane < tail) {
        const uint32_t w = ld_elem_bits<DT>(seg + (head + nvec * kVE + lane) * kEB);
        const float x = __uint_as_float(w);
        bits |= w;
        blk = fmaf(x, x, blk);
    }

    const Vec *v = reinterpret_cast<const Vec *>(seg + head * kEB);
    float acc_hi = 0.f, acc_lo = 0.f;
    int cnt = 0;
    int64_t base = 0;                                     // the same in every lane: all take the same rounds
    for (; base + kUnroll * 32 <= nvec; base += kUnroll * 32) {
        Vec r[kUnroll];
#pragma unroll
        for (int j = 0; j < kUnroll; ++j)
            r[j] = ld_stream(v + base + lane + j * 32);
        blk += vecs_sumsq<DT, kUnroll>(r, bits);
        if (++cnt == kFlush) {
            pair_add(acc_hi, acc_lo, blk);
            blk = 0.f;
            cnt = 0;
        }
    }
    // Fewer than kUnroll vectors left for some lane: one predicated batch, as short
    // as will do.  (Where lanes that could fill a batch took a full one and the others
    // then a predicated one of kUnroll - 1, a piece that did not end within a warp's
    // row of vectors waited twice for its last loads, and every piece summed that
    // many slots.  Partial sums of 10,000 log-normal bf16 units, 90 MB: 19.4 -> 17.1 us,
    // the whole step 25.3 -> 23.0; 3,000 fp32 ones, 60 MB: 12.6 -> 11.5 and 17.9 -> 17.0;
    // 100,000 fp32 units, 1.6 GB: 238.5 -> 238.2.  Indexed from v: with a pointer that
    // moves along the last one took 239.5.)
    const int32_t left = static_cast<int32_t>(nvec - base), rest = left - lane;
    const Vec *q = v + base + lane;
    if (left > kUnroll * 24)
        blk += rest_sumsq<DT, kUnroll>(q, rest, bits);
    else if (left > kUnroll * 16)
        blk += rest_sumsq<DT, kUnroll * 3 / 4>(q, rest, bits);
    else if (left > 0)
        blk += rest_sumsq<DT, kUnroll / 2>(q, rest, bits);
    pair_add(acc_hi, acc_lo, blk);
    // The lanes' totals (non-negative) added as 26-bit fractions of twice the
    // largest one's power of two: the integer sum is exact and the same in every
    // lane, and a lane's rounding to its fraction is at most 2^-26 of the largest
    // total.  As fast as a five-level fp32 xor tree, with a quarter to a thirteenth of
    // its scatter (figures at the head of this file).
    const uint32_t tot = __float_as_uint(acc_hi + acc_lo);
    const uint32_t e = __reduce_max_sync(kFull, tot) >> 23;                    // > 254 for NaN and Inf
    suspect = false;
    if (e - 27u >= 200u) {                                // the largest not in [2^-100, 2^100)
        suspect = (__reduce_or_sync(kFull, bits) & Elem<DT>::kMagnitude) != 0u;
        return 0.0;
    }
    const uint32_t own = tot >> 23;
    const uint32_t sh = min(e - own, 27u);
    const uint32_t frac = own ? ((tot & 0x7fffffu) | 0x800000u) << 2 : 0u;     // 26 bits
    const uint32_t sum = __reduce_add_sync(kFull, (frac + ((1u << sh) >> 1)) >> sh);
    // sum * 2^(e - 152) in binary64, put together on the integer pipe
    const uint32_t lz = __clz(sum);
    const uint32_t m = sum << (lz + 1);
    const double acc = __hiloint2double(static_cast<int>(((902u + e - lz) << 20) | (m >> 12)), static_cast<int>(m << 20));
    return acc;
}

// Sums of squares of several short segments at once: the lanes in groups of
// `lanes` (4, 8 or 16), each streaming n elements at seg with at most kVecs
// vectors a lane.  Returns the group's sum in every lane of it and sets
// `suspect` as warp_segment_sumsq() does, by group.  Called by all 32 lanes.
template <int DT, int kVecs>
__device__ __forceinline__ double group_segment_sumsq(const char *seg, int32_t n, int lanes, int lane, bool &suspect)
{
    constexpr int kEB = Elem<DT>::kBytes;
    constexpr int kVE = kVecBytes / kEB;
    const int gl = lane & (lanes - 1);
    const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(seg)) & (kVecBytes - 1);
    const int32_t head = min(static_cast<int32_t>(((kVecBytes - mis) & (kVecBytes - 1)) / kEB), n);
    const int32_t nvec = (n - head) / kVE;
    const int32_t tail_at = head + nvec * kVE;

    const Vec *v = reinterpret_cast<const Vec *>(seg + head * kEB);
    Vec r[kVecs];
#pragma unroll
    for (int j = 0; j < kVecs; ++j)
        r[j] = gl + lanes * j < nvec ? ld_stream(v + gl + lanes * j) : zero_vec();
    uint32_t bits = 0;
    float edge = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {                          // up to 7 head and tail elements, 4 lanes at least
        if (k == 1 && lanes >= kVE)
            break;
        const int32_t at = gl + lanes * k;
        if (at < head) {
            const uint32_t w = ld_elem_bits<DT>(seg + at * kEB);
            bits |= w;
            edge = fmaf(__uint_as_float(w), __uint_as_float(w), edge);
        }
        if (tail_at + at < n) {
            const uint32_t w = ld_elem_bits<DT>(seg + (tail_at + at) * kEB);
            bits |= w;
            edge = fmaf(__uint_as_float(w), __uint_as_float(w), edge);
        }
    }
    const uint32_t tot = __float_as_uint(vecs_sumsq<DT, kVecs>(r, bits) + edge);
    uint32_t e = tot;
    for (int o = lanes / 2; o > 0; o >>= 1)
        e = max(e, __shfl_xor_sync(kFull, e, o));
    e >>= 23;                                             // > 254 for NaN and Inf
    const bool ok = e - 27u < 200u;
    suspect = false;
    if (__any_sync(kFull, !ok)) {
        for (int o = lanes / 2; o > 0; o >>= 1)
            bits |= __shfl_xor_sync(kFull, bits, o);
        suspect = !ok && (bits & Elem<DT>::kMagnitude) != 0u;
    }
    // in fixed point, as in warp_segment_sumsq()
    const uint32_t own = tot >> 23;
    const uint32_t sh = min(e - own, 27u);
    const uint32_t frac = own ? ((tot & 0x7fffffu) | 0x800000u) << 2 : 0u;
    uint32_t sum = (frac + ((1u << sh) >> 1)) >> sh;
    for (int o = lanes / 2; o > 0; o >>= 1)
        sum += __shfl_xor_sync(kFull, sum, o);
    const uint32_t lz = ok ? __clz(sum) : 0u;
    const uint32_t m = sum << (lz + 1);
    return ok ? __hiloint2double(static_cast<int>(((902u + e - lz) << 20) | (m >> 12)), static_cast<int>(m << 20)) : 0.0;
}

// Exact-product fallback: each element squared in fp64 (exact for fp32 and
// bf16 inputs) and summed in fp64.  Taken only for segments flagged suspect.
template <int DT>
__device__ __noinline__ double warp_segment_sumsq_f64(const char *seg, int64_t n, int lane)
{
    constexpr int kEB = Elem<DT>::kBytes;
    double acc = 0.0;
    for (int64_t i = lane; i < n; i += 32) {
        const double x = static_cast<double>(__uint_as_float(ld_elem_bits<DT>(seg + i * kEB)));
        acc = fma(x, x, acc);
    }
    return warp_allreduce_sum(acc);
}

// Ticket increment with acquire-release semantics at GPU scope: it publishes
// the caller's earlier writes (and, after a barrier, those of its CTA) and,
// for the caller that draws the last ticket, makes every earlier holder's
// writes visible.
__device__ __forceinline__ uint32_t ticket_acq_rel(uint32_t *t)
{
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(t) : "memory");
    return old;
}

}  // namespace
}  // namespace gnmr

#endif  // GNMR_STREAM_CUH
