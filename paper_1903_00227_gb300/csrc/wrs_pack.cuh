// wrs_pack.cuh -- the packing core of the sweep: Alg. 2 run by one warp on a
// stream of light and a stream of heavy items.  Included by wrs_kernels.cuh
// only.  Where a function is written in PTX, a second form without it lets
// the host compiler build the sweep, whose tests check every bucket store.
//
// With the keys of wrs_kernels.cuh (D[i]: deficits of the lights before
// light i; E[j]: excesses of the heavies up to and including heavy j) Alg. 2
// is a merge of the two key sequences, heavy j before light i iff
// E[j] <= D[i].  A warp keeps the next lights and heavies with their keys in
// two rings in shared memory and emits up to 63 buckets a step: lane l finds
// the heavies before light l among the next 32 by a five-step shuffle search,
// one OR-reduction gives the merged order, and lane p writes the buckets of the
// p-th and the (32 + p)-th item.  So a step costs the same whatever the mix of lights and
// heavies, no lane idles, a warp's stores go to two runs of near positions, the
// lights' and the heavies' (16-byte stores by lanes that each own a run of items
// cost 6.7 to 10 ms per 10^9 buckets on a GB300, consecutive ones 2.1 ms), and no
// warp waits for another.
#pragma once

namespace wrs {

// ------------------------------------------------------------- key types
// Signed two's complement integers.  K96 when n Q < 2^95 and shift = 0 (the
// usual case: every key, bucket and item weight n q then fits), else K128.
struct K96 {
    uint64_t lo;
    uint32_t hi;
};
struct K128 {
    uint64_t lo, hi;
};

template <int MODE> struct KeyOf { using T = K96; };
template <> struct KeyOf<2> { using T = K128; };

__device__ __forceinline__ K96 kadd(K96 a, K96 b)
{
    K96 r;
#ifdef __CUDA_ARCH__
    asm("add.cc.u64 %0, %2, %4;\n\taddc.u32 %1, %3, %5;" : "=l"(r.lo), "=r"(r.hi) : "l"(a.lo), "r"(a.hi), "l"(b.lo), "r"(b.hi));
#else
    r.lo = a.lo + b.lo;
    r.hi = a.hi + b.hi + (r.lo < a.lo);
#endif
    return r;
}
__device__ __forceinline__ K96 ksub(K96 a, K96 b)
{
    K96 r;
#ifdef __CUDA_ARCH__
    asm("sub.cc.u64 %0, %2, %4;\n\tsubc.u32 %1, %3, %5;" : "=l"(r.lo), "=r"(r.hi) : "l"(a.lo), "r"(a.hi), "l"(b.lo), "r"(b.hi));
#else
    r.lo = a.lo - b.lo;
    r.hi = a.hi - b.hi - (a.lo < b.lo);
#endif
    return r;
}
__device__ __forceinline__ K128 kadd(K128 a, K128 b)
{
    K128 r;
    const u128 s = (((u128)a.hi << 64) | a.lo) + (((u128)b.hi << 64) | b.lo);
    r.lo = (uint64_t)s;
    r.hi = (uint64_t)(s >> 64);
    return r;
}
__device__ __forceinline__ K128 ksub(K128 a, K128 b)
{
    K128 r;
    const u128 s = (((u128)a.hi << 64) | a.lo) - (((u128)b.hi << 64) | b.lo);
    r.lo = (uint64_t)s;
    r.hi = (uint64_t)(s >> 64);
    return r;
}
__device__ __forceinline__ bool kneg(K96 a) { return (int32_t)a.hi < 0; }
__device__ __forceinline__ bool kneg(K128 a) { return (int64_t)a.hi < 0; }
__device__ __forceinline__ bool kzero(K96 a) { return (a.lo | a.hi) == 0; }
__device__ __forceinline__ bool kzero(K128 a) { return (a.lo | a.hi) == 0; }
template <typename K> __device__ __forceinline__ bool keq(K a, K b) { return a.lo == b.lo && a.hi == b.hi; }
__device__ __forceinline__ K96 kmul(K96 a, uint32_t c) // a < 2^64
{
    const u128 p = (u128)a.lo * c;
    K96 r;
    r.lo = (uint64_t)p;
    r.hi = (uint32_t)(p >> 64);
    return r;
}
__device__ __forceinline__ K128 kmul(K128 a, uint32_t c)
{
    const u128 p = (((u128)a.hi << 64) | a.lo) * c;
    K128 r;
    r.lo = (uint64_t)p;
    r.hi = (uint64_t)(p >> 64);
    return r;
}
template <typename K> __device__ __forceinline__ bool kle(K a, K b) { return !kneg(ksub(b, a)); } // |b - a| in range
template <typename K> __device__ __forceinline__ K kunpack(uint4 v);
template <> __device__ __forceinline__ K96 kunpack<K96>(uint4 v)
{
    K96 r;
    r.lo = v.x | ((uint64_t)v.y << 32);
    r.hi = v.z;
    return r;
}
template <> __device__ __forceinline__ K128 kunpack<K128>(uint4 v)
{
    K128 r;
    r.lo = v.x | ((uint64_t)v.y << 32);
    r.hi = v.z | ((uint64_t)v.w << 32);
    return r;
}
template <typename K> __device__ __forceinline__ K kof(u128 v)
{
    return kunpack<K>(make_uint4((uint32_t)v, (uint32_t)(v >> 32), (uint32_t)(v >> 64), (uint32_t)(v >> 96)));
}
__device__ __forceinline__ K96 kshfl_up(K96 a, int d)
{
    K96 r;
    r.lo = __shfl_up_sync(0xFFFFFFFFu, a.lo, d);
    r.hi = __shfl_up_sync(0xFFFFFFFFu, a.hi, d);
    return r;
}
__device__ __forceinline__ K128 kshfl_up(K128 a, int d)
{
    K128 r;
    r.lo = __shfl_up_sync(0xFFFFFFFFu, a.lo, d);
    r.hi = __shfl_up_sync(0xFFFFFFFFu, a.hi, d);
    return r;
}

__device__ __forceinline__ K96 kshfl(K96 a, int src)
{
    K96 r;
    r.lo = __shfl_sync(0xFFFFFFFFu, a.lo, src);
    r.hi = __shfl_sync(0xFFFFFFFFu, a.hi, src);
    return r;
}
__device__ __forceinline__ K128 kshfl(K128 a, int src)
{
    K128 r;
    r.lo = __shfl_sync(0xFFFFFFFFu, a.lo, src);
    r.hi = __shfl_sync(0xFFFFFFFFu, a.hi, src);
    return r;
}

// Shifts whose counts at and above the width give 0
__device__ __forceinline__ uint64_t shl64(uint64_t v, uint32_t s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s > 63 ? 0 : v << s;
#endif
}
__device__ __forceinline__ uint32_t shl32(uint32_t v, uint32_t s) // 0 for counts of 32 and more
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
#else
    return s > 31 ? 0 : v << s;
#endif
}
__device__ __forceinline__ uint32_t shr32(uint32_t v, uint32_t s)
{
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
#else
    return s > 31 ? 0 : v >> s;
#endif
}
__device__ __forceinline__ uint64_t shr64(uint64_t v, uint32_t s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s > 63 ? 0 : v >> s;
#endif
}

// What a builder's items share: Q, the factor of q, the threshold shift, and
// how a word becomes n q.  With M the word's significand scaled to 32 bits
// and ex its exponent field, q = M 2^-(c0 - ex): for q < 2^32 a shift to the
// right (exact: q is an integer) before the 32 x 32 -> 64 multiply by n, else
// a shift of the product.
//   Q32  keys of type K96 (n Q < 2^95), every q below 2^32
//   Q96  keys of type K96, every light's q below 2^32
//   Q128 keys of type K128 (any weights)
// In the first two no weight is subnormal and a zero weight shifts out.
enum PackMode { kPackQ32, kPackQ96, kPackQ128 };
template <int F32, int MODE>
struct Units {
    using K = typename KeyOf<MODE>::T;
    K Q;
    uint32_t n32;
    int32_t c0;      // 158 + beta
    uint32_t shift;

    __device__ __forceinline__ void init(u128 q, uint64_t n, int beta, uint32_t shift_)
    {
        Q = kof<K>(q);
        n32 = (uint32_t)n;
        c0 = 158 + beta;
        shift = shift_;
    }
    __device__ __forceinline__ K nq(uint32_t x) const
    {
        K r;
        if (!F32) {
            r.lo = (uint64_t)x * n32;
            r.hi = 0;
        } else if (MODE == kPackQ32) {
            r.lo = (uint64_t)shr32((x << 8) | 0x80000000u, (uint32_t)(c0 - (int)(x >> 23))) * n32; // a zero weight: 0
            r.hi = 0;
        } else {
            const uint32_t ex = x >> 23;
            const uint32_t M = (x << 8) | (min(ex, 1u) << 31);
            const int s = c0 - (int)max(ex, 1u);
            const uint64_t P = (uint64_t)M * n32;
            // counts outside 0 .. 63 (also wrapped ones) give 0
            r.lo = shr64(P, (uint32_t)s) | shl64(P, (uint32_t)-s);
            if (MODE == kPackQ96) r.hi = (decltype(r.hi))shr64(P, (uint32_t)(64 + s));
            else r.hi = (decltype(r.hi))(shr64(P, (uint32_t)(64 + s)) | shl64(P, (uint32_t)(-s - 64)));
        }
        return r;
    }
    // n q of a light word (n q <= Q): below 2^64, or 2^95 in the wide mode
    __device__ __forceinline__ K96 nq_light(uint32_t x) const
    {
        K96 r;
        r.hi = 0;
        if (MODE != kPackQ128) { // q < 2^32
            r.lo = (F32 ? (uint64_t)shr32((x << 8) | 0x80000000u, (uint32_t)(c0 - (int)(x >> 23))) : (uint64_t)x) * n32;
            return r;
        }
        const K k = nq(x);
        r.lo = k.lo;
        r.hi = (uint32_t)k.hi;
        return r;
    }
    __device__ __forceinline__ uint64_t thr(K bw) const
    {
        if (MODE != kPackQ128) return bw.lo;
        return shr64(bw.lo, shift) | shl64((uint64_t)bw.hi, 64u - shift);
    }
};

constexpr int kPackBlocks = 24;          // blocks of the sweep (one warp each) per SM

// One warp's rings: the first kRing entries are lights by rank, the others heavies by
// rank.  Per entry the low word of the key relative to the task's first D (and
// the next 32 bits in the wide mode), the 32-bit key, the position.
template <int MODE> struct WarpRings {
    static constexpr bool kWide = MODE == kPackQ128;
    static constexpr int kPer = kWide ? 2 : 4;             // weights a lane reads at once
    static constexpr uint32_t kBatch = 32 * kPer;
    static constexpr uint32_t kRing = kWide ? 128 : 256;   // entries of a ring
    static_assert(32 + kBatch + 1 <= kRing, "what is left over, a batch and an end entry");
    uint64_t low[2 * kRing];
    uint2 kp[2 * kRing];     // (32-bit key, position)
    uint32_t high[kWide ? 2 * kRing : 1];
    __device__ __forceinline__ static uint32_t light(uint32_t r) { return r & (kRing - 1); }
    __device__ __forceinline__ static uint32_t heavy(uint32_t r) { return kRing | (r & (kRing - 1)); }
    template <typename K> __device__ __forceinline__ void put(uint32_t e, K v, uint32_t k32, uint32_t pos)
    {
        low[e] = v.lo;
        if (kWide) high[e] = (uint32_t)v.hi;
        kp[e] = make_uint2(k32, pos);
    }
};
constexpr size_t kPackSmemBytes = sizeof(WarpRings<kPackQ32>);
static_assert(sizeof(WarpRings<kPackQ128>) <= kPackSmemBytes, "rings");

// 32-bit keys: the relative key shifted down so that every D of the task is
// below 2^30.  Equal ones are told apart by the exact low words (they differ
// by less than 2^63, or 2^95 in the wide mode).  A task has at most 2^kTaskBits
// lights, so its D span less than 2^(64 + kTaskBits), as Q < 2^64, or
// 2^(kQBits + kTaskBits) in the wide mode, and 30 bits of that stay above the shift.
constexpr int kTaskBits = 13;
static_assert(64 + kTaskBits - 30 < 63, "kshr32 of a K96, and ties in 64 bits");
static_assert(kQBits + kTaskBits - 30 < 95, "kshr32 of a K128, and ties in 96 bits");
template <typename K> struct KeyFrame {
    K dmax;        // last D of the task, relative to its first
    uint32_t s;
};
template <typename K> __device__ __forceinline__ uint32_t kbits(K a) // bit length of a >= 0
{
    return a.hi ? 128u - (uint32_t)__clzll((long long)(uint64_t)a.hi)
                : (a.lo ? 64u - (uint32_t)__clzll((long long)a.lo) : 0u);
}
template <typename K> __device__ __forceinline__ KeyFrame<K> key_frame(K dmax)
{
    KeyFrame<K> f;
    f.dmax = dmax;
    const uint32_t b = kbits(dmax);
    f.s = b > 30 ? b - 30 : 0;
    return f;
}
// low 32 bits of v >> s
__device__ __forceinline__ uint32_t kshr32(K96 v, uint32_t s) // s < 64
{
    const uint32_t w1 = (uint32_t)(v.lo >> 32);
    return s < 32 ? __funnelshift_r((uint32_t)v.lo, w1, s) : __funnelshift_r(w1, v.hi, s);
}
__device__ __forceinline__ uint32_t kshr32(K128 v, uint32_t s) // s < 96
{
    const uint32_t w1 = (uint32_t)(v.lo >> 32), w2 = (uint32_t)v.hi, w3 = (uint32_t)(v.hi >> 32);
    const uint32_t a = s < 32 ? (uint32_t)v.lo : s < 64 ? w1 : w2, b = s < 32 ? w1 : s < 64 ? w2 : w3;
    return __funnelshift_r(a, b, s);
}
template <typename K> __device__ __forceinline__ uint32_t key32_light(const KeyFrame<K> &f, K v) { return kshr32(v, f.s); }
// -1 below the task's D, the largest value above them
template <typename K> __device__ __forceinline__ uint32_t key32_heavy(const KeyFrame<K> &f, K v)
{
    if (kneg(v)) return 0xFFFFFFFFu;
    return kle(v, f.dmax) ? key32_light(f, v) : 0x7FFFFFFFu;
}

__device__ __forceinline__ K96 kadd96(K96 a, K96 b) { return kadd(a, b); }
__device__ __forceinline__ K128 kadd96(K128 a, K96 b) { return kadd(a, K128{b.lo, b.hi}); }
__device__ __forceinline__ K96 kadd64(K96 a, uint64_t b)
{
    K96 r;
#ifdef __CUDA_ARCH__
    asm("add.cc.u64 %0, %2, %4;\n\taddc.u32 %1, %3, 0;" : "=l"(r.lo), "=r"(r.hi) : "l"(a.lo), "r"(a.hi), "l"(b));
#else
    r.lo = a.lo + b;
    r.hi = a.hi + (r.lo < b);
#endif
    return r;
}
// What one item adds to its list's keys: a light's deficit Q - n q (below
// 2^64, or 2^96 in the wide mode), a heavy's excess n q - Q.
template <int MODE> struct Light {
    uint64_t d;
    __device__ __forceinline__ Light() : d(0) {}
    template <typename U> __device__ __forceinline__ void set(const U &u, uint32_t x, bool on)
    {
        d = on ? u.Q.lo - u.nq_light(x).lo : 0;
    }
    __device__ __forceinline__ K96 add(K96 a) const { return kadd64(a, d); }
};
template <> struct Light<kPackQ128> {
    K96 d;
    __device__ __forceinline__ Light() : d{0, 0} {}
    template <typename U> __device__ __forceinline__ void set(const U &u, uint32_t x, bool on)
    {
        d = ksub(K96{u.Q.lo, (uint32_t)u.Q.hi}, u.nq_light(x));
        if (!on) d = K96{0, 0};
    }
    __device__ __forceinline__ K128 add(K128 a) const { return kadd96(a, d); }
};
template <int MODE> struct Heavy {
    typename KeyOf<MODE>::T d;
    __device__ __forceinline__ Heavy() : d{0, 0} {}
    template <typename U> __device__ __forceinline__ void set(const U &u, uint32_t x, bool on)
    {
        d = ksub(u.nq(x), u.Q);
        if (!on) d = typename KeyOf<MODE>::T{0, 0};
    }
    __device__ __forceinline__ typename KeyOf<MODE>::T add(typename KeyOf<MODE>::T a) const { return kadd(a, d); }
};
template <> struct Heavy<kPackQ32> {
    uint64_t d; // n q < 2^64
    __device__ __forceinline__ Heavy() : d(0) {}
    template <typename U> __device__ __forceinline__ void set(const U &u, uint32_t x, bool on)
    {
        d = on ? u.nq(x).lo - u.Q.lo : 0;
    }
    __device__ __forceinline__ K96 add(K96 a) const { return kadd64(a, d); }
};

// Inclusive warp scan (the shuffle's own predicate guards the additions).
__device__ __forceinline__ K96 warp_scan_key(K96 v)
{
#ifdef __CUDA_ARCH__
    uint32_t a = (uint32_t)v.lo, b = (uint32_t)(v.lo >> 32), c = v.hi;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile("{\n\t.reg .u32 x, y, z;\n\t.reg .pred p;\n\t"
                     "shfl.sync.up.b32 x|p, %0, %3, 0, 0xFFFFFFFF;\n\t"
                     "shfl.sync.up.b32 y, %1, %3, 0, 0xFFFFFFFF;\n\t"
                     "shfl.sync.up.b32 z, %2, %3, 0, 0xFFFFFFFF;\n\t"
                     "@p add.cc.u32 %0, %0, x;\n\t@p addc.cc.u32 %1, %1, y;\n\t@p addc.u32 %2, %2, z;\n\t}"
                     : "+r"(a), "+r"(b), "+r"(c) : "r"(d));
    v.lo = a | ((uint64_t)b << 32);
    v.hi = c;
#else
    for (int d = 1; d < 32; d <<= 1) {
        const K96 o = kshfl_up(v, d);
        if ((threadIdx.x & 31) >= (uint32_t)d) v = kadd(v, o);
    }
#endif
    return v;
}
__device__ __forceinline__ K128 warp_scan_key(K128 v)
{
#ifdef __CUDA_ARCH__
    uint32_t a = (uint32_t)v.lo, b = (uint32_t)(v.lo >> 32), c = (uint32_t)v.hi, e = (uint32_t)(v.hi >> 32);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile("{\n\t.reg .u32 x, y, z, t;\n\t.reg .pred p;\n\t"
                     "shfl.sync.up.b32 x|p, %0, %4, 0, 0xFFFFFFFF;\n\t"
                     "shfl.sync.up.b32 y, %1, %4, 0, 0xFFFFFFFF;\n\t"
                     "shfl.sync.up.b32 z, %2, %4, 0, 0xFFFFFFFF;\n\t"
                     "shfl.sync.up.b32 t, %3, %4, 0, 0xFFFFFFFF;\n\t"
                     "@p add.cc.u32 %0, %0, x;\n\t@p addc.cc.u32 %1, %1, y;\n\t@p addc.cc.u32 %2, %2, z;\n\t"
                     "@p addc.u32 %3, %3, t;\n\t}"
                     : "+r"(a), "+r"(b), "+r"(c), "+r"(e) : "r"(d));
    v.lo = a | ((uint64_t)b << 32);
    v.hi = c | ((uint64_t)e << 32);
#else
    for (int d = 1; d < 32; d <<= 1) {
        const K128 o = kshfl_up(v, d);
        if ((threadIdx.x & 31) >= (uint32_t)d) v = kadd(v, o);
    }
#endif
    return v;
}

// Member counts ride in the top bits of a scanned sum: bits 22 .. 31 of a
// K96 (sums of at most 128 values below 2^79), bits 54 .. 63 of a K128's high
// word (below 2^111).
__device__ __forceinline__ K96 kput(K96 v, uint32_t c) { v.hi += c << 22; return v; }
__device__ __forceinline__ K128 kput(K128 v, uint32_t c) { v.hi += (uint64_t)c << 54; return v; }
__device__ __forceinline__ uint32_t kcount(K96 v) { return v.hi >> 22; }
__device__ __forceinline__ uint32_t kcount(K128 v) { return (uint32_t)(v.hi >> 54); }
__device__ __forceinline__ K96 kvalue(K96 v) { v.hi &= (1u << 22) - 1u; return v; }
__device__ __forceinline__ K128 kvalue(K128 v) { v.hi &= (1ull << 54) - 1ull; return v; }

// This lane's N weights from at + N lane on that lie below `end`; `fill` past it.
template <int N>
__device__ __forceinline__ void load_lane(const uint32_t *__restrict__ w, int vec, uint64_t at, uint64_t end,
                                          uint32_t fill, uint32_t (&x)[N])
{
    const uint64_t i = at + N * (threadIdx.x & 31);
    if (N == 4 && vec && i + N <= end) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(w + i));
        x[0] = v.x; x[1] = v.y; x[N - 2] = v.z; x[N - 1] = v.w;
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = i + k < end ? __ldg(w + i + k) : fill;
    }
}

// Bit k: weight at + N lane + k lies below `end`.
template <int N> __device__ __forceinline__ uint32_t lane_words(uint64_t at, uint64_t end)
{
    const uint64_t i = at + N * (threadIdx.x & 31);
    return i >= end ? 0u : (1u << min((uint64_t)N, end - i)) - 1u;
}

// Ranks of this lane's members (mask m, bit k: item k) among the warp's, in
// item order; tot: the warp's members.
template <int N> __device__ __forceinline__ uint32_t warp_rank(uint32_t m, uint32_t &tot)
{
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
    uint32_t r = 0;
    tot = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, (m >> k) & 1u);
        r += (uint32_t)__popc(b & lt);
        tot += (uint32_t)__popc(b);
    }
    return r;
}

} // namespace wrs
