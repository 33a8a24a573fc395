// wrs_kernels.cuh -- the kernels of the build and of the query.  Included by
// wrs.cu only.
//
// Build (alias table of n weights; Alg. 3 "PSA", Sec. 4.2, producing the
// table of Alg. 2, Sec. 4.1, bucket for bucket):
//   k_stats, k_stats_combine  W := sum w_i, exactly (opening line of Alg. 3)
//   k_classify  per tile of 2048 (or 256) weights: light/heavy classification (Alg. 3's
//               two traversals) and the tile's light and heavy weight sums
//               and counts (Sec. 4.2.2 "Using Block-Wise Prefix Sums": tiles
//               play the role of the blocks), plus the offsets of the tile's
//               heavies when they are few
//   k_tilescan  inclusive prefix of the tile aggregates: a single-pass scan
//               with decoupled look-back between thread blocks
//   k_split     per tile, Alg. 3's split search on the tile prefix sums
//   k_sweep     per run of tiles, the buckets of its lights and the heavies packed
//               with them (Alg. 3's pack)
// Query:
//   k_sample    k alias queries (Sec. 2.2; Sec. 5 Cor. "kWR"), branchless
//               selection between bucket and alias (Sec. 10, "Optimizations").
//
// Units (exact): q_i is the integer weight, Q = sum q_i, a bucket holds Q and
// item i weighs n*q_i.  With the light list l and heavy list h in index
// order, light x (0-based rank) has key D[x] = x*Q - n*(q of lights before
// x) and heavy y has key E[y] = n*(q of heavies up to y) - (y+1)*Q.  Alg. 2
// packs heavy y before light x iff E[y] <= D[x] (its residual then fits).
// Hence the bucket of light x holds n*q with alias the first heavy y with
// E[y] > D[x], and the bucket of heavy y holds Q - (D[x] - E[y]) where x is
// the first light with D[x] >= E[y]; its alias is the next heavy item in
// index order (a full bucket points to itself).  Both are the split of
// Alg. 3 taken at one item: the state of Alg. 2 when that item is packed.
#pragma once

#include "wrs_device.cuh"
#include "wrs_pack.cuh"

namespace wrs {

// ------------------------------------------------------------- loading
__device__ __forceinline__ void load_items(const uint32_t *__restrict__ w, uint64_t n, int vec,
                                           uint64_t first, uint32_t (&x)[kItems])
{
    if (vec && first + kItems <= n) {
        const uint4 *p = reinterpret_cast<const uint4 *>(w + first);
#pragma unroll
        for (int j = 0; j < kItems / 4; ++j) {
            uint4 v = __ldg(p + j);
            x[4 * j + 0] = v.x; x[4 * j + 1] = v.y; x[4 * j + 2] = v.z; x[4 * j + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kItems; ++k) x[k] = (first + k < n) ? __ldg(w + first + k) : 0u;
    }
}

__device__ __forceinline__ TileSum load_prefix(const TileSum *incl, uint32_t b)
{
    TileSum p;
    if (b == 0) {
        p.l_lo = p.l_hi = p.h_lo = p.h_hi = 0;
        p.cl = 0;
    } else {
        const uint4 *src = reinterpret_cast<const uint4 *>(incl + (b - 1));
        uint4 a = __ldcg(src), c = __ldcg(src + 1), d = __ldcg(src + 2);
        p.l_lo = a.x | ((uint64_t)a.y << 32); p.l_hi = a.z | ((uint64_t)a.w << 32);
        p.h_lo = c.x | ((uint64_t)c.y << 32); p.h_hi = c.z | ((uint64_t)c.w << 32);
        p.cl = d.x;
    }
    return p;
}

// ------------------------------------------------------------ k_stats
// Per block: the exact sum of q over a grid-stride share of the weights, in
// units of 2^base with base the lowest set bit seen so far (rebased when a
// smaller one appears), plus validity flags.
struct Acc {
    int base;
    u128 acc;
    uint32_t flags;
    uint32_t mx;     // largest word
};

__device__ __forceinline__ void acc_merge(Acc &a, const Acc &b)
{
    a.flags |= b.flags;
    a.mx = max(a.mx, b.mx);
    if (b.base == INT_MAX) return;
    if (a.base == INT_MAX) { a.base = b.base; a.acc = b.acc; return; }
    u128 lo_acc = a.acc, hi_acc = b.acc;
    int lo_base = a.base, d = b.base - a.base;
    if (d < 0) { lo_acc = b.acc; hi_acc = a.acc; lo_base = b.base; d = -d; }
    if (hi_acc) {
        if (bitlen128(hi_acc) + d > kQBits) a.flags |= kPartOverflow;
        else lo_acc += hi_acc << d;
    }
    a.base = lo_base;
    a.acc = lo_acc;
    if (hi64(a.acc) >> (kQBits - 64)) a.flags |= kPartOverflow;
}

// Add one weight.  Addends below 2^61 (shift <= 37) go to the 64-bit side
// accumulator a64, which the caller folds into acc at least every 8 items.
template <int F32>
__device__ __forceinline__ void acc_take(Acc &a, uint64_t &a64, uint32_t x)
{
    if (!F32) { a64 += x; return; }
    const uint32_t ex = (x >> 23) & 0xFFu;
    a.mx = max(a.mx, x);
    if ((x >> 31) || ex == 0xFFu) { a.flags |= kPartInvalid; return; }
    uint32_t m = x & 0x7FFFFFu;
    if (ex) m |= 0x800000u;
    if (!m) return;
    const int e = (ex ? (int)ex : 1) - 150;
    const int lsb = e + __ffs(m) - 1;
    if (lsb < a.base) { // rare: a lower set bit than any before; rebase
        a.acc += a64;
        a64 = 0;
        if (a.acc) {
            const int d = a.base - lsb;
            if (bitlen128(a.acc) + d > kQBits) { a.flags |= kPartOverflow; a.acc = 0; }
            else a.acc <<= d;
        }
        a.base = lsb;
    }
    const int sh = e - a.base;
    if (sh <= 37) {
        a64 += sh >= 0 ? ((uint64_t)m << sh) : (uint64_t)(m >> (-sh));
    } else {
        if ((32 - __clz(m)) + sh > kQBits) { a.flags |= kPartOverflow; return; }
        a.acc += (u128)m << sh;
    }
}

__device__ __forceinline__ void acc_fold(Acc &a, uint64_t &a64)
{
    a.acc += a64;
    a64 = 0;
    if (hi64(a.acc) >> (kQBits - 64)) { a.flags |= kPartOverflow; a.acc = 0; }
}

__device__ __forceinline__ Acc acc_shfl_down(const Acc &a, int d)
{
    Acc b;
    b.base = __shfl_down_sync(0xFFFFFFFFu, a.base, d);
    b.acc = shfl_down128(a.acc, d);
    b.flags = __shfl_down_sync(0xFFFFFFFFu, a.flags, d);
    b.mx = __shfl_down_sync(0xFFFFFFFFu, a.mx, d);
    return b;
}

__device__ Acc acc_block_reduce(Acc a)
{
    __shared__ int s_base[kWarps];
    __shared__ u128 s_acc[kWarps];
    __shared__ uint32_t s_flags[kWarps], s_mx[kWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        Acc b = acc_shfl_down(a, d);
        acc_merge(a, b);
    }
    if (lane == 0) { s_base[wid] = a.base; s_acc[wid] = a.acc; s_flags[wid] = a.flags; s_mx[wid] = a.mx; }
    __syncthreads();
    if (wid == 0) {
        Acc b;
        if (lane < kWarps) { b.base = s_base[lane]; b.acc = s_acc[lane]; b.flags = s_flags[lane]; b.mx = s_mx[lane]; }
        else { b.base = INT_MAX; b.acc = 0; b.flags = 0; b.mx = 0; }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            Acc c = acc_shfl_down(b, d);
            acc_merge(b, c);
        }
        a = b;
    }
    return a; // valid in thread 0
}

// Add the exact value S * 2^(e0 - 150) of some weights, whose lowest set bit
// is at 2^(e0 - 150 + ctz(o)), to an accumulator kept in units of 2^base
// (base: the lowest set bit seen so far).
__device__ __forceinline__ void acc_add_chunk(Acc &a, uint64_t S, uint64_t o, int e0)
{
    const int lsb = e0 - 150 + __ffsll((long long)o) - 1;
    if (lsb < a.base) { // a lower set bit than any before: rebase
        if (a.acc) {
            const int d = a.base - lsb;
            if (bitlen128(a.acc) + d > kQBits) { a.flags |= kPartOverflow; a.acc = 0; }
            else a.acc <<= d;
        }
        a.base = lsb;
    }
    const int sh = e0 - 150 - a.base; // >= -ctz(o), and S is a multiple of 2^ctz(o)
    a.acc += sh >= 0 ? ((u128)S << sh) : (u128)(S >> (-sh));
    if (hi64(a.acc) >> (kQBits - 64)) { a.flags |= kPartOverflow; a.acc = 0; }
}

// Block `bid` of `nblk` blocks sharing the weights of one table; thread 0
// writes the block's partial to *out.  Binary32 weights go in warp chunks
// of 256 (lane l: weights 8l .. 8l+7): when each of a lane's eight is a
// normal number and the exponents of a lane's eight span at most 31
// binades, the lane forms their exact sum in 64 bits as sum m * 2^(e - e0)
// (e0: its smallest exponent; one multiply-add per weight) and their lowest
// set bit from the OR of those terms, and adds it to its accumulator; other
// weights take the exact per-weight path.
template <int F32>
__device__ __forceinline__ void stats_body(const uint32_t *__restrict__ w, uint64_t n, int vec, uint32_t bid,
                                           uint32_t nblk, Partial *__restrict__ out)
{
    Acc a;
    a.base = F32 ? INT_MAX : 0;
    a.acc = 0;
    a.flags = 0;
    a.mx = 0; // not needed for integer weights
    uint64_t a64 = 0;
    if (!F32) {
        const uint64_t tid = (uint64_t)bid * kThreads + threadIdx.x;
        const uint64_t nth = (uint64_t)nblk * kThreads;
        const uint64_t nv = vec ? n / 4 : 0;
        const uint4 *w4 = reinterpret_cast<const uint4 *>(w);
        uint64_t i = tid;
        for (; i + 3 * nth < nv; i += 4 * nth) {
            const uint4 v0 = __ldg(w4 + i), v1 = __ldg(w4 + i + nth), v2 = __ldg(w4 + i + 2 * nth), v3 = __ldg(w4 + i + 3 * nth);
            a64 += (uint64_t)v0.x + v0.y + v0.z + v0.w;
            a64 += (uint64_t)v1.x + v1.y + v1.z + v1.w;
            a64 += (uint64_t)v2.x + v2.y + v2.z + v2.w;
            a64 += (uint64_t)v3.x + v3.y + v3.z + v3.w;
        }
        for (; i < nv; i += nth) {
            const uint4 v = __ldg(w4 + i);
            a64 += (uint64_t)v.x + v.y + v.z + v.w;
        }
        for (uint64_t j = nv * 4 + tid; j < n; j += nth) a64 += __ldg(w + j);
        acc_fold(a, a64); // n < 2^32 words below 2^32: the total fits 64 bits
    } else {
        const uint32_t lane = threadIdx.x & 31;
        const uint64_t nchunks = (n + kChunk - 1) / kChunk;
        const uint64_t cw = (uint64_t)nblk * kWarps;
        uint32_t vmax = 0; // any word >= 0x7F800000 is Inf, NaN or has the sign bit set
        uint64_t c = (uint64_t)bid * kWarps + (threadIdx.x >> 5);
        uint32_t x[kItems];
        if (c < nchunks) load_items(w, n, vec, c * kChunk + lane * kItems, x);
        for (; c < nchunks; c += cw) {
            const uint64_t first = c * kChunk + lane * kItems;
            uint32_t xn[kItems];
            const bool more = c + cw < nchunks;
            if (more) load_items(w, n, vec, (c + cw) * kChunk + lane * kItems, xn);
            bool fast = (c + 1) * kChunk <= n; // a full chunk
            uint32_t e0 = 0;
            if (fast) {
                uint32_t emin = 0xFFFFFFFFu, emax = 0;
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    vmax = max(vmax, x[k]);
                    const uint32_t ex = x[k] >> 23; // >= 255 for Inf, NaN and negative words
                    emin = min(emin, ex);
                    emax = max(emax, ex);
                }
                e0 = emin;
                fast = e0 >= 1 && emax < 255 && emax - e0 <= 31; // this lane's eight: normal, finite, 31 binades
            }
            if (fast) {
                uint64_t sum = 0, orr = 0;
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    const uint32_t m = (x[k] & 0x7FFFFFu) | 0x800000u;
                    const uint64_t v = (uint64_t)m * (1u << ((x[k] >> 23) - e0)); // < 2^55
                    sum += v;
                    orr |= v;
                }
                acc_add_chunk(a, sum, orr, (int)e0); // this lane's eight terms (orr > 0: every m has its top bit)
            } else {
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    if (first + k < n) {
                        acc_take<1>(a, a64, x[k]);
                        acc_fold(a, a64);
                    }
                }
            }
            if (more) {
#pragma unroll
                for (int k = 0; k < kItems; ++k) x[k] = xn[k];
            }
        }
        if (vmax >= 0x7F800000u) a.flags |= kPartInvalid;
        a.mx = max(a.mx, vmax);
    }
    a = acc_block_reduce(a);
    if (threadIdx.x == 0) {
        Partial p;
        p.lo = lo64(a.acc); p.hi = hi64(a.acc); p.base = a.base; p.flags = a.flags; p.mx = a.mx; p.mode = 0;
        *out = p;
    }
}

template <int F32>
__global__ void __launch_bounds__(kThreads) k_stats(const uint32_t *__restrict__ w, uint64_t n, int vec,
                                                    Partial *__restrict__ part)
{
    stats_body<F32>(w, n, vec, blockIdx.x, gridDim.x, part + blockIdx.x);
}

// Is n * val(v) <= Q * 2^beta for the binary32 pattern v (v >= +0, finite)?
__device__ bool f32_light(uint32_t v, uint64_t n, u128 Q, int beta)
{
    uint32_t ex = (v >> 23) & 0xFFu, m = v & 0x7FFFFFu;
    if (ex) m |= 0x800000u;
    if (!m) return true;
    int d = (ex ? (int)ex : 1) - 150 - beta;
    u128 nm = (u128)m * n;
    if (d >= 0) {
        if (bitlen128(nm) + d > 127) return false;
        return (nm << d) <= Q;
    }
    int dd = -d;
    if (bitlen128(Q) + dd > 127) return true;
    return nm <= (Q << dd);
}

__device__ __forceinline__ uint32_t write_header(const Acc &a, uint64_t n, uint32_t f32, DevHeader *hdr, uint32_t &mode);

__device__ __forceinline__ void stats_combine_body(Partial *part, uint32_t nparts, uint64_t n,
                                                   uint32_t f32, DevHeader *hdr)
{
    Acc a;
    a.base = INT_MAX; a.acc = 0; a.flags = 0; a.mx = 0;
    for (uint32_t i = threadIdx.x; i < nparts; i += kThreads) {
        Partial p = part[i];
        Acc b;
        b.base = p.base; b.acc = mk128(p.lo, p.hi); b.flags = p.flags; b.mx = p.mx;
        if (!f32) b.base = 0;
        acc_merge(a, b);
    }
    a = acc_block_reduce(a);
    // every thread has read its partials before the reduction's barrier
    if (threadIdx.x == 0) write_header(a, n, f32, hdr, part[0].mode);
}

// The table header from the exact total (thread 0): status, beta, Q, shift,
// qp and the light threshold on the raw words; and how the sweep forms n q and
// its keys (PackMode), which is not the caller's business and goes to `mode`.
__device__ __forceinline__ uint32_t write_header(const Acc &a, uint64_t n, uint32_t f32, DevHeader *hdr, uint32_t &mode)
{
    uint32_t status = kOk;
    if (a.flags & kPartInvalid) status = kEInval;
    else if (a.flags & kPartOverflow) status = kEOverflow;
    else if (a.acc == 0) status = kEInval;
    const u128 Q = a.acc;
    int shift = bitlen128(Q) - 64;
    if (shift < 0) shift = 0;
    uint32_t light_max = 0;
    int beta = f32 ? (a.base == INT_MAX ? 0 : a.base) : 0;
    if (status == kOk) {
        if (!f32) {
            light_max = (uint32_t)(lo64(Q) / n); // Q < 2^64, Q/n < 2^32
        } else {
            uint32_t lo = 0, hi = 0x7F7FFFFFu; // largest v with f32_light(v)
            while (lo < hi) {
                uint32_t mid = lo + (hi - lo + 1) / 2;
                if (f32_light(mid, n, Q, beta)) lo = mid; else hi = mid - 1;
            }
            light_max = lo;
        }
    }
    hdr->tile_counter = 0;
    hdr->beta = beta;
    hdr->shift = (uint32_t)shift;
    hdr->q_lo = lo64(Q);
    hdr->q_hi = hi64(Q);
    hdr->qp = lo64(Q >> shift);
    hdr->light_max = light_max;
    mode = kPackQ128;
    if (shift == 0 && bitlen128(Q) + (32 - __clz((int)(uint32_t)n)) <= 95) {
        const bool normal = !f32 || beta >= -94;
        if (normal && (!f32 || (int)(a.mx >> 23) <= 158 + beta)) mode = kPackQ32;
        else if (normal && (int)(light_max >> 23) <= 158 + beta) mode = kPackQ96;
    }
    hdr->f32 = f32;
    hdr->n = n;
    hdr->n_light = 0;
    hdr->pad[0] = 0;
    hdr->pad[1] = 0;
    __threadfence();
    hdr->status = status;
    return status;
}

__global__ void __launch_bounds__(kThreads) k_stats_combine(Partial *part, uint32_t nparts,
                                                            uint64_t n, uint32_t f32, DevHeader *hdr)
{
    stats_combine_body(part, nparts, n, f32, hdr);
}

// ---------------------------------------------------------- k_classify
// q of a weight known to be below 2^61 (shift <= 37)
__device__ __forceinline__ uint64_t q64_of(uint32_t x, uint32_t f32, int beta)
{
    if (!f32) return x;
    const uint32_t ex = (x >> 23) & 0xFFu;
    uint32_t m = x & 0x7FFFFFu;
    if (ex) m |= 0x800000u;
    const int sh = (ex ? (int)ex : 1) - 150 - beta;
    return sh >= 0 ? ((uint64_t)m << sh) : (uint64_t)(m >> (-sh));
}

__device__ __forceinline__ void tilesum_st(TileSum *p, const TileSum &v)
{
    uint4 *d = reinterpret_cast<uint4 *>(p);
    d[0] = make_uint4((uint32_t)v.l_lo, (uint32_t)(v.l_lo >> 32), (uint32_t)v.l_hi, (uint32_t)(v.l_hi >> 32));
    d[1] = make_uint4((uint32_t)v.h_lo, (uint32_t)(v.h_lo >> 32), (uint32_t)v.h_hi, (uint32_t)(v.h_hi >> 32));
    d[2] = make_uint4(v.cl, v.nheavy, v.first_heavy, 0u);
}

__device__ __forceinline__ TileSum tilesum_ldcg(const TileSum *p)
{
    const uint4 *s = reinterpret_cast<const uint4 *>(p);
    uint4 a = __ldcg(s), c = __ldcg(s + 1), d = __ldcg(s + 2);
    TileSum r;
    r.l_lo = a.x | ((uint64_t)a.y << 32); r.l_hi = a.z | ((uint64_t)a.w << 32);
    r.h_lo = c.x | ((uint64_t)c.y << 32); r.h_hi = c.z | ((uint64_t)c.w << 32);
    r.cl = d.x; r.nheavy = d.y; r.first_heavy = d.z; r.pad = d.w;
    return r;
}

// Sum of a u128 over the warp, returned to every lane: the warp-wide
// reduction instruction adds 16-bit limbs exactly (each limb's sum over 32
// lanes is below 2^21); the high half is skipped when every lane's is zero.
__device__ __forceinline__ u128 warp_sum128(u128 v)
{
    const uint64_t lo = lo64(v), hi = hi64(v);
    u128 r = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        r += (u128)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)(lo >> (16 * c)) & 0xFFFFu) << (16 * c);
    if (__any_sync(0xFFFFFFFFu, hi != 0)) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            r += (u128)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)(hi >> (16 * c)) & 0xFFFFu) << (64 + 16 * c);
    }
    return r;
}

// Exclusive scan of a u32 over the warp.
__device__ __forceinline__ uint32_t warp_excl_scan_u32(uint32_t v)
{
    const int lane = threadIdx.x & 31;
    uint32_t s = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, s, d);
        if (lane >= d) s += o;
    }
    return s - v;
}

// Tiles t_first, t_first + t_stride, ... of one table, ONE WARP per tile
// (no block barrier per tile).  A tile is TILE / 256 chunks of 256 weights; lane
// l holds weights 8l .. 8l+7 of a chunk.  Per tile: light count, light and
// heavy sums of q, heavy count, offset of the first heavy, and the offsets of
// its heavies when it has at most kSparseOf(TILE) of them.
template <int F32, int TILE>
__device__ __forceinline__ void classify_body(const uint32_t *__restrict__ w, uint64_t n, int vec,
                                              const DevHeader *__restrict__ hdr, TileSum *__restrict__ agg,
                                              uint16_t *__restrict__ slist, uint32_t ntiles, uint32_t t_first,
                                              uint32_t t_stride)
{
    constexpr int kTile = TILE, kChunks = TILE / kChunk, kSparse = kSparseOf(TILE);
    __shared__ uint16_t s_list[kWarps][kSparse];
    if (block_stopped(hdr)) return;
    const uint32_t light_max = hdr->light_max;
    const int beta = hdr->beta;
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint16_t *list = s_list[wid];
    uint32_t x[kItems];
    if (t_first < ntiles) load_items(w, n, vec, (uint64_t)t_first * kTile + lane * kItems, x);
    for (uint32_t t = t_first; t < ntiles; t += t_stride) {
        const uint64_t tile0 = (uint64_t)t * kTile;
        u128 Lp = 0, Hp = 0;             // this lane's light and heavy sums over the tile (units of 2^beta)
        uint32_t cl = 0, ch = 0;          // this lane's light and heavy counts
        uint32_t chp = 0, fh = kNone;     // heavies before the chunk (kept while at most kSparse), first heavy
#pragma unroll 1
        for (uint32_t c = 0; c < (uint32_t)kChunks; ++c) {
            const uint64_t first = tile0 + c * kChunk + lane * kItems;
            const bool full = tile0 + (c + 1) * kChunk <= n; // the same in every lane
            uint32_t lm = 0, vm = 0xFFu;
            uint32_t emin = 0xFFFFFFFFu, emax = 0;
            if (full) {
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    if (x[k] <= light_max) lm |= 1u << k;
                    if (F32) {
                        const uint32_t ex = x[k] >> 23; // a valid word has its sign bit clear
                        emin = min(emin, ex);
                        emax = max(emax, ex);
                    }
                }
            } else {
                vm = 0;
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    if (first + k < n) {
                        vm |= 1u << k;
                        if (x[k] <= light_max) lm |= 1u << k;
                    }
                }
            }
            const uint32_t hm = vm & ~lm;
            bool chunk_fast = false;
            uint32_t e0 = 0;
            if (F32 && full) {
                e0 = __reduce_min_sync(0xFFFFFFFFu, emin);
                chunk_fast = e0 >= 1 && __reduce_max_sync(0xFFFFFFFFu, emax) - e0 <= 31;
            }
            if (chunk_fast) {
                // every weight normal, exponents within 31 binades: m * 2^(e - e0)
                // in 64 bits (one multiply-add each, below 2^58 per lane), then
                // scaled to units of 2^beta (exact: every term q * 2^-sh is a
                // multiple of 2^-sh when sh < 0)
                uint64_t l64 = 0, h64 = 0;
#pragma unroll
                for (int k = 0; k < kItems; ++k) {
                    const uint64_t v = (uint64_t)((x[k] & 0x7FFFFFu) | 0x800000u) * (1u << ((x[k] >> 23) - e0));
                    if ((lm >> k) & 1u) l64 += v; else h64 += v;
                }
                const int sh = (int)e0 - 150 - beta;
                Lp += sh >= 0 ? (u128)l64 << sh : (u128)(l64 >> (-sh));
                Hp += sh >= 0 ? (u128)h64 << sh : (u128)(h64 >> (-sh));
            } else {
                bool narrow = true; // every q below 2^61: eight of them fit 64 bits
                if (F32) {
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        const uint32_t ex = (x[k] >> 23) & 0xFFu;
                        if (((vm >> k) & 1u) && (ex ? (int)ex : 1) - 150 - beta > 37) narrow = false;
                    }
                }
                if (narrow) {
                    uint64_t l64 = 0, h64 = 0;
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        const uint64_t q = q64_of(x[k], F32, beta);
                        if ((lm >> k) & 1u) l64 += q;
                        if ((hm >> k) & 1u) h64 += q;
                    }
                    Lp += l64;
                    Hp += h64;
                } else {
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        if ((vm >> k) & 1u) {
                            const u128 q = q_of(x[k], F32, beta);
                            if ((lm >> k) & 1u) Lp += q; else Hp += q;
                        }
                    }
                }
            }
            cl += (uint32_t)__popc(lm);
            ch += (uint32_t)__popc(hm);
            // prefetch the next chunk (or the next tile's first)
            const uint64_t nf = c + 1 < (uint32_t)kChunks ? first + kChunk
                                                          : (uint64_t)(t + t_stride) * kTile + lane * kItems;
            const bool more = c + 1 < (uint32_t)kChunks || t + t_stride < ntiles;
            if (chp <= (uint32_t)kSparse || fh == kNone) {
                const uint32_t hb = __ballot_sync(0xFFFFFFFFu, hm != 0);
                if (fh == kNone && hb) {
                    const int src = __ffs(hb) - 1;
                    const uint32_t hs = __shfl_sync(0xFFFFFFFFu, hm, src);
                    fh = c * kChunk + (uint32_t)src * kItems + (uint32_t)(__ffs(hs) - 1);
                }
                if (chp <= (uint32_t)kSparse && hb) { // offsets of the first heavies, in order
                    uint32_t pos = chp + warp_excl_scan_u32((uint32_t)__popc(hm));
#pragma unroll
                    for (int k = 0; k < kItems; ++k) {
                        if ((hm >> k) & 1u) {
                            if (pos < (uint32_t)kSparse) list[pos] = (uint16_t)(c * kChunk + lane * kItems + k);
                            ++pos;
                        }
                    }
                    chp += __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(hm));
                }
            }
            if (more) load_items(w, n, vec, nf, x);
        }
        const u128 L = warp_sum128(Lp), H = warp_sum128(Hp);
        const uint32_t tl = __reduce_add_sync(0xFFFFFFFFu, cl), th = __reduce_add_sync(0xFFFFFFFFu, ch);
        __syncwarp();
        if (lane == 0) {
            TileSum a;
            a.l_lo = lo64(L); a.l_hi = hi64(L); a.h_lo = lo64(H); a.h_hi = hi64(H);
            a.cl = tl; a.nheavy = th; a.first_heavy = fh; a.pad = 0;
            tilesum_st(agg + t, a);
        }
        if (th <= (uint32_t)kSparse && lane < th) slist[(uint64_t)t * kSparse + lane] = list[lane];
        __syncwarp();
    }
}

template <int F32, int TILE>
__global__ void __launch_bounds__(kThreads) k_classify(const uint32_t *__restrict__ w, uint64_t n, int vec,
                                                       const DevHeader *__restrict__ hdr, TileSum *__restrict__ agg,
                                                       uint16_t *__restrict__ slist, uint32_t ntiles)
{
    classify_body<F32, TILE>(w, n, vec, hdr, agg, slist, ntiles, blockIdx.x * kWarps + (threadIdx.x >> 5),
                       gridDim.x * kWarps);
}

// ---------------------------------------------------------- k_tilescan
// Inclusive prefix of the tile aggregates.  Each block takes 256 consecutive
// tiles (block ids in launch order from an atomic counter, so every block it
// waits for is already running), scans them, publishes the chunk aggregate,
// then warp 0 looks back over the predecessors' published values until it
// meets an inclusive prefix, and publishes its own.  Every wait is bounded by
// `wait_limit` polls: a wait that runs out stores WRS_ETIMEOUT and the block
// carries on, so no block ever waits forever.
__device__ __forceinline__ void tilesum_add(TileSum &a, const TileSum &b)
{
    u128 l = mk128(a.l_lo, a.l_hi) + mk128(b.l_lo, b.l_hi);
    u128 h = mk128(a.h_lo, a.h_hi) + mk128(b.h_lo, b.h_hi);
    a.l_lo = lo64(l); a.l_hi = hi64(l); a.h_lo = lo64(h); a.h_hi = hi64(h);
    a.cl += b.cl;
}

__device__ __forceinline__ TileSum tilesum_shfl_xor(const TileSum &a, int m)
{
    TileSum b;
    b.l_lo = __shfl_xor_sync(0xFFFFFFFFu, a.l_lo, m); b.l_hi = __shfl_xor_sync(0xFFFFFFFFu, a.l_hi, m);
    b.h_lo = __shfl_xor_sync(0xFFFFFFFFu, a.h_lo, m); b.h_hi = __shfl_xor_sync(0xFFFFFFFFu, a.h_hi, m);
    b.cl = __shfl_xor_sync(0xFFFFFFFFu, a.cl, m);
    b.nheavy = 0; b.first_heavy = kNone; b.pad = 0;
    return b;
}

__device__ __forceinline__ void tilescan_body(DevHeader *hdr, const TileSum *__restrict__ agg, TileSum *chunk_agg,
                                              TileSum *chunk_incl, TileSum *__restrict__ incl, uint32_t *flags,
                                              uint32_t ntiles, uint32_t epoch, uint32_t wait_limit,
                                              uint32_t skip_chunk)
{
    __shared__ uint32_t s_chunk, s_status;
    __shared__ U2 s_scan[kWarps];
    __shared__ uint32_t s_cnt[kWarps];
    __shared__ TileSum s_ex;
    if (threadIdx.x == 0) {
        s_status = *(volatile uint32_t *)&hdr->status;
        s_chunk = s_status ? 0u : atomicAdd(&hdr->tile_counter, 1u);
    }
    __syncthreads();
    if (s_status) return;
    const uint32_t c = s_chunk;
    const uint32_t t = c * kScanChunk + threadIdx.x;
    TileSum a;
    if (t < ntiles) a = tilesum_ldcg(agg + t);
    else { a.l_lo = a.l_hi = a.h_lo = a.h_hi = 0; a.cl = 0; a.nheavy = 0; a.first_heavy = kNone; a.pad = 0; }
    U2 tot;
    const U2 ex = block_exclusive_scan2(U2{mk128(a.l_lo, a.l_hi), mk128(a.h_lo, a.h_hi)}, tot, s_scan);
    uint32_t ctot;
    const uint32_t cex = block_exclusive_scan_u32(a.cl, ctot, s_cnt);
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        TileSum ca;
        ca.l_lo = lo64(tot.a); ca.l_hi = hi64(tot.a); ca.h_lo = lo64(tot.b); ca.h_hi = hi64(tot.b);
        ca.cl = ctot; ca.nheavy = 0; ca.first_heavy = kNone; ca.pad = 0;
        const bool publish = (c != skip_chunk);
        TileSum exc;
        exc.l_lo = exc.l_hi = exc.h_lo = exc.h_hi = 0; exc.cl = 0; exc.nheavy = 0; exc.first_heavy = kNone; exc.pad = 0;
        if (c == 0) {
            if (lane == 0) {
                tilesum_st(chunk_incl, ca);
                if (publish) st_release(flags, (epoch << 2) | kFlagIncl);
            }
        } else {
            if (lane == 0) {
                tilesum_st(chunk_agg + c, ca);
                if (publish) st_release(flags + c, (epoch << 2) | kFlagAgg);
            }
            int64_t p = (int64_t)c - 1 - lane;
            bool timed_out = false;
            for (;;) {
                uint32_t st = kFlagIncl; // virtual predecessor before chunk 0
                if (p >= 0) {
                    uint32_t polls = 0;
                    for (;;) {
                        const uint32_t fv = ld_acquire(flags + p);
                        st = ((fv >> 2) == epoch) ? (fv & 3u) : 0u;
                        if (st != 0u || ++polls >= wait_limit) break;
                        __nanosleep(32);
                    }
                }
                if (__any_sync(0xFFFFFFFFu, st == 0u)) { timed_out = true; break; }
                const uint32_t incl_mask = __ballot_sync(0xFFFFFFFFu, st == kFlagIncl);
                const int stop = incl_mask ? __ffs(incl_mask) - 1 : 32;
                TileSum v;
                if (lane <= stop && p >= 0) v = tilesum_ldcg(st == kFlagIncl ? chunk_incl + p : chunk_agg + p);
                else { v.l_lo = v.l_hi = v.h_lo = v.h_hi = 0; v.cl = 0; }
#pragma unroll
                for (int m = 16; m > 0; m >>= 1) {
                    TileSum o = tilesum_shfl_xor(v, m);
                    tilesum_add(v, o);
                }
                tilesum_add(exc, v);
                if (incl_mask) break;
                p -= 32;
            }
            if (lane == 0) {
                if (timed_out) set_status(hdr, kETimeout);
                TileSum r = ca;
                tilesum_add(r, exc);
                tilesum_st(chunk_incl + c, r);
                if (publish) st_release(flags + c, (epoch << 2) | kFlagIncl);
            }
        }
        if (lane == 0) s_ex = exc;
    }
    __syncthreads();
    if (t < ntiles) {
        TileSum r;
        const u128 l = mk128(s_ex.l_lo, s_ex.l_hi) + ex.a + mk128(a.l_lo, a.l_hi);
        const u128 h = mk128(s_ex.h_lo, s_ex.h_hi) + ex.b + mk128(a.h_lo, a.h_hi);
        r.l_lo = lo64(l); r.l_hi = hi64(l); r.h_lo = lo64(h); r.h_hi = hi64(h);
        r.cl = s_ex.cl + cex + a.cl;
        r.nheavy = a.nheavy; r.first_heavy = a.first_heavy; r.pad = 0;
        tilesum_st(incl + t, r);
    }
}

__global__ void __launch_bounds__(kThreads) k_tilescan(DevHeader *hdr, const TileSum *__restrict__ agg,
                                                       TileSum *chunk_agg, TileSum *chunk_incl,
                                                       TileSum *__restrict__ incl, uint32_t *flags,
                                                       uint32_t ntiles, uint32_t epoch, uint32_t wait_limit,
                                                       uint32_t skip_chunk)
{
    tilescan_body(hdr, agg, chunk_agg, chunk_incl, incl, flags, ntiles, epoch, wait_limit, skip_chunk);
}

// ------------------------------------------------------------ k_split
// For every tile boundary c = 0 .. ntiles, from the tile prefix sums: the
// keys there (D: of the first light from tile c on, E: after the heavies
// before tile c), the tile's heavies, the table's PackMode, and
//   hb = max{ b : E(b) <= D(c) }  -- the tile holding the first heavy item
//        with E > D(c), the heavy current when the first light from tile c
//        on is packed (the split of Alg. 3 on the heavy prefix sums);
//   next_heavy = position of the first heavy item after tile c.
struct Prefix {
    uint64_t cl, ch;
    u128 L, H;
};

template <int TILE> __device__ __forceinline__ Prefix prefix_at(const TileSum *incl, uint32_t b, uint64_t n)
{
    TileSum t = load_prefix(incl, b);
    Prefix p;
    p.cl = t.cl;
    uint64_t end = (uint64_t)b * TILE;
    if (end > n) end = n;
    p.ch = end - p.cl;
    p.L = mk128(t.l_lo, t.l_hi);
    p.H = mk128(t.h_lo, t.h_hi);
    return p;
}

__device__ __forceinline__ u128 key_E(const Prefix &p, uint64_t n, u128 Q) { return times_n(p.H, n) - (u128)p.ch * Q; }
__device__ __forceinline__ u128 key_D(const Prefix &p, uint64_t n, u128 Q) { return (u128)p.cl * Q - times_n(p.L, n); }

// Boundary c of one table (one thread per boundary); part: its first partial.
template <int TILE>
__device__ __forceinline__ void split_body(const TileSum *__restrict__ incl, uint32_t ntiles, uint64_t n,
                                           DevHeader *hdr, const Partial *__restrict__ part,
                                           Split *__restrict__ split, uint32_t c)
{
    if (*(volatile uint32_t *)&hdr->status) return;
    const u128 Q = mk128(hdr->q_lo, hdr->q_hi);
    const uint64_t n_light = load_prefix(incl, ntiles).cl;
    if (c == 0) hdr->n_light = n_light;
    if (c > ntiles) return;
    const Prefix pc = prefix_at<TILE>(incl, c, n);
    const u128 Dc = key_D(pc, n, Q), Ec = key_E(pc, n, Q);
    uint32_t lo = 0, hi = ntiles;
    while (lo < hi) {
        uint32_t mid = lo + (hi - lo + 1) / 2;
        if (key_E(prefix_at<TILE>(incl, mid, n), n, Q) <= Dc) lo = mid; else hi = mid - 1;
    }
    Split s;
    s.hb = lo;
    s.nheavy = 0;
    s.next_heavy = kNone;
    s.mode = part->mode;
    s.d_lo = lo64(Dc); s.d_hi = hi64(Dc);
    s.e_lo = lo64(Ec); s.e_hi = hi64(Ec);
    if (c < ntiles) {
        const Prefix pn = prefix_at<TILE>(incl, c + 1, n);
        const uint64_t total_h = n - n_light;
        s.nheavy = (uint32_t)(pn.ch - pc.ch);
        if (pn.ch < total_h) { // heavy rank pn.ch is the first heavy of tile max{b : ch(b) <= pn.ch}
            lo = c + 1; hi = ntiles - 1;
            while (lo < hi) {
                uint32_t mid = lo + (hi - lo + 1) / 2;
                if (prefix_at<TILE>(incl, mid, n).ch <= pn.ch) lo = mid; else hi = mid - 1;
            }
            const TileSum tb = tilesum_ldcg(incl + lo);
            s.next_heavy = lo * (uint32_t)TILE + tb.first_heavy;
        }
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(&s);
    uint4 *dst = reinterpret_cast<uint4 *>(split + c);
    dst[0] = src[0]; dst[1] = src[1]; dst[2] = src[2];
}

template <int TILE>
__global__ void __launch_bounds__(kThreads) k_split(const TileSum *__restrict__ incl, uint32_t ntiles, uint64_t n,
                                                    DevHeader *hdr, const Partial *__restrict__ part,
                                                    Split *__restrict__ split)
{
    split_body<TILE>(incl, ntiles, n, hdr, part, split, blockIdx.x * kThreads + threadIdx.x);
}

// ------------------------------------------------------------ k_sweep
// A task is a run of consecutive tiles c_first .. c_last - 1 (one subproblem
// of Alg. 3): one warp packs the lights of these tiles and every heavy item
// whose key E lies in (D(c_first), D(c_last)], exactly the items Alg. 2 packs
// while it consumes these lights (wrs_pack.cuh).  The lights come from the
// tiles themselves, 128 weights at a time; the heavies in index order from the
// tile k_split named for the first of them, 128 weights at a time from a dense
// tile or by the member lists of a run of sparse tiles (at most
// kSparseOf(TILE) heavies each), until one lies past the task's last D.  While
// the current heavy reaches past every light of the next 128-weight batches
// (its key is that far ahead), the lights go straight from the loaded words to
// their buckets: Zipf 1.5 has 2000 lights per heavy.
//
// Bound by instruction issue (n = 10^8 uniform: 9.5 warp instructions per
// weight at 70 % issue; about 290 per batch of own weights, 320 per batch of
// heavies' tile, 115 per search and 64 per 32 buckets stored).  It replaces a
// block per eight tiles with 128-bit keys of a whole tile in shared memory, a
// merge walked by threads and five barriers a tile.  It moves 41 B of DRAM per
// weight for 20 of work (uniform): outputs leave in merge order, where a light's
// and a heavy's 16-byte buckets share 32-byte sectors, and the resident warps'
// tasks span some 480 MB of buckets, so the L2 evicts sectors half written.
// n = 10^8, uniform / Zipf
// 0.8 / Zipf 1.5: 1.54 / 1.50 / 1.18 -> 1.18 / 1.22 / 0.42 ms; n = 10^9 uniform
// 15.4 -> 10.9 ms, Zipf 1.5 12.2 -> 3.6 ms.  One warp per block: the scheduler
// replaces each warp as it ends, 19 -> 23 resident warps per SM (1.47 -> 1.40 ms
// uniform).  The rings fit 24 warps per SM, the registers (80) too.
__device__ __forceinline__ uint4 split_head(const Split *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
template <typename K> __device__ __forceinline__ K split_D(const Split *p)
{
    return kunpack<K>(__ldg(reinterpret_cast<const uint4 *>(p) + 1));
}
template <typename K> __device__ __forceinline__ K split_E(const Split *p)
{
    return kunpack<K>(__ldg(reinterpret_cast<const uint4 *>(p) + 2));
}

constexpr uint32_t kDirect = 128;        // weights a warp packs at once under one far heavy
// Own tiles per task at most.  More tiles share a task's start (its split
// record, its first heavies' tile), fewer leave a shorter last wave and lights
// and heavies that lie closer together: 1 / 2 / 4 / 8 / 16 tiles take 6.45 /
// 6.38 / 6.62 / 6.90 / 7.36 ms for n = 6*10^8 uniform, 3.83 / 3.61 / 3.57 /
// 3.61 / 3.81 ms for n = 10^9 Zipf 1.5, and 6.98 / 6.63 / 6.54 / 6.57 / - ms
// for n = 6*10^8 Zipf 0.8.  (The 32-bit keys would cover 2^14 Q, eight tiles.)
constexpr int kSweepTiles = 4;
static_assert(kSweepTiles * kTile <= 1 << kTaskBits, "the 32-bit keys' range");

template <int F32, int MODE, int TILE>
__device__ __forceinline__ bool sweep_task(WarpRings<MODE> &R, const uint32_t *__restrict__ w, uint64_t n, int vec,
                                           DevHeader *hdr, const Split *__restrict__ split,
                                           const uint16_t *__restrict__ slist, uint32_t ntiles,
                                           uint4 *__restrict__ table, uint32_t c_first, uint32_t c_last, u128 Q)
{
    using K = typename Units<F32, MODE>::K;
    constexpr bool kWide = MODE == kPackQ128;
    constexpr int kTile = TILE, kSparse = kSparseOf(TILE);
    constexpr int kPer = WarpRings<MODE>::kPer;
    constexpr uint32_t kBatch = WarpRings<MODE>::kBatch, kRing = WarpRings<MODE>::kRing;
    const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    const uint32_t light_max = hdr->light_max;
    Units<F32, MODE> U;
    U.init(Q, n, hdr->beta, hdr->shift);
    bool bad = false;

    // lights: ranks [li, lh) are in the ring, weights from `at` on are not read yet (x: the next batch)
    // Words past `end` read as 0xFFFFFFFF.  No binary32 table has a light threshold
    // that high, but u32 weights that are all 0xFFFFFFFF have: there the last
    // batch's words are told apart by their index.
    uint64_t at = (uint64_t)c_first * kTile;
    const uint64_t end = min((uint64_t)c_last * kTile, n);
    uint32_t li = 0, lh = 0, x[kPer];
    load_lane(w, vec, at, end, 0xFFFFFFFFu, x);
    const K d_base = split_D<K>(split + c_first);
    const KeyFrame<K> f = key_frame(ksub(split_D<K>(split + c_last), d_base));
    K drun{0, 0}; // D of light lh
    // heavies: ranks [hj, hh) are in the ring; the next come from weight sa of tile s on (y: the next batch)
    uint32_t s = split_head(split + c_first).x;
    uint32_t hj = 0, hh = 0, y[kPer];
    uint4 rs = make_uint4(0, 0, 0, 0);
    uint64_t sa = 0, send = 0;
    bool past = false;  // the last heavy in the ring lies past the task's last D
    K erun{0, 0};       // E of heavy hh - 1
    if (s < ntiles) {
        rs = split_head(split + s);
        erun = ksub(split_E<K>(split + s), d_base);
        sa = (uint64_t)s * kTile;
        send = min(sa + kTile, n);
        if (rs.z > (uint32_t)kSparse) load_lane(w, vec, sa, send, 0u, y);
    }
    if (lane == 0) R.kp[R.heavy(0)].y = kNone;

    // 128 Q in units of the 32-bit keys, rounded up: the most a batch of lights can add to D
    const uint32_t batch_units = min(kshr32(kmul(U.Q, kDirect), f.s) + 2u, 1u << 30);
    const bool far_batches = kbits(kmul(U.Q, kDirect)) < f.s + 30;
    if (lane == 0) R.put(R.light(0), drun, 0u, kNone);

    for (;;) {
        check_ok(lh - li < kRing && hh - hj < kRing, hdr); // the rings hold their entries and the end entry
        if (lh - li < 32 && at < end && (hh != hj || s >= ntiles)) { // the next own weights
            // Direct: the current heavy reaches past every light of the next
            // batches, so these lights go straight from the weights to their buckets.
            const uint32_t klast = R.kp[R.light(lh)].x; // of D[lh]
            const uint32_t kfirst = hh == hj ? 0u : R.kp[R.heavy(hj)].x;
            uint32_t batches = 0;
            if (far_batches && (int32_t)kfirst > 0) {
                if (kfirst == 0x7FFFFFFFu) batches = 1u << 20;
                else if (kfirst > klast + batch_units) batches = (kfirst - klast - 1) / batch_units;
            }
            if (batches >= 2 && li == lh) {
                const uint32_t hp = R.kp[R.heavy(hj)].y;
                K sum{0, 0};
                K96 Ql;
                Ql.lo = U.Q.lo;
                Ql.hi = (uint32_t)U.Q.hi;
                uint32_t z[4], c = 0;
                const uint64_t left = (end - at + kDirect - 1) / kDirect;
                if (batches > left) batches = (uint32_t)left;
#pragma unroll
                for (int k = 0; k < 4; ++k) z[k] = at + 32 * k + lane < end ? __ldg(w + at + 32 * k + lane) : 0xFFFFFFFFu;
                for (;;) {
                    uint32_t zn[4];
                    const uint64_t an = at + kDirect;
                    const bool more = c + 1 < batches;
                    if (more) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) zn[k] = an + 32 * k + lane < end ? __ldg(w + an + 32 * k + lane) : 0xFFFFFFFFu;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (z[k] <= light_max && (F32 || at + 32 * k + lane < end)) {
                            const K96 nq = U.nq_light(z[k]);
                            const K96 df = ksub(Ql, nq);
                            sum = kadd96(sum, df);
                            const uint32_t me = (uint32_t)at + 32 * k + lane;
                            K bw;
                            bw.lo = nq.lo;
                            bw.hi = nq.hi;
                            put_bucket(table, me, U.thr(bw), kzero(df) ? me : hp, n, hdr);
                        }
                    }
                    at = an;
                    ++c;
                    if (!more) break;
#pragma unroll
                    for (int k = 0; k < 4; ++k) z[k] = zn[k];
                }
                if (at < end) load_lane(w, vec, at, end, 0xFFFFFFFFu, x);
                drun = kadd(drun, kshfl(warp_scan_key(sum), 31));
                lh += kRing; // the same entry; ranks only have to differ from the task's first light's, 0
                li = lh;
                if (lane == 0) R.put(R.light(lh), drun, key32_light(f, drun), kNone);
                __syncwarp();
                continue;
            }
            if (batches < 2) {
                uint32_t m = 0;
#pragma unroll
                for (int k = 0; k < kPer; ++k)
                    if (x[k] <= light_max) m |= 1u << k;
                if (!F32 && at + kBatch > end) m &= lane_words<kPer>(at, end); // the fill may be light
                Light<MODE> v[kPer];
                K sum{0, 0};
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    v[k].set(U, x[k], (m >> k) & 1u);
                    sum = v[k].add(sum);
                }
                const uint32_t pos = (uint32_t)at + kPer * lane;
                at += kBatch;
                if (at < end) load_lane(w, vec, at, end, 0xFFFFFFFFu, x);
                sum = kput(sum, (uint32_t)__popc(m));
                const K exc = ksub(warp_scan_key(sum), sum);
                K run = kadd(drun, kvalue(exc));
                uint32_t r = lh + kcount(exc);
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    if ((m >> k) & 1u) {
                        const uint32_t e = R.light(r);
                        R.put(e, run, key32_light(f, run), pos + k);
                        ++r;
                    }
                    run = v[k].add(run);
                }
                if (lane == 31) R.put(R.light(r), run, key32_light(f, run), kNone); // the entry after the last light
                drun = kshfl(run, 31);
                lh = __shfl_sync(0xFFFFFFFFu, r, 31);
                __syncwarp();
                continue;
            }
        }
        if (hh - hj < 33 && !past && s < ntiles) { // the next batch of heavies (the last one's alias is the one after it)
            uint32_t tot;
            if (rs.z > (uint32_t)kSparse) {
                uint32_t m = 0;
#pragma unroll
                for (int k = 0; k < kPer; ++k)
                    if (y[k] > light_max) m |= 1u << k; // past the end: never heavy
                uint32_t r = 0;
                if (MODE != kPackQ32) r = hh + warp_rank<kPer>(m, tot); // the sums may need their top bits
                Heavy<MODE> v[kPer];
                K sum{0, 0};
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    v[k].set(U, y[k], (m >> k) & 1u);
                    sum = v[k].add(sum);
                }
                const uint32_t pos = (uint32_t)sa + kPer * lane;
                sa += kBatch;
                bool next_tile = false;
                if (sa < send) load_lane(w, vec, sa, send, 0u, y);
                else next_tile = true;
                if (MODE == kPackQ32) sum = kput(sum, (uint32_t)__popc(m));
                const K inc = warp_scan_key(sum);
                K exc = ksub(inc, sum);
                if (MODE == kPackQ32) {
                    r = hh + kcount(exc);
                    exc = kvalue(exc);
                }
                K run = kadd(erun, exc);
                bool skip = false; // every heavy of the batch comes before the task's first light
                if (hh == 0) {
                    K after = run;
#pragma unroll
                    for (int k = 0; k < kPer; ++k) after = v[k].add(after);
                    after = kshfl(after, 31);
                    skip = kneg(after) || kzero(after);
                    if (skip) erun = after;
                }
                if (!skip) {
#pragma unroll
                    for (int k = 0; k < kPer; ++k) {
                        if ((m >> k) & 1u) {
                            run = v[k].add(run);
                            const uint32_t e = R.heavy(r);
                            R.put(e, run, key32_heavy(f, run), pos + k);
                            ++r;
                        }
                    }
                    erun = kshfl(run, 31);
                    hh = __shfl_sync(0xFFFFFFFFu, r, 31);
                }
                if (next_tile) {
                    s = rs.y == kNone ? ntiles : rs.y / (uint32_t)kTile;
                    if (s < ntiles) {
                        rs = split_head(split + s);
                        sa = (uint64_t)s * kTile;
                        send = min(sa + kTile, n);
                        if (rs.z > (uint32_t)kSparse) load_lane(w, vec, sa, send, 0u, y);
                    }
                }
            } else {
                // sparse tiles s .. s + 31 up to the first dense one, while their heavies fit a batch
                const uint32_t t = s + lane;
                uint4 rt = make_uint4(0, 0, 0, 0);
                bool ok = t < ntiles && t >= s;
                if (ok) rt = split_head(split + t);
                ok = ok && rt.z <= (uint32_t)kSparse;
                uint32_t inc = ok ? rt.z : kRing; // a refused tile ends the run
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                    if (lane >= (uint32_t)d) inc += o;
                }
                const uint32_t took = (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, inc <= kBatch)); // a prefix, not empty
                tot = __shfl_sync(0xFFFFFFFFu, inc, took - 1);
                const uint32_t next = __shfl_sync(0xFFFFFFFFu, rt.y, took - 1);
                __syncwarp();
                if (lane < took) {
                    const uint32_t r0 = hh + inc - rt.z;
                    for (uint32_t q = 0; q < rt.z; ++q) {
                        const uint32_t pos = t * (uint32_t)kTile + slist[(uint64_t)t * kSparse + q];
                        const uint32_t e = R.heavy(r0 + q);
                        R.kp[e] = make_uint2(__ldg(w + pos), pos);
                    }
                }
                __syncwarp();
                for (uint32_t r0 = 0; r0 < tot; r0 += 32) { // words -> keys, 32 at a time
                    const uint32_t e = R.heavy(hh + r0 + lane);
                    const bool in = r0 + lane < tot;
                    const K v = in ? ksub(U.nq(R.kp[e].x), U.Q) : K{0, 0};
                    const K run = kadd(erun, warp_scan_key(v));
                    if (in) R.put(e, run, key32_heavy(f, run), R.kp[e].y);
                    erun = kshfl(run, 31);
                }
                hh += tot;
                s = next == kNone ? ntiles : next / (uint32_t)kTile;
                if (s < ntiles) {
                    rs = split_head(split + s);
                    sa = (uint64_t)s * kTile;
                    send = min(sa + kTile, n);
                    if (rs.z > (uint32_t)kSparse) load_lane(w, vec, sa, send, 0u, y);
                }
            }
            past = !kle(erun, f.dmax) && hh != hj;
            if (s >= ntiles && lane == 0) R.kp[R.heavy(hh)].y = kNone; // no heavy after the last
            __syncwarp();
            continue;
        }
        // Merge the next outputs, up to 63: those that the next 31 lights, D
        // of the one after them and the next 32 heavies decide.
        const uint32_t na = min(31u, lh - li), nb = hh - hj;
        const uint32_t kd = R.kp[R.light(li + lane)].x;
        uint32_t ke = R.kp[R.heavy(hj + lane)].x;
        if (lane >= nb) ke = 0x7FFFFFFFu;
        uint32_t cnt = 0; // heavies before light `lane` among the 32
        if ((int32_t)__shfl_sync(0xFFFFFFFFu, ke, 0) <= (int32_t)__shfl_sync(0xFFFFFFFFu, kd, na)) {
#pragma unroll
            for (uint32_t st = 16; st; st >>= 1) {
                const uint32_t v = __shfl_sync(0xFFFFFFFFu, ke, cnt + (st - 1));
                if ((int32_t)v <= (int32_t)kd) cnt += st;
            }
            if ((int32_t)__shfl_sync(0xFFFFFFFFu, ke, cnt) <= (int32_t)kd) ++cnt;
            if (f.s != 0) {
                const uint32_t last = __shfl_sync(0xFFFFFFFFu, ke, cnt - 1);
                if (__any_sync(0xFFFFFFFFu, last == kd && cnt > 0 && lane <= na)) { // rare: told apart by the exact keys
                    while (cnt > 0 && lane <= na) {
                        const uint32_t eh = R.heavy(hj + cnt - 1), el = R.light(li + lane);
                        if (R.kp[eh].x != kd) break;
                        const uint64_t a = R.low[el], b = R.low[eh];
                        if (kWide ? (int32_t)(R.high[el] - R.high[eh] - (a < b ? 1u : 0u)) >= 0 : (int64_t)(a - b) >= 0) break;
                        --cnt;
                    }
                    __syncwarp();
                }
            }
        }
        // merged position of light `lane`; the outputs end where light na
        // would come, or after the 32nd heavy
        const uint32_t p = lane + cnt;
        uint32_t total = __shfl_sync(0xFFFFFFFFu, p, na);
        if (total == 0) break;
        if (total == na + 32) total = 32 + (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, cnt < 32 && lane < na));
        if (total > 32 && total < 48) total = 32; // a second pass for few outputs does not pay
        const bool now = lane < na && p < total;
        uint32_t lights = __reduce_or_sync(0xFFFFFFFFu, now ? shl32(1u, p) : 0u);
        const uint32_t lights2 = total > 32 ? __reduce_or_sync(0xFFFFFFFFu, now ? shl32(1u, p - 32u) : 0u) : 0u;
        for (;;) { // outputs 0 .. 31, then 32 .. 62
            const bool is_light = (lights >> lane) & 1u;
            const uint32_t a = (uint32_t)__popc(lights & lt), b = lane - a; // lights and heavies before it (of its pass)
            if (lane < total) {
                // light: Q - (D[a + 1] - D[a]), alias heavy b; heavy: Q + E[b] - D[a], alias heavy b + 1
                const uint32_t ea = R.light(li + a), eb = R.heavy(hj + b);
                const uint32_t eo = is_light ? R.light(li + a + 1) : eb, et = is_light ? ea : R.heavy(hj + b + 1);
                const uint32_t hp = R.kp[eb].y, ot = R.kp[et].y;
                const uint32_t me = is_light ? ot : hp;
                uint32_t alias = is_light ? hp : ot;
                const uint64_t dl = R.low[ea], ol = R.low[eo];
                bool wrong;
                uint64_t thr;
                if (!kWide) { // exact modulo 2^64: 0 <= bucket <= Q < 2^64
                    const uint64_t df = ol - dl, flip = is_light ? ~0ull : 0ull;
                    const uint64_t bw = U.Q.lo + (df ^ flip) + (is_light ? 1u : 0u);
                    if (bw == U.Q.lo) alias = me;
                    wrong = bw > U.Q.lo;
                    thr = bw;
                } else {      // modulo 2^96
                    K da, od;
                    da.lo = dl;
                    da.hi = R.high[ea];
                    od.lo = ol;
                    od.hi = R.high[eo];
                    K bw = kadd(U.Q, is_light ? ksub(da, od) : ksub(od, da));
                    bw.hi &= 0xFFFFFFFFu;
                    if (keq(bw, U.Q)) alias = me;
                    wrong = !kle(bw, U.Q);
                    thr = U.thr(bw);
                }
                // heavies before the task's first light belong to the task before
                if (is_light || li + a != 0) {
                    if (alias == kNone || wrong) bad = true; // a part-filled last heavy; D - E >= Q
                    else put_bucket(table, me, thr, alias, n, hdr);
                }
            }
            const uint32_t outs = min(total, 32u), took = (uint32_t)__popc(lights);
            li += took;
            hj += outs - took;
            total -= outs;
            if (total == 0) break;
            lights = lights2;
        }
        __syncwarp(); // entries read before they are replaced
    }
    if (!kzero(ksub(drun, f.dmax))) bad = true;
    // end of the subproblem: the heavy carried on lies in the tile k_split
    // found independently
    if (WRS_CHECK && lane == 0 && hj < hh)
        check_ok(R.kp[R.heavy(hj)].y / (uint32_t)kTile == split_head(split + c_last).x, hdr);
    return bad;
}

// Task (c_first, c_last) of one table for this warp.
template <int F32, int TILE>
__device__ __forceinline__ void sweep_body(const uint32_t *__restrict__ w, uint64_t n, int vec, DevHeader *hdr,
                                           const Split *__restrict__ split, const uint16_t *__restrict__ slist,
                                           uint32_t ntiles, uint4 *__restrict__ table, uint32_t c_first,
                                           uint32_t c_last, bool force_wide = false)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (__shfl_sync(0xFFFFFFFFu, *(volatile const uint32_t *)&hdr->status, 0)) return; // the whole warp or none
    const u128 Q = mk128(hdr->q_lo, hdr->q_hi);
    const uint32_t mode = force_wide ? (uint32_t)kPackQ128 : split_head(split + c_first).w; // the table's
    bool bad;
    if (mode == kPackQ32)
        bad = sweep_task<F32, kPackQ32, TILE>(*reinterpret_cast<WarpRings<kPackQ32> *>(smem_raw), w, n, vec, hdr, split,
                                        slist, ntiles, table, c_first, c_last, Q);
    else if (F32 && mode == kPackQ96)
        bad = sweep_task<F32, kPackQ96, TILE>(*reinterpret_cast<WarpRings<kPackQ96> *>(smem_raw), w, n, vec, hdr, split,
                                        slist, ntiles, table, c_first, c_last, Q);
    else
        bad = sweep_task<F32, kPackQ128, TILE>(*reinterpret_cast<WarpRings<kPackQ128> *>(smem_raw), w, n, vec, hdr,
                                         split, slist, ntiles, table, c_first, c_last, Q);
    if (bad) set_status(hdr, kEInternal);
}

// Block (warp) v packs own tiles [v * group, (v + 1) * group); force_wide runs
// the 128-bit keys even when 96 bits hold them.
template <int F32, int TILE>
__global__ void __launch_bounds__(32, kPackBlocks) k_sweep(const uint32_t *__restrict__ w, uint64_t n, int vec,
                                                              DevHeader *hdr, const Split *__restrict__ split,
                                                              const uint16_t *__restrict__ slist, uint32_t ntiles,
                                                              uint4 *__restrict__ table, uint32_t group, int force_wide)
{
    const uint32_t c_first = blockIdx.x * group;
    sweep_body<F32, TILE>(w, n, vec, hdr, split, slist, ntiles, table, c_first, min(c_first + group, ntiles),
                    force_wide != 0);
}

// The exact sum was asked to fit 64 bits (accumulator mode U64): Q >= 2^64
// fails the build with WRS_EOVERFLOW before the sweep.
__global__ void k_require_u64(DevHeader *hdr)
{
    if (threadIdx.x == 0 && hdr->status == 0 && hdr->q_hi != 0) set_status(hdr, kEOverflow);
}

// ----------------------------------------------------------- k_sample
// A query reads one random 16-B bucket.  The .L2::64B size hint makes the L2
// fetch 64 B per miss instead of 128 B: half the DRAM bytes per sample, a few
// percent faster (random sampling is bound by DRAM accesses, not bytes).
__device__ __forceinline__ uint4 ld_bucket(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L2::64B.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Queries a thread has in flight.  A table beyond the L2 is bound by random
// DRAM reads (48 * 10^9 a second): 8 in flight at 102 registers, two blocks per
// SM (3 10^8 samples of 10^9 buckets 6.28 ms; the code below for small tables
// with 8 in flight at one, two or three blocks 6.34, 6.42, 6.55).  A table in the L2
// is bound by the L1's one line per cycle and the arithmetic: 4 in flight,
// 32-bit indices and no bounds tests in full rounds, so that twice the warps
// fit (10^8 samples of 300,000 buckets 0.48 -> 0.39 ms).
constexpr int kSampleUnroll = 8, kSampleUnrollSmall = 4;
constexpr uint64_t kSampleSmallN = 1ull << 22; // 64 MB of buckets

// Samples first, first + stride, ... (below k) of one table.
__device__ __forceinline__ void sample_body(const uint4 *__restrict__ tab, uint64_t n, uint64_t qp, uint64_t k,
                                            uint32_t key0, uint32_t key1, uint32_t sid0, uint32_t sid1,
                                            uint32_t *__restrict__ out, uint64_t first, uint64_t stride,
                                            const DevHeader *chk = nullptr)
{
    for (uint64_t s = first; s < k; s += kSampleUnroll * stride) {
        uint64_t r[kSampleUnroll], v[kSampleUnroll];
        uint4 b[kSampleUnroll];
#pragma unroll
        for (int j = 0; j < kSampleUnroll; ++j) {
            const uint64_t sj = s + j * stride;
            P4 c;
            c.x0 = (uint32_t)sj; c.x1 = (uint32_t)(sj >> 32); c.x2 = sid0; c.x3 = sid1;
            const P4 o = philox4x32_10(c, key0, key1);
            const uint64_t u = o.x0 | ((uint64_t)o.x1 << 32);
            v[j] = o.x2 | ((uint64_t)o.x3 << 32);
            r[j] = __umul64hi(u, n);
        }
#pragma unroll
        for (int j = 0; j < kSampleUnroll; ++j)
            if (s + j * stride < k) b[j] = ld_bucket(tab + r[j]);
#pragma unroll
        for (int j = 0; j < kSampleUnroll; ++j) {
            const uint64_t sj = s + j * stride;
            if (sj < k) {
                const uint64_t thr = b[j].x | ((uint64_t)b[j].y << 32);
                if (WRS_CHECK && chk) check_ok(b[j].z < n, const_cast<DevHeader *>(chk));
                const uint32_t pick = (__umul64hi(v[j], qp) < thr) ? (uint32_t)r[j] : b[j].z;
                __stcs(out + sj, pick);
            }
        }
    }
}

// The same from a table that fits the L2.
__device__ __forceinline__ void sample_body_small(const uint4 *__restrict__ tab, uint64_t n, uint64_t qp, uint64_t k,
                                            uint32_t key0, uint32_t key1, uint32_t sid0, uint32_t sid1,
                                            uint32_t *__restrict__ out, uint64_t first, uint64_t stride,
                                            const DevHeader *chk = nullptr)
{
    const uint32_t n32 = (uint32_t)n; // n < 2^32
    for (uint64_t s = first; s < k; s += kSampleUnrollSmall * stride) {
        const bool all = s + (kSampleUnrollSmall - 1) * stride < k;
        uint32_t r[kSampleUnrollSmall];
        uint64_t v[kSampleUnrollSmall];
        uint4 b[kSampleUnrollSmall];
#pragma unroll
        for (int j = 0; j < kSampleUnrollSmall; ++j) {
            const uint64_t sj = s + j * stride;
            P4 c;
            c.x0 = (uint32_t)sj; c.x1 = (uint32_t)(sj >> 32); c.x2 = sid0; c.x3 = sid1;
            const P4 o = philox4x32_10(c, key0, key1);
            v[j] = o.x2 | ((uint64_t)o.x3 << 32);
            r[j] = (uint32_t)(((uint64_t)o.x1 * n32 + __umulhi(o.x0, n32)) >> 32); // floor(u n / 2^64)
        }
#pragma unroll
        for (int j = 0; j < kSampleUnrollSmall; ++j)
            if (all || s + j * stride < k) b[j] = ld_bucket(tab + r[j]);
#pragma unroll
        for (int j = 0; j < kSampleUnrollSmall; ++j) {
            const uint64_t sj = s + j * stride;
            if (all || sj < k) {
                const uint64_t thr = b[j].x | ((uint64_t)b[j].y << 32);
                if (WRS_CHECK && chk) check_ok(b[j].z < n, const_cast<DevHeader *>(chk));
                const uint32_t pick = (__umul64hi(v[j], qp) < thr) ? r[j] : b[j].z;
                __stcs(out + sj, pick);
            }
        }
    }
}

// Samples [s0, k) of one table.
__global__ void __launch_bounds__(256) k_sample(const uint4 *__restrict__ tab, uint64_t n,
                                                const DevHeader *__restrict__ hdr, uint64_t s0, uint64_t k,
                                                uint32_t key0, uint32_t key1, uint32_t sid0, uint32_t sid1,
                                                uint32_t *__restrict__ out)
{
    if (hdr->status) return;
    sample_body(tab, n, hdr->qp, k, key0, key1, sid0, sid1, out,
                s0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, (uint64_t)gridDim.x * blockDim.x, hdr);
}

__global__ void __launch_bounds__(256, 4) k_sample_small(const uint4 *__restrict__ tab, uint64_t n,
                                                         const DevHeader *__restrict__ hdr, uint64_t s0, uint64_t k,
                                                         uint32_t key0, uint32_t key1, uint32_t sid0, uint32_t sid1,
                                                         uint32_t *__restrict__ out)
{
    if (hdr->status) return;
    sample_body_small(tab, n, hdr->qp, k, key0, key1, sid0, sid1, out,
                      s0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, (uint64_t)gridDim.x * blockDim.x, hdr);
}

} // namespace wrs
