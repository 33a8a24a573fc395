// The sweep on the host: write_header, split_body and sweep_body of
// wrs_kernels.cuh compiled by the host compiler, the 32 lanes of a warp run as
// coroutines that meet at every warp-wide operation.  The headers are built with
// WRS_CHECK=1, so put_bucket refuses a store outside the table and counts it.
// Built and driven by test_sweep_host.py.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>
#include <ucontext.h>

// ------------------------------------------------ what the headers take from CUDA
#define __device__
#define __host__
#define __global__ static
#define __shared__
#define __forceinline__ inline
#define __noinline__ __attribute__((unused)) static
#define __restrict__
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))

struct uint2 { uint32_t x, y; };
struct uint4 { uint32_t x, y, z, w; };
static inline uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
static inline uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }

constexpr int kLanes = 32;
static int g_lane;
static struct { struct { operator uint32_t() const { return (uint32_t)g_lane; } } x; } threadIdx;
static struct { uint32_t x; } blockIdx, gridDim, blockDim;

using std::max;
using std::min;
template <typename T> static inline T __ldg(const T *p) { return *p; }
template <typename T> static inline T __ldcg(const T *p) { return *p; }
template <typename T> static inline void __stcs(T *p, T v) { *p = v; }
static inline int __popc(uint32_t v) { return __builtin_popcount(v); }
static inline int __clz(int v) { return v ? __builtin_clz((uint32_t)v) : 32; }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
static inline int __ffsll(long long v) { return __builtin_ffsll(v); }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s)
{
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> (s & 31));
}
template <typename T> static inline T atomicAdd(T *p, T v) { const T o = *p; *p = o + v; return o; }
static inline uint32_t atomicCAS(uint32_t *p, uint32_t a, uint32_t b) { const uint32_t o = *p; if (o == a) *p = b; return o; }
static inline void __threadfence() {}
static inline void __nanosleep(uint32_t) {}

// Lanes as coroutines: a lane that reaches a warp-wide operation yields until
// every lane has.
static ucontext_t g_main, g_ctx[kLanes];
static std::vector<char> g_stack[kLanes];
static bool g_done[kLanes];
static uint32_t g_gen[kLanes];
static uint64_t g_slot[2][kLanes];
static std::function<void()> g_fn;
static bool g_stuck; // some lanes returned while others waited for them

static void lane_main()
{
    g_fn();
    g_done[g_lane] = true;
    swapcontext(&g_ctx[g_lane], &g_main);
}
static const uint64_t *meet(uint64_t v)
{
    const int me = g_lane;
    const uint32_t par = g_gen[me] & 1, gen = ++g_gen[me];
    g_slot[par][me] = v;
    for (;;) {
        bool all = true;
        for (int i = 0; i < kLanes; ++i) all = all && g_gen[i] >= gen;
        if (all) return g_slot[par];
        swapcontext(&g_ctx[me], &g_main);
    }
}
static void run_warp(std::function<void()> f)
{
    g_fn = std::move(f);
    for (int i = 0; i < kLanes; ++i) {
        g_stack[i].resize(1 << 17);
        getcontext(&g_ctx[i]);
        g_ctx[i].uc_stack.ss_sp = g_stack[i].data();
        g_ctx[i].uc_stack.ss_size = g_stack[i].size();
        g_ctx[i].uc_link = &g_main;
        makecontext(&g_ctx[i], lane_main, 0);
        g_done[i] = false;
        g_gen[i] = 0;
    }
    for (bool any = true; any;) {
        any = false;
        bool moved = false;
        for (int i = 0; i < kLanes; ++i) {
            if (g_done[i]) continue;
            any = true;
            g_lane = i;
            const uint32_t gen = g_gen[i];
            swapcontext(&g_main, &g_ctx[i]);
            moved = moved || g_done[i] || g_gen[i] != gen;
        }
        if (any && !moved) { g_stuck = true; return; }
    }
}

template <typename T> static inline T lane_value(T v, int src)
{
    uint64_t w = 0;
    memcpy(&w, &v, sizeof(T));
    w = meet(w)[src & 31];
    memcpy(&v, &w, sizeof(T));
    return v;
}
template <typename T> static inline T __shfl_sync(uint32_t, T v, int src) { return lane_value(v, src); }
template <typename T> static inline T __shfl_up_sync(uint32_t, T v, int d)
{
    return lane_value(v, g_lane >= d ? g_lane - d : g_lane);
}
template <typename T> static inline T __shfl_down_sync(uint32_t, T v, int d)
{
    return lane_value(v, g_lane + d < kLanes ? g_lane + d : g_lane);
}
template <typename T> static inline T __shfl_xor_sync(uint32_t, T v, int m) { return lane_value(v, g_lane ^ m); }
template <typename F> static inline uint32_t lane_fold(uint32_t v, F f)
{
    const uint64_t *s = meet(v);
    uint32_t r = (uint32_t)s[0];
    for (int i = 1; i < kLanes; ++i) r = f(r, (uint32_t)s[i]);
    return r;
}
static inline uint32_t __reduce_or_sync(uint32_t, uint32_t v) { return lane_fold(v, [](uint32_t a, uint32_t b) { return a | b; }); }
static inline uint32_t __reduce_add_sync(uint32_t, uint32_t v) { return lane_fold(v, [](uint32_t a, uint32_t b) { return a + b; }); }
static inline uint32_t __reduce_min_sync(uint32_t, uint32_t v) { return lane_fold(v, [](uint32_t a, uint32_t b) { return min(a, b); }); }
static inline uint32_t __reduce_max_sync(uint32_t, uint32_t v) { return lane_fold(v, [](uint32_t a, uint32_t b) { return max(a, b); }); }
static inline uint32_t __ballot_sync(uint32_t, bool p) { return __reduce_or_sync(0, (uint32_t)p << g_lane); }
static inline bool __any_sync(uint32_t, bool p) { return __ballot_sync(0, p) != 0; }
static inline void __syncwarp() { meet(0); }
static inline void __syncthreads() { abort(); } // block-wide code is not run here

// The PTX statements (asm volatile("...")) sit in functions that are not run
// here; the host compiler need not know their constraints.
#define volatile(...) ("")

#include "wrs_kernels.cuh"

namespace wrs {
alignas(16) unsigned char smem_raw[kPackSmemBytes]; // a block's shared memory
}

namespace {

using namespace wrs;

// Tile sums by plain loops, then the split records and every task of `group`
// tiles, one warp after another.
template <int F32, int TILE>
void build(const uint32_t *w, uint64_t n, int vec, uint32_t group, bool wide, DevHeader *hdr, uint4 *table)
{
    Acc a;
    a.base = F32 ? INT_MAX : 0;
    a.acc = 0;
    a.flags = 0;
    a.mx = 0;
    uint64_t a64 = 0;
    for (uint64_t i = 0; i < n; ++i) {
        acc_take<F32>(a, a64, w[i]);
        acc_fold(a, a64);
    }
    Partial part;
    if (write_header(a, n, F32, hdr, part.mode)) return;
    const uint32_t ntiles = (uint32_t)((n + TILE - 1) / TILE);
    std::vector<TileSum> incl(ntiles);
    std::vector<Split> split(ntiles + 1);
    std::vector<uint16_t> slist((size_t)ntiles * kSparseOf(TILE), 0xFFFF);
    u128 L = 0, H = 0;
    uint32_t cl = 0;
    for (uint32_t t = 0; t < ntiles; ++t) {
        TileSum &s = incl[t];
        s.nheavy = 0;
        s.first_heavy = kNone;
        s.pad = 0;
        for (uint64_t i = (uint64_t)t * TILE; i < min((uint64_t)(t + 1) * TILE, n); ++i) {
            const u128 q = q_of(w[i], F32, hdr->beta);
            if (w[i] <= hdr->light_max) { L += q; ++cl; continue; }
            H += q;
            const uint32_t off = (uint32_t)(i - (uint64_t)t * TILE);
            if (s.nheavy == 0) s.first_heavy = off;
            if (s.nheavy < (uint32_t)kSparseOf(TILE)) slist[(size_t)t * kSparseOf(TILE) + s.nheavy] = (uint16_t)off;
            ++s.nheavy;
        }
        s.cl = cl;
        s.l_lo = lo64(L); s.l_hi = hi64(L); s.h_lo = lo64(H); s.h_hi = hi64(H);
    }
    for (uint32_t c = 0; c <= ntiles; ++c) split_body<TILE>(incl.data(), ntiles, n, hdr, &part, split.data(), c);
    for (uint32_t c = 0; c < ntiles; c += group) {
        memset(smem_raw, 0xA5, sizeof(smem_raw));
        run_warp([&] {
            sweep_body<F32, TILE>(w, n, vec, hdr, split.data(), slist.data(), ntiles, table, c, min(c + group, ntiles),
                                  wide);
        });
    }
}

} // namespace

// Builds the table of w[0 .. n) into table[0 .. n) (zeroed by the caller, who
// sees how often each bucket was stored in its fourth word) with tiles of
// `tile` weights, tasks of `group` of them; `wide`: 128-bit keys.  status and
// failed: the header's status and count of failed checks.  Returns 0, or 1 when
// the lanes of a warp lost each other.
extern "C" int sweep_host(const uint32_t *w, uint64_t n, int f32, uint32_t tile, uint32_t group, int wide,
                           uint32_t *table, uint32_t *status, uint64_t *failed)
{
    DevHeader hdr;
    memset(&hdr, 0, sizeof(hdr));
    g_stuck = false;
    const int vec = (reinterpret_cast<uintptr_t>(w) % 16) == 0;
    auto *f = f32 ? (tile == (uint32_t)kTile ? build<1, kTile> : build<1, kFineTile>)
                  : (tile == (uint32_t)kTile ? build<0, kTile> : build<0, kFineTile>);
    f(w, n, vec, group, wide != 0, &hdr, reinterpret_cast<uint4 *>(table));
    *status = hdr.status;
    *failed = hdr.pad[0];
    return g_stuck;
}

// Device bytes of a table of capacity cap: what wrs_table_create allocates.
extern "C" uint64_t table_bytes_host(uint64_t cap) { return bucket_area(cap) + layout_for(cap).total; }
