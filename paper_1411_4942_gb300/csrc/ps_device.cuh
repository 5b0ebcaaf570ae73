// ps_device.cuh -- device-side building blocks of the path-sampling library:
// the graph descriptor, Philox4x32-10, Lemire bounded draws, list searches,
// the adjacency test and a decoupled look-back scan.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ps {

typedef unsigned long long u64;

// ---------------------------------------------------------------- layout

// One edge (u < v) of the relabelled graph, 32 bytes = one DRAM sector:
// everything a sample needs after choosing the edge.  iu / jv are the
// positions of v in N(u) and of u in N(v); ou / ov the row offsets.
struct __align__(32) EdgeRec {
    int32_t u, v, du, dv, iu, jv, ou, ov;
};

// Device view of one loaded graph (passed by value to kernels and stored in
// the batched launch's descriptor table).
struct GraphDev {
    const int64_t *off;      // [n + 1] canonical row offsets
    const int32_t *col;      // [nnz]   canonical adjacency, rows ascending
    const EdgeRec *rec;      // [m]
    const uint64_t *ptau;    // [m] inclusive prefix of tau
    const uint64_t *plam;    // [m] inclusive prefix of lambda
    const int32_t *gtau;     // [Bt + 1] guide: first edge of each r >> tau_shift bucket
    const int32_t *glam;     // [Bl + 1]
    const uint32_t *hub;     // [hubs][hub_words] adjacency bitmaps of the top labels
    uint64_t filt_off;       // the edge filter starts this many words after `hub`
    uint32_t filt_words;     // words of the edge filter
    const int32_t *vtab;     // per-vertex hash tables: slots [2 off(x), 2 off(x+1)), or null
    uint64_t W, Lambda;
    int64_t n, m;
    int32_t hub_start;       // labels >= hub_start have a bitmap row
    int32_t hub_words;
    int32_t tau_shift, lam_shift;
    int32_t adj_mode;        // kAdjHash, kAdjSearch or kAdjVtab
    int32_t hub_bit_base;    // hub rows hold the bits of labels >= hub_bit_base (a multiple of 32)
};

// Adjacency test variants (chosen by the tuning; results are identical).
enum { kAdjHash = 1, kAdjSearch = 2, kAdjVtab = 3 };

// status block (uint64 words at the start of the workspace)
enum {
    ST_FLAGS = 0,
    ST_DMAX = 1,
    ST_M_UPPER = 2,
    ST_W_LO = 3, ST_W_HI = 4,
    ST_L_LO = 5, ST_L_HI = 6,
    ST_N1_LO = 7, ST_N1_HI = 8,
    ST_HUBS = 9,
    ST_TIER = 10,      // 5 words: row boundaries of the sort tiers
    ST_LONG = 15,      // first row longer than kLongRow (its arcs are walked by a block)
    ST_COUNTER = 16,   // tile counter of the allocation-free scan
    ST_WORDS = 64
};

enum : u64 {
    F_ARG = 1ull,
    F_NOT_SIMPLE = 2ull,
    F_ASYM = 4ull,
    F_OVERFLOW = 8ull,
    F_TIMEOUT = 16ull
};

__device__ __forceinline__ void raise_flag(u64 *status, u64 f) {
    atomicOr(reinterpret_cast<unsigned long long *>(status + ST_FLAGS),
             static_cast<unsigned long long>(f));
}

// Bound on every device spin-wait (iterations with nanosleep back-off).
constexpr uint32_t kSpinLimit = 1u << 24;

// ------------------------------------------------------------------ loads

// Read-only gathers of data written by earlier kernels.  PS_LOAD_MODE picks
// the cache path: 0 = the non-coherent path through L1 (__ldg); 1 = L2 only
// (ld.global.cg); 2 = non-coherent without L1 allocation.
#ifndef PS_LOAD_MODE
#define PS_LOAD_MODE 0
#endif
#if PS_LOAD_MODE == 0
#define PS_LD "ld.global.nc"
#elif PS_LOAD_MODE == 1
#define PS_LD "ld.global.cg"
#elif PS_LOAD_MODE == 2
#define PS_LD "ld.global.nc.L1::no_allocate"
#endif

__device__ __forceinline__ int32_t ldg_i32(const int32_t *p) {
#if PS_LOAD_MODE == 0
    return __ldg(p);
#else
    int32_t v;
    asm(PS_LD ".s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
#endif
}
__device__ __forceinline__ int64_t ldg_i64(const int64_t *p) {
#if PS_LOAD_MODE == 0
    return static_cast<int64_t>(__ldg(reinterpret_cast<const long long *>(p)));
#else
    int64_t v;
    asm(PS_LD ".s64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
#endif
}
__device__ __forceinline__ uint64_t ldg_u64(const uint64_t *p) {
#if PS_LOAD_MODE == 0
    return static_cast<uint64_t>(__ldg(reinterpret_cast<const unsigned long long *>(p)));
#else
    uint64_t v;
    asm(PS_LD ".u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
#endif
}
// A gather that nothing nearby reads again: it takes no line of L1.
__device__ __forceinline__ int32_t ldg_i32_once(const int32_t *p) {
#if PS_LOAD_MODE == 1
    return ldg_i32(p);
#else
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
#endif
}
// Gathers of the skewed "hot" structures (guide entries, prefix probes).
// (Evict-last L2 hints on these and on the hub rows' adjacency lists were
// measured: no gain.)
__device__ __forceinline__ int32_t ldg_i32_hot(const int32_t *p) { return ldg_i32(p); }
__device__ __forceinline__ uint64_t ldg_u64_hot(const uint64_t *p) { return ldg_u64(p); }

__device__ __forceinline__ EdgeRec ldg_rec(const EdgeRec *p) {
    EdgeRec e;
    // one 256-bit load (records are 32-byte aligned): two 128-bit loads cost a
    // second pass through L1's tags
    asm(PS_LD ".v8.s32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(e.u), "=r"(e.v), "=r"(e.du), "=r"(e.dv), "=r"(e.iu), "=r"(e.jv), "=r"(e.ou), "=r"(e.ov)
        : "l"(p));
    return e;
}

// ----------------------------------------------------------------- Philox

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of the
// two-multiplier S-box, key advanced by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int i = 0; i < 10; i++) {
        if (i) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// Random block t of sample `id` for sampler `stream` (0: 3-path, 1: centred):
// key (seed lo, seed hi), counter (id lo, id hi, t, stream).
__device__ __forceinline__ uint4 sample_block(uint64_t seed, uint64_t id, uint32_t t,
                                              uint32_t stream) {
    return philox4x32_10(make_uint4(static_cast<uint32_t>(id), static_cast<uint32_t>(id >> 32), t,
                                    stream),
                         make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32)));
}

// Lemire's multiply-and-reject (ACM TOMACS 2019): one attempt.  The
// threshold (2^64 mod s) is only computed when the low half is below s.
__device__ __forceinline__ bool lemire64(uint64_t x, uint64_t s, uint64_t &out) {
    const uint64_t lo = x * s;
    if (lo < s) {
        const uint64_t thr = (0ull - s) % s;
        if (lo < thr) return false;
    }
    out = __umul64hi(x, s);
    return true;
}

__device__ __forceinline__ bool lemire32(uint32_t x, uint32_t s, uint32_t &out) {
    const uint64_t p = static_cast<uint64_t>(x) * s;
    const uint32_t lo = static_cast<uint32_t>(p);
    if (lo < s) {
        const uint32_t thr = (0u - s) % s;
        if (lo < thr) return false;
    }
    out = static_cast<uint32_t>(p >> 32);
    return true;
}

// Rejected first attempts walk blocks t = 1, 2, ... on the same word slot.
static __device__ __noinline__ uint64_t draw_r_retry(uint64_t seed, uint64_t id, uint32_t stream,
                                              uint64_t s) {
    uint64_t r = 0;
    for (uint32_t t = 1; t < 4096u; t++) {
        const uint4 w = sample_block(seed, id, t, stream);
        if (lemire64((static_cast<uint64_t>(w.y) << 32) | w.x, s, r)) return r;
    }
    return 0;  // unreachable for any s (probability < 2^-4000)
}

static __device__ __noinline__ uint32_t draw_small_retry(uint64_t seed, uint64_t id, uint32_t stream,
                                                  int slot, uint32_t s) {
    uint32_t r = 0;
    for (uint32_t t = 1; t < 4096u; t++) {
        const uint4 w = sample_block(seed, id, t, stream);
        if (lemire32(slot == 2 ? w.z : w.w, s, r)) return r;
    }
    return 0;
}

// --------------------------------------------------------------- searches

// First j in [lo, hi] with P[j] > r, given P[hi] > r.
__device__ __forceinline__ int64_t upper_bound_in(const uint64_t *P, int64_t lo, int64_t hi,
                                                  uint64_t r) {
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (ldg_u64_hot(P + mid) > r) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// Edge of r: guide bucket r >> shift gives a range [G[b], G[b + 1]] that
// holds the answer; search it exactly.
__device__ __forceinline__ int64_t find_edge(const uint64_t *P, const int32_t *G, int shift,
                                             uint64_t r) {
    const uint64_t b = r >> shift;
    const int64_t lo = ldg_i32_hot(G + b);
    const int64_t hi = ldg_i32_hot(G + b + 1);
    if (lo == hi) return lo;
    return upper_bound_in(P, lo, hi, r);
}

// Is `key` in the sorted list col[o, o + d)?
__device__ __forceinline__ bool in_sorted(const int32_t *col, int64_t o, int64_t d, int32_t key) {
    int64_t lo = o, hi = o + d;  // answer position in [lo, hi)
    while (hi - lo > 8) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (ldg_i32(col + mid) <= key) lo = mid;
        else hi = mid;
    }
    bool hit = false;
#pragma unroll
    for (int i = 0; i < 8; i++)
        if (lo + i < hi) hit |= (ldg_i32(col + lo + i) == key);
    return hit;
}

// Adjacency test of Alg. 2 / Alg. 4 ("determine the induced subgraph").
// The smaller label has the smaller (or equal) degree, so its list is
// searched; pairs of hubs read one bit of the hub bitmap.
__device__ __forceinline__ bool adjacent(const GraphDev &g, int32_t x, int32_t y) {
    if (x == y) return false;
    const int32_t a = min(x, y), b = max(x, y);
    if (a >= g.hub_start) {  // then b > a >= hub_bit_base
        const uint32_t *row = g.hub + static_cast<int64_t>(a - g.hub_start) * g.hub_words;
        return (__ldg(row + ((b - g.hub_bit_base) >> 5)) >> (b & 31)) & 1u;
    }
    const int64_t o = ldg_i64(g.off + a);
    const int64_t e = ldg_i64(g.off + a + 1);
    return in_sorted(g.col, o, e - o, b);
}

// Same when the row of a (the smaller label) is already known.
__device__ __forceinline__ bool adjacent_known(const GraphDev &g, int32_t a, int64_t oa,
                                               int64_t da, int32_t b) {
    if (a >= g.hub_start) {  // then b > a >= hub_bit_base
        const uint32_t *row = g.hub + static_cast<int64_t>(a - g.hub_start) * g.hub_words;
        return (__ldg(row + ((b - g.hub_bit_base) >> 5)) >> (b & 31)) & 1u;
    }
    return in_sorted(g.col, oa, da, b);
}

// ------------------------------------------------------------- edge filter

// The O(1) adjacency test of Theorem 3.5, in one 4-byte read for nearly every
// pair.  Hub rows (bitmaps of the top-degree labels) answer a pair whose
// larger label is a hub and whose smaller label lies in the rows' span: the
// edges are drawn in proportion to tau, so most pairs name a hub.  The other
// pairs are almost never edges (99.8% of those asked on R-MAT 20 and on the
// 3M-vertex graph are not), so they go to a filter: every edge that no hub
// row holds sets kFilterBits bits of one 32-bit word, and a pair with one of its bits unset
// is not an edge.  A pair with all bits set (an edge, or a false positive)
// is looked up in the sorted row of its smaller label, so every answer is
// exact.  The filter replaces a hash set of the edges (8-byte keys in
// 32-byte buckets, 18 bytes written per edge at load, a 32-byte sector and
// eight registers per test, a second probe in about every tenth test).
constexpr int kFilterBits = 3;

__device__ __forceinline__ uint64_t edge_hash(int32_t a, int32_t c) {
    uint64_t h = (static_cast<uint64_t>(static_cast<uint32_t>(a)) << 32) | static_cast<uint32_t>(c);
    h *= 0x9E3779B97F4A7C15ull;
    h ^= h >> 32;
    return h * 0xD6E8FEB86659FD93ull;
}

// Word and bits of the pair a < c: the word from the hash's high half, the
// bit numbers from the upper bits of its low half.
__device__ __forceinline__ uint32_t filter_word(uint64_t h, uint32_t words) {
    return __umulhi(static_cast<uint32_t>(h >> 32), words);
}
__device__ __forceinline__ uint32_t filter_mask(uint64_t h) {
    const uint32_t s = static_cast<uint32_t>(h) >> (32 - 5 * kFilterBits);
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < kFilterBits; i++) m |= 1u << ((s >> (5 * i)) & 31);
    return m;
}

// Does the pair a < c have a hub-row bit?
__device__ __forceinline__ bool in_hub_rows(const GraphDev &g, int32_t a, int32_t c) {
    return c >= g.hub_start && a >= g.hub_bit_base;
}

// Where the larger label of a pair can be looked up without reading offsets
// first: the row of the smaller one (d < 0: not known).
struct PairRow {
    int32_t o, d;
};

// Is c in the sorted row col[o, o + d)?  Cut to a quarter at every step, three
// reads side by side; the last kRowLeaf entries in whole 16-byte blocks (the
// columns start and end on such in the workspace).
constexpr int kRowBlocks = 3;
constexpr int kRowLeaf = 4 * kRowBlocks - 3;
__device__ __forceinline__ bool row_contains(const int32_t *col, int32_t o, int32_t d, int32_t c) {
    while (d > kRowLeaf) {
        const int32_t step = d >> 2;  // 3 step < d
        const int32_t v1 = ldg_i32(col + o + step), v2 = ldg_i32(col + o + 2 * step), v3 = ldg_i32(col + o + 3 * step);
        const int32_t skip = (v1 <= c ? step : 0) + (v2 <= c ? step : 0) + (v3 <= c ? step : 0);
        o += skip;
        d = skip == 3 * step ? d - skip : step;
    }
    bool in = false;
    const int32_t end = o + d;
#pragma unroll
    for (int j = 0; j < kRowBlocks; j++) {
        const int32_t at = (o & ~3) + 4 * j;
        const int4 v = at < end ? __ldg(reinterpret_cast<const int4 *>(col + at)) : make_int4(-1, -1, -1, -1);
        in |= (v.x == c && at >= o) || (v.y == c && at + 1 >= o && at + 1 < end) ||
              (v.z == c && at + 2 >= o && at + 2 < end) || (v.w == c && at + 3 < end);
    }
    return in;
}

// N independent tests (x != y for each; row[i]: the smaller label's row, if
// known), every pair's word -- of its hub row or of the filter, chosen without
// a branch -- in flight together; the filter hits are then confirmed one by
// one at a single call site (three separate second probes made nearly every
// warp take all three).  Few pairs hit on R-MAT and Chung-Lu graphs, many on
// clustered ones, where the search of a row is what a test costs: with known
// rows, quarters and blocks against halves and single reads, 2^22 centred
// samples of a ring lattice of 2M edges (transitivity 0.7) took 288 -> 239 us,
// of a geometric graph of 20M edges 589 -> 567 us, and R-MAT and Chung-Lu graphs
// the same within 1% (a hash set of the edges: 244 and 565 us).  Two or three
// hits side by side gained 2% there and cost 13% on the others.
template <int N>
__device__ __forceinline__ void pair_tests(const GraphDev &g, const int32_t (&x)[N], const int32_t (&y)[N],
                                           const PairRow (&row)[N], bool (&r)[N]) {
    uint32_t word[N], mask[N];
    uint32_t pend = 0;
#pragma unroll
    for (int i = 0; i < N; i++) {
        const int32_t a = min(x[i], y[i]), c = max(x[i], y[i]);
        const bool hub = in_hub_rows(g, a, c);
        const uint64_t h = edge_hash(a, c);
        const uint64_t hw = static_cast<uint64_t>(static_cast<uint32_t>(c - g.hub_start)) * static_cast<uint32_t>(g.hub_words) +
                            static_cast<uint32_t>((a - g.hub_bit_base) >> 5);
        const uint64_t fw = g.filt_off + filter_word(h, g.filt_words);
        mask[i] = hub ? 1u << (a & 31) : filter_mask(h);
        word[i] = __ldg(g.hub + (hub ? hw : fw));
        pend |= hub ? 0u : 1u << i;
    }
#pragma unroll
    for (int i = 0; i < N; i++) {
        r[i] = (word[i] & mask[i]) == mask[i];
        pend &= r[i] ? ~0u : ~(1u << i);
    }
    while (pend) {
        const int k = __ffs(pend) - 1;
        pend &= pend - 1;
        int32_t p = x[0], q = y[0];
        PairRow w = row[0];
#pragma unroll
        for (int i = 1; i < N; i++) {
            p = k == i ? x[i] : p;
            q = k == i ? y[i] : q;
            w.o = k == i ? row[i].o : w.o;
            w.d = k == i ? row[i].d : w.d;
        }
        if (w.d < 0) {
            const int32_t a = min(p, q);
            w.o = static_cast<int32_t>(ldg_i64(g.off + a));  // below 2^31, as nnz
            w.d = static_cast<int32_t>(ldg_i64(g.off + a + 1)) - w.o;
        }
        const bool in = row_contains(g.col, w.o, w.d, max(p, q));
#pragma unroll
        for (int i = 0; i < N; i++) r[i] = r[i] && (k != i || in);
    }
}

__device__ __forceinline__ bool pair_test(const GraphDev &g, int32_t x, int32_t y) {
    if (x == y) return false;
    const int32_t xs[1] = {x}, ys[1] = {y};
    const PairRow none[1] = {{0, -1}};
    bool r[1];
    pair_tests<1>(g, xs, ys, none, r);
    return r[0];
}

// ------------------------------------------------ per-vertex hash tables

// Each adjacency list in its own open-addressing table (Theorem 3.5 assumes
// hash-table adjacency lists): the table of vertex x is the 2 d_x int32
// slots starting at 2 off(x), holding the neighbours of x (empty = -1),
// linear probing with wrap-around inside the table.  The slot of y is
// (mix(y) * 2 d_x) >> 32.  Lookups go to the table of the endpoint that is a
// sampled edge's endpoint or else the larger label, so they concentrate on
// the tables of high-degree vertices, which stay in L2.
constexpr int32_t kEmptyLabel = -1;

__device__ __forceinline__ uint32_t label_mix(int32_t y) {
    uint32_t h = static_cast<uint32_t>(y) * 0x9E3779B1u;
    h ^= h >> 15;
    h *= 0x85EBCA77u;
    h ^= h >> 13;
    return h;
}

__device__ __forceinline__ uint64_t vtab_start(int32_t y, uint64_t size) {
    return (static_cast<uint64_t>(label_mix(y)) * size) >> 32;
}

static __device__ __noinline__ bool vtab_probe_on(const int32_t *t, uint64_t size, int32_t y, uint64_t s) {
    for (uint64_t i = 1; i < size; i++) {
        s = (s + 1 == size) ? 0 : s + 1;
        const int32_t x = __ldg(t + s);
        if (x == y) return true;
        if (x == kEmptyLabel) return false;
    }
    return false;
}

// Is y a neighbour of the vertex whose row is [off, off + d)?
struct VtabQuery {
    const int32_t *t;
    uint64_t size, s;
    int32_t y;
    __device__ __forceinline__ void start(const int32_t *vtab, int64_t off, int64_t d, int32_t key) {
        t = vtab + 2 * off;
        size = static_cast<uint64_t>(2 * d);
        y = key;
        s = size ? vtab_start(key, size) : 0;
    }
    __device__ __forceinline__ int32_t first() const { return size ? __ldg(t + s) : kEmptyLabel; }
    __device__ __forceinline__ bool resolve(int32_t x) const {
        if (x == y) return true;
        if (x == kEmptyLabel) return false;
        return vtab_probe_on(t, size, y, s);
    }
};

}  // namespace ps
