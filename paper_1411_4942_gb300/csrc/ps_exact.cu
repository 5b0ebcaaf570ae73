// ps_exact.cu -- ps_count_exact: exact 4-vertex counts by enumeration, the
// ground truth that the sampled estimates are checked against where brute
// force is out of reach.  The paper gets its exact counts from separate
// enumeration code (Section 6); here they are the non-induced counts N_1..N_6
// of Eq. (1), turned into the induced counts C_1..C_6 by inverting Eq. (1):
//
//   N_1 = sum_v C(d_v, 3)            3-stars (already a total of the prefix step)
//   N_2 = W - 3 T                    W counts every 3-path once, every triangle 3 times (Section 3)
//   N_3 = sum_triangles (d_a + d_b + d_c - 6)        a triangle plus an edge at one corner
//   N_4 = 4-cycles
//   N_5 = sum_e C(t_e, 2)            two triangles sharing the chord e
//   N_6 = 4-cliques
//
// On the canonical graph (labels in degree order, rows ascending), with U(a)
// the neighbours of a above it (at most sqrt(2m) of them):
//
// Triangles and 4-cliques are found at their lowest vertex a, whose U(a)
// becomes a bit matrix in shared memory: bit (p, q), p < q, says that the
// p-th and the q-th of U(a) are adjacent.  A set bit is a triangle (found by
// walking U(b) for every b in U(a) and looking each entry up among U(a)), and
// the common bits of rows p and q count the 4-cliques over that triangle.
// T, N_3 and N_5 follow from the triangles per edge.
//
// 4-cycles are counted at the vertex c opposite their highest vertex a: the
// wedges c - b - a with a above both give cnt[a] common neighbours, and
// C(cnt[a], 2) cycles.  From c the work is even (the largest share of one
// vertex on R-MAT 20 is 0.01%) and nearly all its ends a are hub labels
// (99.0% are among the top 16384), so the counters sit in shared memory.
#include "ps_internal.h"

namespace ps {

namespace {

// Scratch words of the counters.
enum : int {
    XA_T3 = 0,       // sum of t_e = 3 T; 128-bit pairs, as all sums
    XA_N3X2 = 2,     // 2 N_3
    XA_N4 = 4,
    XA_N5 = 6,
    XA_N6 = 8,
    XA_TIERS = 10,   // lengths of the vertex lists, one word per tier
    XA_HEAVY = 15,   // length of the 4-cycle pass's list
    XA_WORDS = 16,
};

// Vertices by |U(a)|: a warp, a block of 256, 256 or 1024 threads each, and
// those whose matrix does not fit shared memory.
constexpr int kTiers = 5;
constexpr int kTierK0 = 64, kTierK1 = 256, kTierK2 = 512, kTierK3 = 1024;

constexpr int kCliqueCap = 1024;  // common upper neighbours kept per warp in shared memory (last tier)

template <int ADJ>
__device__ __forceinline__ bool has_edge(const GraphDev &g, int32_t x, int32_t y) {
    if (ADJ == kAdjHash) return pair_test(g, x, y);
    if (ADJ == kAdjVtab) {
        if (x == y) return false;
        const int32_t h = max(x, y);
        const int64_t o = ldg_i64(g.off + h);
        VtabQuery q;
        q.start(g.vtab, o, ldg_i64(g.off + h + 1) - o, min(x, y));
        return q.resolve(q.first());
    }
    return adjacent(g, x, y);
}

// First position p in col[lo, hi) with col[p] >= key.
__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *col, int64_t lo, int64_t hi, int32_t key) {
    while (lo < hi) {
        const int64_t mid = lo + ((hi - lo) >> 1);
        if (ldg_i32(col + mid) < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The vertices with |U(a)| >= 2, listed by tier (warp-aggregated appends).
__global__ void __launch_bounds__(256)
k_tier_lists(int64_t n, const int32_t *__restrict__ dnew, const int32_t *__restrict__ lowcnt, int32_t *lists,
             u64 *acc) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t a0 = (int64_t)blockIdx.x * blockDim.x; a0 < n; a0 += stride) {
        const int64_t a = a0 + threadIdx.x;
        const int32_t k = a < n ? dnew[a] - lowcnt[a] : 0;
        int tier = kTiers;
        if (k >= 2) tier = (k > kTierK0) + (k > kTierK1) + (k > kTierK2) + (k > kTierK3);
        const uint32_t peers = __match_any_sync(0xffffffffu, tier);
        const int leader = __ffs(peers) - 1;
        u64 at = 0;
        if (tier < kTiers && (int)(threadIdx.x & 31) == leader)
            at = atomicAdd(reinterpret_cast<unsigned long long *>(acc + XA_TIERS + tier), (unsigned long long)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, leader);
        if (tier < kTiers) lists[tier * n + static_cast<int64_t>(at) + __popc(peers & lanemask_lt())] = static_cast<int32_t>(a);
    }
}

__device__ __forceinline__ uint32_t label_slot(int32_t c, uint32_t mask) {
    const uint32_t h = static_cast<uint32_t>(c) * 0x9E3779B1u;
    return (h >> 15) & mask;
}

// Shared memory of one vertex: U(a), where each U(b) starts in `col`, its
// length and its first edge number, the triangles at a through each of U(a),
// an open-addressing table of U(a) (positions; load at most 1/4) and the bit
// matrix.
template <int KMAX>
struct CliqueSmem {
    int32_t u[KMAX], start[KMAX], len[KMAX], first[KMAX];
    uint32_t tri[KMAX];
    uint32_t tab[4 * KMAX];
    uint32_t bits[KMAX * (KMAX / 32)];
};

// T threads per vertex with |U(a)| <= KMAX.  Bound by the lookups (4.4e9 on
// R-MAT 20, one shared-memory probe each, most of them misses) and by one
// global atomic per triangle; the matrix turns the 4-clique pairs of a
// triangle into |U(a)| / 32 words.  Replaced one warp per edge (a, b) testing
// every entry of U(a) against b in the graph's adjacency structure, and every
// pair of the hits: R-MAT 20 246 -> 17 ms over the four sizes.
template <int KMAX, int T, int BLOCK>
__global__ void __launch_bounds__(BLOCK)
k_cliques(GraphDev g, const int32_t *__restrict__ lowcnt, const int64_t *__restrict__ ubase,
          const int32_t *__restrict__ list, const u64 *__restrict__ count, uint32_t *tcount, u64 *acc) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    constexpr int NW = T / 32;
    constexpr uint32_t kNone = 0xffffffffu;
    constexpr uint32_t hmask = 4 * KMAX - 1;
    CliqueSmem<KMAX> &S = reinterpret_cast<CliqueSmem<KMAX> *>(s_raw)[threadIdx.x / T];
    const int t = threadIdx.x % T, lane = threadIdx.x & 31, warp = t >> 5;
    auto sync = [] {
        if (T == 32) __syncwarp();
        else __syncthreads();
    };
    const int64_t items = static_cast<int64_t>(*count);
    const int64_t groups = (int64_t)gridDim.x * (BLOCK / T);
    uint64_t k4 = 0;
    for (int64_t it = (int64_t)blockIdx.x * (BLOCK / T) + threadIdx.x / T; it < items; it += groups) {
        const int32_t a = list[it];
        const int64_t a_end = ldg_i64(g.off + a + 1);
        const int64_t a_up = ldg_i64(g.off + a) + ldg_i32(lowcnt + a);
        const int k = static_cast<int>(a_end - a_up);
        const int W = (k + 31) >> 5;
        for (int p = t; p < k; p += T) {
            const int32_t b = ldg_i32(g.col + a_up + p);
            const int64_t o = ldg_i64(g.off + b), e = ldg_i64(g.off + b + 1);
            const int32_t l = ldg_i32(lowcnt + b);
            S.u[p] = b;
            S.start[p] = static_cast<int32_t>(o + l);
            S.len[p] = static_cast<int32_t>(e - o - l);
            S.first[p] = static_cast<int32_t>(ldg_i64(ubase + b));
            S.tri[p] = 0;
        }
        for (int q = t; q < 4 * KMAX; q += T) S.tab[q] = kNone;
        for (int q = t; q < k * W; q += T) S.bits[q] = 0;
        sync();
        for (int p = t; p < k; p += T) {
            uint32_t h = label_slot(S.u[p], hmask);
            while (atomicCAS(&S.tab[h], kNone, static_cast<uint32_t>(p)) != kNone) h = (h + 1) & hmask;
        }
        sync();
        const int32_t top = S.u[k - 1];
        for (int p = warp; p + 1 < k; p += NW) {
            const int32_t len = S.len[p], s0 = S.start[p], f0 = S.first[p];
            uint32_t hits = 0;
            for (int i0 = lane; i0 < len; i0 += 128) {
                // four reads in flight; the row ascends, so past `top` nothing follows
                int32_t c[4];
#pragma unroll
                for (int j = 0; j < 4; j++) c[j] = i0 + 32 * j < len ? ldg_i32(g.col + s0 + i0 + 32 * j) : INT32_MAX;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if (c[j] > top) continue;
                    uint32_t h = label_slot(c[j], hmask), q = S.tab[h];
                    while (q != kNone && S.u[q] != c[j]) {
                        h = (h + 1) & hmask;
                        q = S.tab[h];
                    }
                    if (q != kNone) {
                        atomicOr(&S.bits[p * W + (q >> 5)], 1u << (q & 31));
                        atomicAdd(&S.tri[q], 1u);
                        atomicAdd(tcount + f0 + i0 + 32 * j, 1u);
                        hits++;
                    }
                }
                if (c[0] > top) break;
            }
            hits = __reduce_add_sync(0xffffffffu, hits);
            if (lane == 0 && hits) atomicAdd(&S.tri[p], hits);
        }
        sync();
        const int64_t ua = ldg_i64(ubase + a);
        for (int p = t; p < k; p += T)
            if (S.tri[p]) atomicAdd(tcount + ua + p, S.tri[p]);
        // 4-cliques: G lanes (a power of two, >= W) hold a row's words; the
        // groups of a warp take different rows
        int G = 1;
        while (G < W) G <<= 1;
        const int gl = lane & (G - 1), rows = 32 / G;
        for (int p0 = warp * rows; p0 < k; p0 += NW * rows) {
            const int p = p0 + lane / G;
            const uint32_t mine = p < k && gl < W ? S.bits[p * W + gl] : 0u;
            for (int w = p0 >> 5; w < W; w++) {
                uint32_t word = __shfl_sync(0xffffffffu, mine, w, G);
                while (word) {
                    const int q = w * 32 + __ffs(word) - 1;
                    word &= word - 1;
                    if (gl < W) k4 += __popc(mine & S.bits[q * W + gl]);
                }
            }
        }
        sync();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k4 += __shfl_down_sync(0xffffffffu, k4, o);
    if (lane == 0 && k4) atomic_add128(acc + XA_N6, k4, 0);
}

// Vertices of the last tier, a block each, a warp per edge (a, b): every
// c > b of U(a) adjacent to b is a triangle; the hits are kept (up to
// kCliqueCap) and their adjacent pairs counted.
template <int ADJ>
__global__ void __launch_bounds__(256)
k_cliques_wide(GraphDev g, const int32_t *__restrict__ lowcnt, const int64_t *__restrict__ ubase,
               const int32_t *__restrict__ list, const u64 *__restrict__ count, uint32_t *tcount, u64 *acc) {
    __shared__ int32_t s_common[8][kCliqueCap];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *common = s_common[warp];
    const int64_t items = static_cast<int64_t>(*count);
    uint64_t k4 = 0;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int32_t a = list[it];
        const int64_t a_end = ldg_i64(g.off + a + 1);
        const int64_t a_up = ldg_i64(g.off + a) + ldg_i32(lowcnt + a);
        const int64_t ua = ldg_i64(ubase + a);
        for (int64_t p = warp; a_up + p < a_end; p += 8) {
            const int32_t b = ldg_i32(g.col + a_up + p);
            const int64_t b_up = ldg_i64(g.off + b) + ldg_i32(lowcnt + b), b_end = ldg_i64(g.off + b + 1);
            const int64_t ub = ldg_i64(ubase + b);
            int found = 0;
            for (int64_t base = a_up + p + 1; base < a_end; base += 32) {
                const int64_t i = base + lane;
                int32_t c = -1;
                bool in = false;
                if (i < a_end) {
                    c = ldg_i32(g.col + i);
                    in = has_edge<ADJ>(g, b, c);
                }
                const uint32_t mask = __ballot_sync(0xffffffffu, in);
                if (in) {
                    const int pos = found + __popc(mask & lanemask_lt());
                    if (pos < kCliqueCap) common[pos] = c;
                    const int64_t pc = lower_bound_i32(g.col, b_up, b_end, c);
                    atomicAdd(tcount + ua + (i - a_up), 1u);
                    atomicAdd(tcount + ub + (pc - b_up), 1u);
                }
                found += __popc(mask);
            }
            if (lane == 0 && found) atomicAdd(tcount + ua + p, static_cast<uint32_t>(found));
            __syncwarp();
            if (found <= kCliqueCap) {
                for (int x = 0; x + 1 < found; x++) {
                    const int32_t c = common[x];
                    for (int y = x + 1 + lane; y < found; y += 32) k4 += has_edge<ADJ>(g, c, common[y]) ? 1 : 0;
                }
            } else {
                // too many to keep: walk the rest of U(a) again for each c
                for (int64_t i = a_up + p + 1; i < a_end; i++) {
                    const int32_t c = ldg_i32(g.col + i);
                    if (!has_edge<ADJ>(g, b, c)) continue;
                    for (int64_t q = i + 1 + lane; q < a_end; q += 32) {
                        const int32_t d = ldg_i32(g.col + q);
                        k4 += (has_edge<ADJ>(g, b, d) && has_edge<ADJ>(g, c, d)) ? 1 : 0;
                    }
                }
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k4 += __shfl_down_sync(0xffffffffu, k4, o);
    if (lane == 0 && k4) atomic_add128(acc + XA_N6, k4, 0);
}

// From the triangles per edge: 3 T = sum t_e, N_5 = sum C(t_e, 2), and
// 2 N_3 = sum t_e (d_u + d_v - 4): a triangle's d_a + d_b + d_c - 6 is
// (d - 2) summed over its vertices, each of them on two of its edges.
__global__ void __launch_bounds__(256)
k_triangle_totals(int64_t m, const uint32_t *__restrict__ tcount, const EdgeRec *__restrict__ rec, u64 *acc) {
    uint64_t tlo = 0, thi = 0, nlo = 0, nhi = 0, plo = 0, phi = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
        const uint64_t t = tcount[j];
        if (!t) continue;
        const int4 e = __ldg(reinterpret_cast<const int4 *>(rec + j));  // u, v, d_u, d_v
        add128(tlo, thi, t);
        add128(nlo, nhi, t * (static_cast<uint64_t>(e.z) + static_cast<uint64_t>(e.w) - 4));
        add128(plo, phi, t * (t - 1) / 2);
    }
    warp_add128(tlo, thi);
    warp_add128(nlo, nhi);
    warp_add128(plo, phi);
    if ((threadIdx.x & 31) == 0 && (tlo | thi)) {
        atomic_add128(acc + XA_T3, tlo, thi);
        atomic_add128(acc + XA_N3X2, nlo, nhi);
        if (plo | phi) atomic_add128(acc + XA_N5, plo, phi);
    }
}

// ----------------------------------------------------------------- 4-cycles

// Shared-memory counters cover the top kCycleTop labels, from `base` up, as
// 16-bit halves: labels kCycleTop / 2 apart share a word, so the sorted ends
// of a row fall in different banks.
constexpr int kCycleTop = 1 << 14;
constexpr int kCycleWords = kCycleTop / 2;
constexpr int kCycleBlock = 256;

// For every b the part of N(b) that ends wedges in the counters: the entries
// above b and at least `base` (start, length); low[b]: the first entry >= base.
__global__ void __launch_bounds__(256)
k_cycle_segments(GraphDev g, const int32_t *__restrict__ lowcnt, int32_t base, int2 *seg, int32_t *low) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < g.n; b += stride) {
        const int64_t o = ldg_i64(g.off + b), e = ldg_i64(g.off + b + 1);
        const int64_t up = o + ldg_i32(lowcnt + b);
        const int64_t h = b >= base ? up : lower_bound_i32(g.col, up, e, base);
        seg[b] = make_int2(static_cast<int32_t>(h), static_cast<int32_t>(e - h));
        if (low) low[b] = static_cast<int32_t>(h);
    }
}

// One block per c: for each b in N(c) the ends a > max(b, c) with a >= base
// are counted.  Adding up the counters' old values gives sum C(cnt, 2) in one
// pass.  For c < base every listed end qualifies, so a neighbour costs one
// 8-byte read; only a c among the top labels searches N(b) for its place.
// Bound by the shared-memory atomics (5.6e9 on R-MAT 20).  Replaced counters
// in global memory (4 n bytes per block, 1.3 GB in flight) walked twice from
// the highest vertex: R-MAT 20 166 -> 8.7 ms, and 2.6 ms for the cycles
// without a top label (four ends in flight per lane: 10.2 -> 8.7 ms).
__global__ void __launch_bounds__(kCycleBlock)
k_cycles4(GraphDev g, int32_t base, const int2 *__restrict__ seg, u64 *acc) {
    __shared__ __align__(16) uint32_t s_cnt[kCycleWords];
    __shared__ int32_t s_start[kCycleBlock], s_len[kCycleBlock];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint64_t lo = 0, hi = 0;
    auto clear = [&] {
        for (int q = t; q < kCycleWords / 4; q += kCycleBlock) reinterpret_cast<uint4 *>(s_cnt)[q] = make_uint4(0, 0, 0, 0);
    };
    clear();
    for (int64_t c = blockIdx.x; c < g.n; c += gridDim.x) {
        const int64_t oc = ldg_i64(g.off + c);
        const int64_t d = ldg_i64(g.off + c + 1) - oc;
        if (d < 2) continue;
        // a counter reaches at most d: from 2^16 on the words hold one 32-bit
        // counter each, and the labels above c are taken kCycleWords at a time
        const bool wide = d >= 65536;
        int64_t from = wide ? c + 1 : base;
        if (from < base) from = base;  // the ends below base are counted by the other pass
        uint64_t sum = 0;
        for (; from < g.n; from += wide ? kCycleWords : kCycleTop) {
            __syncthreads();  // counters cleared, segments of the last round read
            for (int64_t i0 = 0; i0 < d; i0 += kCycleBlock) {
                if (i0) __syncthreads();
                int32_t st = 0, len = 0;
                if (i0 + t < d) {
                    const int32_t b = ldg_i32(g.col + oc + i0 + t);
                    const int2 sg = __ldg(seg + b);
                    st = sg.x;
                    len = sg.y;
                    if (c >= base && b < c && len) {
                        const int64_t x = lower_bound_i32(g.col, st, st + static_cast<int64_t>(len), static_cast<int32_t>(c) + 1);
                        len -= static_cast<int32_t>(x - st);
                        st = static_cast<int32_t>(x);
                    }
                }
                s_start[t] = st;
                s_len[t] = len;
                __syncthreads();
                const int nb = d - i0 < kCycleBlock ? static_cast<int>(d - i0) : kCycleBlock;
                for (int x = warp; x < nb; x += kCycleBlock / 32) {
                    const int32_t *row = g.col + s_start[x];
                    const int32_t n_x = s_len[x];
                    for (int32_t i0x = lane; i0x < n_x; i0x += 128) {
                        // four reads in flight before their counts
                        uint32_t idx[4];
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const int32_t i = i0x + 32 * j;
                            idx[j] = i < n_x ? static_cast<uint32_t>(ldg_i32(row + i) - static_cast<int32_t>(from)) : ~0u;
                        }
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            if (!wide && idx[j] != ~0u) {
                                const int sh = idx[j] >= kCycleWords ? 16 : 0;
                                const uint32_t old = atomicAdd(&s_cnt[idx[j] & (kCycleWords - 1)], 1u << sh);
                                sum += (old >> sh) & 0xffffu;
                            } else if (wide && idx[j] < static_cast<uint32_t>(kCycleWords)) {
                                sum += atomicAdd(&s_cnt[idx[j]], 1u);
                            }
                        }
                    }
                }
            }
            __syncthreads();
            clear();
        }
        add128(lo, hi, sum);
    }
    warp_add128(lo, hi);
    if (lane == 0 && (lo | hi)) atomic_add128(acc + XA_N4, lo, hi);
}

// The cycles whose highest vertex is below `base` lie wholly below it (1% of
// the wedges on R-MAT 20; a block per c over global counters took 11.7 ms
// there, this and the kernel after it 2.6 ms).  A warp per c: with at most kLowWedges wedges the
// ends are counted in a table of the warp's own in shared memory, else c is
// listed for the kernel below.
constexpr int kLowWedges = 256;
constexpr int kLowSlots = 2 * kLowWedges;

// The part of N(b), b < base, in (max(b, c), base).
__device__ __forceinline__ int2 low_segment(const GraphDev &g, const int32_t *lowcnt, const int32_t *low, int32_t b,
                                            int32_t c) {
    int64_t st = ldg_i64(g.off + b) + ldg_i32(lowcnt + b);
    const int64_t e = ldg_i32(low + b);
    if (b < c && st < e) st = lower_bound_i32(g.col, st, e, c + 1);
    return make_int2(static_cast<int32_t>(st), static_cast<int32_t>(e - st));
}

__global__ void __launch_bounds__(256)
k_cycles4_low(GraphDev g, const int32_t *__restrict__ lowcnt, int32_t base, const int32_t *__restrict__ low,
              int32_t *heavy, u64 *acc) {
    __shared__ int32_t s_key[8][kLowSlots];
    __shared__ uint32_t s_cnt[8][kLowSlots];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *key = s_key[warp];
    uint32_t *cnt = s_cnt[warp];
    for (int q = lane; q < kLowSlots; q += 32) {
        key[q] = -1;
        cnt[q] = 0;
    }
    __syncwarp();
    uint64_t sum = 0;
    const int64_t nw = (int64_t)gridDim.x * 8;
    for (int64_t c = (int64_t)blockIdx.x * 8 + warp; c < base; c += nw) {
        const int64_t oc = ldg_i64(g.off + c);
        const int32_t d = static_cast<int32_t>(ldg_i32(low + c) - oc);  // its neighbours below base
        if (d < 2) continue;
        uint32_t wedges = 0;
        for (int32_t i = lane; i < d && wedges <= kLowWedges; i += 32)
            wedges += static_cast<uint32_t>(low_segment(g, lowcnt, low, ldg_i32(g.col + oc + i), static_cast<int32_t>(c)).y);
        wedges = wedges > kLowWedges ? kLowWedges + 1 : wedges;
        wedges = __reduce_add_sync(0xffffffffu, wedges);
        if (wedges < 2) continue;
        if (wedges > kLowWedges) {
            if (lane == 0)
                heavy[atomicAdd(reinterpret_cast<unsigned long long *>(acc + XA_HEAVY), 1ull)] = static_cast<int32_t>(c);
            continue;
        }
        for (int32_t i = lane; i < d; i += 32) {
            const int2 sg = low_segment(g, lowcnt, low, ldg_i32(g.col + oc + i), static_cast<int32_t>(c));
            for (int32_t q = 0; q < sg.y; q++) {
                const int32_t a = ldg_i32(g.col + sg.x + q);
                uint32_t h = label_slot(a, kLowSlots - 1);
                while (true) {
                    const int32_t k = atomicCAS(key + h, -1, a);
                    if (k == -1 || k == a) break;
                    h = (h + 1) & (kLowSlots - 1);
                }
                sum += atomicAdd(cnt + h, 1u);
            }
        }
        __syncwarp();
        for (int q = lane; q < kLowSlots; q += 32) {
            key[q] = -1;
            cnt[q] = 0;
        }
        __syncwarp();
    }
    uint64_t hi = 0;
    warp_add128(sum, hi);
    if (lane == 0 && (sum | hi)) atomic_add128(acc + XA_N4, sum, hi);
}

// The listed c, a block each: as k_cycles4, with the block's counters (n
// words, all zero between vertices) in global memory, cleared by walking the
// ends again.
__global__ void __launch_bounds__(kCycleBlock)
k_cycles4_heavy(GraphDev g, const int32_t *__restrict__ lowcnt, const int32_t *__restrict__ low,
                const int32_t *__restrict__ heavy, uint32_t *cnt_all, u64 *acc) {
    __shared__ int32_t s_start[kCycleBlock], s_len[kCycleBlock];
    uint32_t *cnt = cnt_all + static_cast<int64_t>(blockIdx.x) * g.n;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t items = static_cast<int64_t>(acc[XA_HEAVY]);
    uint64_t lo = 0, hi = 0;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int32_t c = heavy[it];
        const int64_t oc = ldg_i64(g.off + c);
        const int32_t d = static_cast<int32_t>(ldg_i32(low + c) - oc);
        uint64_t sum = 0;
        for (int pass = 0; pass < 2; pass++) {
            for (int32_t i0 = 0; i0 < d; i0 += kCycleBlock) {
                __syncthreads();  // the last round's segments read, the first pass counted
                const int2 sg = i0 + t < d ? low_segment(g, lowcnt, low, ldg_i32(g.col + oc + i0 + t), c) : make_int2(0, 0);
                s_start[t] = sg.x;
                s_len[t] = sg.y;
                __syncthreads();
                const int nb = d - i0 < kCycleBlock ? d - i0 : kCycleBlock;
                for (int x = warp; x < nb; x += kCycleBlock / 32) {
                    const int32_t *row = g.col + s_start[x];
                    for (int32_t i = lane; i < s_len[x]; i += 32) {
                        uint32_t *p = cnt + ldg_i32(row + i);
                        if (pass == 0) sum += atomicAdd(p, 1u);
                        else *p = 0u;
                    }
                }
            }
        }
        __syncthreads();  // cleared before the next vertex counts
        add128(lo, hi, sum);
    }
    warp_add128(lo, hi);
    if (lane == 0 && (lo | hi)) atomic_add128(acc + XA_N4, lo, hi);
}

template <int KMAX, int T, int BLOCK>
int launch_cliques(const ps_graph *g, int tier, const int32_t *lists, uint32_t *tcount, u64 *acc, cudaStream_t s) {
    constexpr int smem = static_cast<int>(sizeof(CliqueSmem<KMAX>)) * (BLOCK / T);
    auto kernel = k_cliques<KMAX, T, BLOCK>;
    PS_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    int occ = 0;
    PS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, BLOCK, smem));
    kernel<<<g->sm_count * (occ > 0 ? occ : 1), BLOCK, smem, s>>>(g->dev, g->lowcnt, g->ubase, lists + tier * g->n,
                                                                  acc + XA_TIERS + tier, tcount, acc);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

template <int ADJ>
int launch_wide(const ps_graph *g, const int32_t *lists, uint32_t *tcount, u64 *acc, cudaStream_t s) {
    k_cliques_wide<ADJ><<<g->sm_count * 6, 256, 0, s>>>(g->dev, g->lowcnt, g->ubase, lists + (kTiers - 1) * g->n,
                                                        acc + XA_TIERS + kTiers - 1, tcount, acc);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

struct ExactLayout {
    size_t tcount, acc, lists, seg, low, cnt, fixed;
};

ExactLayout exact_layout(int64_t n, int64_t m) {
    ExactLayout L;
    const size_t n1 = static_cast<size_t>(n > 0 ? n : 1);
    L.tcount = 0;
    L.acc = align256(static_cast<size_t>(m > 0 ? m : 1) * sizeof(uint32_t));
    L.lists = L.acc + align256(XA_WORDS * sizeof(uint64_t));
    L.seg = L.lists + align256(kTiers * n1 * sizeof(int32_t));
    L.low = L.seg + align256(n1 * sizeof(int2));
    L.cnt = L.low + align256(n1 * sizeof(int32_t));
    L.fixed = L.cnt;
    return L;
}

using u128 = unsigned __int128;
using i128 = __int128;

}  // namespace

}  // namespace ps

using namespace ps;

extern "C" size_t ps_exact_scratch_bytes(const ps_graph *g, int max_blocks) {
    if (!g || !g->prefixed) return 0;
    const ExactLayout L = exact_layout(g->n, g->m);
    const int blocks = max_blocks > 0 ? max_blocks : 2 * g->sm_count;
    return L.fixed + static_cast<size_t>(blocks) * static_cast<size_t>(g->n > 0 ? g->n : 1) * sizeof(int32_t);
}

extern "C" int ps_count_exact(const ps_graph *g, void *d_scratch, size_t scratch_bytes, ps_stream_t stream,
                              uint64_t N[6], int64_t C[6]) {
    if (!g || !N || !C) return PS_ERR_ARG;
    if (!g->prefixed) return PS_ERR_STATE;
    const ExactLayout L = exact_layout(g->n, g->m);
    const size_t per_block = static_cast<size_t>(g->n > 0 ? g->n : 1) * sizeof(int32_t);
    if (!d_scratch || (reinterpret_cast<uintptr_t>(d_scratch) & 255u) != 0 ||
        scratch_bytes < L.fixed + per_block)
        return PS_ERR_WORKSPACE;
    int blocks = static_cast<int>((scratch_bytes - L.fixed) / per_block);
    if (blocks > 2 * g->sm_count) blocks = 2 * g->sm_count;
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) return PS_ERR_CUDA;
    if (cur != g->device && cudaSetDevice(g->device) != cudaSuccess) return PS_ERR_CUDA;
    struct Restore {
        int dev, prev;
        ~Restore() {
            if (dev != prev) cudaSetDevice(prev);
        }
    } restore{g->device, cur};

    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(d_scratch);
    uint32_t *tcount = reinterpret_cast<uint32_t *>(base + L.tcount);
    u64 *acc = reinterpret_cast<u64 *>(base + L.acc);
    int32_t *lists = reinterpret_cast<int32_t *>(base + L.lists);
    int2 *seg = reinterpret_cast<int2 *>(base + L.seg);
    int32_t *low = reinterpret_cast<int32_t *>(base + L.low);
    uint32_t *cnt = reinterpret_cast<uint32_t *>(base + L.cnt);
    PS_CUDA_TRY(cudaMemsetAsync(base, 0, L.acc + XA_WORDS * sizeof(uint64_t), s));
    if (g->m > 0) {
        const int sms = g->sm_count;
        k_tier_lists<<<sms * 8, 256, 0, s>>>(g->n, g->dnew, g->lowcnt, lists, acc);
        PS_LAUNCH_CHECK();
        int rc = PS_OK;
        if (g->d_max > kTierK3) {
            switch (g->dev.adj_mode) {
                case kAdjHash: rc = launch_wide<kAdjHash>(g, lists, tcount, acc, s); break;
                case kAdjVtab: rc = launch_wide<kAdjVtab>(g, lists, tcount, acc, s); break;
                default: rc = launch_wide<kAdjSearch>(g, lists, tcount, acc, s); break;
            }
        }
        if (!rc && g->d_max > kTierK2) rc = launch_cliques<kTierK3, 1024, 1024>(g, 3, lists, tcount, acc, s);
        if (!rc && g->d_max > kTierK1) rc = launch_cliques<kTierK2, 256, 256>(g, 2, lists, tcount, acc, s);
        if (!rc && g->d_max > kTierK0) rc = launch_cliques<kTierK1, 256, 256>(g, 1, lists, tcount, acc, s);
        if (!rc) rc = launch_cliques<kTierK0, 32, 256>(g, 0, lists, tcount, acc, s);
        if (rc) return rc;
        k_triangle_totals<<<sms * 8, 256, 0, s>>>(g->m, tcount, g->rec, acc);
        PS_LAUNCH_CHECK();
        const int32_t top = static_cast<int32_t>(g->n > kCycleTop ? g->n - kCycleTop : 0);
        k_cycle_segments<<<sms * 8, 256, 0, s>>>(g->dev, g->lowcnt, top, seg, top ? low : nullptr);
        PS_LAUNCH_CHECK();
        k_cycles4<<<sms * 6, kCycleBlock, 0, s>>>(g->dev, top, seg, acc);
        PS_LAUNCH_CHECK();
        if (top) {
            PS_CUDA_TRY(cudaMemsetAsync(cnt, 0, static_cast<size_t>(blocks) * per_block, s));
            // (the vertex lists of the cliques are done with)
            k_cycles4_low<<<sms * 6, 256, 0, s>>>(g->dev, g->lowcnt, top, low, lists, acc);
            PS_LAUNCH_CHECK();
            k_cycles4_heavy<<<blocks, kCycleBlock, 0, s>>>(g->dev, g->lowcnt, low, lists, cnt, acc);
            PS_LAUNCH_CHECK();
        }
    }
    static_assert(XA_WORDS <= Readback::kWords, "the words fit a read-back");
    Readback r;
    const int rc = r.queue(acc, XA_WORDS, nullptr, 0, s);
    if (rc) return rc;
    PS_CUDA_TRY(cudaStreamSynchronize(s));
    const uint64_t *h = r.words;
    auto pair = [&](int w) { return (static_cast<u128>(h[w + 1]) << 64) | h[w]; };
    const ps_stats &S = g->stats;
    const u128 T3 = pair(XA_T3);
    u128 n[7];
    n[1] = (static_cast<u128>(S.N1_hi) << 64) | S.N1_lo;
    if (static_cast<u128>(S.W) < T3) return PS_ERR_OVERFLOW;  // cannot happen on a valid graph
    n[2] = static_cast<u128>(S.W) - T3;
    n[3] = pair(XA_N3X2) / 2;
    n[4] = pair(XA_N4);
    n[5] = pair(XA_N5);
    n[6] = pair(XA_N6);
    for (int i = 1; i <= 6; i++) {
        if (n[i] >> 64) return PS_ERR_OVERFLOW;
        N[i - 1] = static_cast<uint64_t>(n[i]);
    }
    // Eq. (1) is upper triangular with unit diagonal: back-substitute
    const i128 c6 = static_cast<i128>(n[6]);
    const i128 c5 = static_cast<i128>(n[5]) - 6 * c6;
    const i128 c4 = static_cast<i128>(n[4]) - c5 - 3 * c6;
    const i128 c3 = static_cast<i128>(n[3]) - 4 * c5 - 12 * c6;
    const i128 c2 = static_cast<i128>(n[2]) - 2 * c3 - 4 * c4 - 6 * c5 - 12 * c6;
    const i128 c1 = static_cast<i128>(n[1]) - c3 - 2 * c5 - 4 * c6;
    const i128 c[6] = {c1, c2, c3, c4, c5, c6};
    for (int i = 0; i < 6; i++) {
        if (c[i] > static_cast<i128>(INT64_MAX) || c[i] < static_cast<i128>(INT64_MIN)) return PS_ERR_OVERFLOW;
        C[i] = static_cast<int64_t>(c[i]);
    }
    return PS_OK;
}
