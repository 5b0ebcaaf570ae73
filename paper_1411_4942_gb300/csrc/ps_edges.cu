// ps_edges.cu -- the edge table of Sections 3-4 by transposition.
//
// Edge j = (u, v), u < v, is the j-th upper arc in row-major order of the
// canonical CSR: j = ubase[u] + (iu - lowcnt[u]), iu the position of v in
// N(u).  Its record also needs jv, the position of u in N(v).  Listing the
// lower arcs (v -> u, u < v) in row-major order gives the same edges ordered
// by (v, u); a STABLE sort of that list by u orders them by (u, v), which is
// exactly the edge order.  So after the sort, entry j names edge j: u is its
// key, the arc's index i gives jv = i - off(v), and v is the (j - ubase[u])-th
// upper neighbour of u.  No per-edge search is needed, and every record is
// written in order (coalesced 32-byte stores).  The same kernel computes the
// weights tau_j and lambda_j and their exact prefixes (a look-back scan in
// edge order), so the prefix step never reads the records back.
//
// The sort is an LSD radix sort with 8-bit digits over the bits of n - 1 (3
// passes for up to 2^24 vertices; ps_sort.cu).
//
// Scratch (the load step's own; nothing here is live afterwards): the
// ping-pong (key, value) buffers use the prefix regions of the workspace
// (P_tau and P_lambda, 8 bytes per edge each) and, for the sorted list, the
// G_tau region (written only later, by the guide-table build); the digit
// counts have their own region.
#include <algorithm>

#include "ps_internal.h"

namespace ps {

// (1) The lower arcs of every row, compacted in row-major order: entry
// t = lbase(r) + p for the p-th entry of row r (p < lowcnt[r]), where
// lbase(r) = off(r) - ubase[r] counts the lower arcs of the rows before r.
// key = the smaller endpoint, value = the arc's index.  Rows up to kLongRow
// entries (labels below ST_LONG; rows are in degree order): warp w takes
// rows [32 w, 32 w + 32), whose lower arcs are one contiguous range of the
// output, written 32 * kListBatch entries at a time, each lane finding its
// entries' rows among the warp's 32 by a shuffle search of their lbase values
// (the batch's column reads are independent, so they are in flight
// together).  Longer rows: a warp per row up to kTierC entries, a block per
// row above.  An asymmetric input can have
// more lower arcs than the buffers hold; those beyond m_cap are dropped (the
// status check after the load rejects the graph).
//
// The listing also sets the bits of every edge that no hub row holds in the
// edge filter (one atomic without a result per edge): it streams little else,
// so the filter stays in L2.  (From the edge-table kernel, which streams 60
// bytes per edge, the same atomics took 0.96 ms on the 3M-vertex graph.)
struct EdgeFilter {
    uint32_t *words;  // null: no filter
    uint32_t count;
    int32_t hub_bit_base;

    // The edge u < v, hubs from hub_start up.
    __device__ __forceinline__ void add(int32_t u, int32_t v, int32_t hub_start) const {
        if (!words || (v >= hub_start && u >= hub_bit_base)) return;
        const uint64_t h = edge_hash(u, v);
        atomicOr(words + filter_word(h, count), filter_mask(h));
    }
};

constexpr int kListBatch = 4;
constexpr int64_t kFewRows = int64_t{1} << 18;

__global__ void __launch_bounds__(256)
k_lower_arcs(int64_t n, const int64_t *__restrict__ coff, const int32_t *__restrict__ ccol,
             const int64_t *__restrict__ ubase, uint32_t *__restrict__ key, uint32_t *__restrict__ val,
             int64_t m_cap, const u64 *__restrict__ status, EdgeFilter F) {
    const int32_t hub_start = static_cast<int32_t>(n - static_cast<int64_t>(status[ST_HUBS]));
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * blockDim.x / 32;
    const int64_t r_long = static_cast<int64_t>(status[ST_LONG]);
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; w * 32 < r_long; w += nwarps) {
        const int64_t r = w * 32 + lane;
        const int64_t r_end = (w * 32 + 32 < r_long) ? w * 32 + 32 : r_long;
        const int64_t lb_end = ldg_i64(coff + r_end) - ldg_i64(ubase + r_end);
        int64_t o = 0, lb = lb_end;  // lanes past the last row never match
        if (r < r_end) {
            o = ldg_i64(coff + r);
            lb = o - ldg_i64(ubase + r);
        }
        const int64_t lb0 = __shfl_sync(0xffffffffu, lb, 0);
        for (int64_t t0 = lb0; t0 < lb_end; t0 += 32 * kListBatch) {
            int64_t t[kListBatch], i[kListBatch];
            int32_t c[kListBatch], row[kListBatch];
#pragma unroll
            for (int u = 0; u < kListBatch; u++) {
                t[u] = t0 + 32 * u + lane;
                // the last lane whose row starts at or before t holds t
                int at = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int64_t x = __shfl_sync(0xffffffffu, lb, at + step);
                    if (x <= t[u]) at += step;
                }
                row[u] = static_cast<int32_t>(w * 32 + at);
                i[u] = __shfl_sync(0xffffffffu, o, at) + (t[u] - __shfl_sync(0xffffffffu, lb, at));
            }
#pragma unroll
            for (int u = 0; u < kListBatch; u++) c[u] = (t[u] < lb_end && t[u] < m_cap) ? ldg_i32(ccol + i[u]) : 0;
#pragma unroll
            for (int u = 0; u < kListBatch; u++)
                if (t[u] < lb_end && t[u] < m_cap) {
                    key[t[u]] = static_cast<uint32_t>(c[u]);
                    val[t[u]] = static_cast<uint32_t>(i[u]);
                    F.add(c[u], row[u], hub_start);
                }
        }
    }
}

// Rows of kLongRow + 1 .. kTierC entries: a warp per row, the next row's
// offsets fetched while the current one is copied.  With SHORT, before them
// the shorter rows, 8 lanes each (150k rows of about 20 entries 32 -> 20 us),
// or a warp each where there are no more rows than warps.
constexpr int kShortLanes = 8;
template <bool SHORT>
__global__ void __launch_bounds__(256)
k_lower_arcs_mid(const int64_t *__restrict__ coff, const int32_t *__restrict__ ccol,
                 const int32_t *__restrict__ lowcnt, const int64_t *__restrict__ ubase,
                 uint32_t *__restrict__ key, uint32_t *__restrict__ val, int64_t m_cap,
                 const u64 *__restrict__ status, int64_t n, EdgeFilter F) {
    const int32_t hub_start = static_cast<int32_t>(n - static_cast<int64_t>(status[ST_HUBS]));
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * blockDim.x / 32;
    const bool share = SHORT && n > nw;
    if (share) {
        const int at = lane % kShortLanes;
        const int64_t s_end = static_cast<int64_t>(status[ST_LONG]);
        for (int64_t q = static_cast<int64_t>(status[ST_TIER]) + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kShortLanes;
             q < s_end; q += nw * (32 / kShortLanes)) {
            const int64_t o = ldg_i64(coff + q), lb = o - ldg_i64(ubase + q);
            const int32_t low = ldg_i32(lowcnt + q);
            for (int32_t p0 = 0; p0 < low; p0 += kShortLanes * kListBatch) {
                int32_t c[kListBatch];
#pragma unroll
                for (int u = 0; u < kListBatch; u++) {
                    const int32_t p = p0 + kShortLanes * u + at;
                    c[u] = (p < low && lb + p < m_cap) ? ldg_i32(ccol + o + p) : 0;
                }
#pragma unroll
                for (int u = 0; u < kListBatch; u++) {
                    const int32_t p = p0 + kShortLanes * u + at;
                    if (p < low && lb + p < m_cap) {
                        key[lb + p] = static_cast<uint32_t>(c[u]);
                        val[lb + p] = static_cast<uint32_t>(o + p);
                        F.add(c[u], static_cast<int32_t>(q), hub_start);
                    }
                }
            }
        }
    }
    const int64_t r_end = static_cast<int64_t>(status[ST_TIER + 3]);
    int64_t r = static_cast<int64_t>(status[SHORT && !share ? ST_TIER : ST_LONG]) +
                ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    int64_t o_ = 0, ub_ = 0;
    int32_t low_ = 0;
    if (r < r_end) {
        o_ = ldg_i64(coff + r);
        ub_ = ldg_i64(ubase + r);
        low_ = ldg_i32(lowcnt + r);
    }
    for (; r < r_end; r += nw) {
        const int64_t o = o_, lb = o_ - ub_;
        const int32_t low = low_;
        if (r + nw < r_end) {
            o_ = ldg_i64(coff + r + nw);
            ub_ = ldg_i64(ubase + r + nw);
            low_ = ldg_i32(lowcnt + r + nw);
        }
        for (int64_t p0 = 0; p0 < low; p0 += 32 * kListBatch) {
            int32_t c[kListBatch];
#pragma unroll
            for (int u = 0; u < kListBatch; u++) {
                const int64_t p = p0 + 32 * u + lane;
                c[u] = (p < low && lb + p < m_cap) ? ldg_i32(ccol + o + p) : 0;
            }
#pragma unroll
            for (int u = 0; u < kListBatch; u++) {
                const int64_t p = p0 + 32 * u + lane;
                if (p < low && lb + p < m_cap) {
                    key[lb + p] = static_cast<uint32_t>(c[u]);
                    val[lb + p] = static_cast<uint32_t>(o + p);
                    F.add(c[u], static_cast<int32_t>(r), hub_start);
                }
            }
        }
    }
}

// Rows above kTierC entries: a block per row.
__global__ void __launch_bounds__(256)
k_lower_arcs_long(int64_t n, const int64_t *__restrict__ coff, const int32_t *__restrict__ ccol,
                  const int32_t *__restrict__ lowcnt, const int64_t *__restrict__ ubase,
                  uint32_t *__restrict__ key, uint32_t *__restrict__ val, int64_t m_cap,
                  const u64 *__restrict__ status, EdgeFilter F) {
    const int32_t hub_start = static_cast<int32_t>(n - static_cast<int64_t>(status[ST_HUBS]));
    const int64_t r0 = static_cast<int64_t>(status[ST_TIER + 3]);
    for (int64_t r = r0 + blockIdx.x; r < n; r += gridDim.x) {
        const int64_t o = ldg_i64(coff + r), low = ldg_i32(lowcnt + r);
        const int64_t lb = o - ldg_i64(ubase + r);
        for (int64_t p0 = 0; p0 < low; p0 += 256 * kListBatch) {
            int32_t c[kListBatch];
#pragma unroll
            for (int u = 0; u < kListBatch; u++) {
                const int64_t p = p0 + 256 * u + threadIdx.x;
                c[u] = (p < low && lb + p < m_cap) ? ldg_i32(ccol + o + p) : 0;
            }
#pragma unroll
            for (int u = 0; u < kListBatch; u++) {
                const int64_t p = p0 + 256 * u + threadIdx.x;
                if (p < low && lb + p < m_cap) {
                    key[lb + p] = static_cast<uint32_t>(c[u]);
                    val[lb + p] = static_cast<uint32_t>(o + p);
                    F.add(c[u], static_cast<int32_t>(r), hub_start);
                }
            }
        }
    }
}

// (2) Edge j from the sorted entry j: u its key, i its arc (in row v, at
// position jv), v the (j - ubase[u])-th upper neighbour of u.  The checks
// that u's upper range holds j and that arc i lies in v's row (where, holding
// u < v, it is a lower arc) hold exactly when the input is symmetric (every
// lower arc has its upper partner and vice versa); otherwise F_ASYM.  A
// thread builds Q edges at j0, j0 + step, ..., their loads issued together
// stage by stage (the chain sorted entry -> row of u -> v -> row of v is
// otherwise a string of dependent round trips per edge), and returns their
// weights (zero past m or for a bad edge).  The rows' offsets and degrees come
// as one 8-byte word each, and a record is one store: L1's tags were the
// busiest unit (65% of peak), with two loads per row and two stores 32 bytes
// apart from lane to lane.  115M edges 2.00 -> 1.77 ms, 15.7M 272 -> 242 us
// (0.95 ms and 0.13 ms at the copy rate).
template <int Q>
__device__ __forceinline__ void edge_group(int64_t j0, int step, int64_t m, int64_t n,
                                           const uint32_t *__restrict__ skey, const uint32_t *__restrict__ sval,
                                           const int2 *__restrict__ row_span, const int2 *__restrict__ row_upper,
                                           const int32_t *__restrict__ ccol, EdgeRec *rec, U64x2 (&w)[Q], bool &asym) {
    // every offset, label and degree is below 2^31 (nnz < 2^31), so the
    // stages work in 32 bits
    int32_t u[Q], i[Q], ou[Q], du[Q], iu[Q], v[Q], ov[Q], dv[Q];
    bool ok[Q];
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int64_t j = j0 + step * q;
        const uint32_t uk = j < m ? __ldg(skey + j) : 0u;
        i[q] = j < m ? static_cast<int32_t>(__ldg(sval + j)) : 0;
        ok[q] = j < m && uk < static_cast<uint64_t>(n);
        u[q] = ok[q] ? static_cast<int32_t>(uk) : 0;
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int2 span = __ldg(row_span + u[q]), upper = __ldg(row_upper + u[q]);
        ou[q] = span.x;
        du[q] = span.y;
        const int64_t rank_in_upper = j0 + step * q - upper.y;
        const int64_t pos = upper.x + rank_in_upper;
        ok[q] = ok[q] && rank_in_upper >= 0 && pos < du[q];
        iu[q] = ok[q] ? static_cast<int32_t>(pos) : 0;
    }
#pragma unroll
    for (int q = 0; q < Q; q++) v[q] = ok[q] ? ldg_i32(ccol + ou[q] + iu[q]) : 0;
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int2 span = __ldg(row_span + v[q]);
        ov[q] = span.x;
        dv[q] = span.y;
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
        const int64_t j = j0 + step * q;
        w[q] = U64x2{0, 0};
        if (j >= m) continue;
        const int32_t jv = i[q] - ov[q];
        if (!ok[q] || jv < 0 || jv >= dv[q]) {
            asym = true;
            continue;
        }
        asm volatile("st.global.v8.s32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                     :
                     : "l"(rec + j), "r"(u[q]), "r"(v[q]), "r"(du[q]), "r"(dv[q]), "r"(iu[q]), "r"(jv), "r"(ou[q]), "r"(ov[q])
                     : "memory");
        w[q] = edge_weights(du[q], dv[q], iu[q], jv);
    }
}

// The edge table and the exact prefixes of its weights in one pass: each
// block takes a tile of the look-back scan (kRecScanItems edges per thread,
// lane-contiguous rows of 32), builds its edges kRecItems rows at a time,
// parks their weights in shared memory and scans them (so the records are
// never read back for the prefix sums).
constexpr int kRecItems = 4;
constexpr int kRecScanItems = 8;
static_assert(kRecScanItems % kRecItems == 0, "whole groups per tile");
static_assert(kScanBlock * kRecScanItems >= kScanTile, "the workspace holds scan slots per kScanTile items");

// (Capped at 64 registers, four blocks per SM: while one block waits at the
// tile's barriers or on its look-back, the others build records; the
// uncapped 80-register build, three blocks per SM, took 1 ms more per load
// on the 3M-vertex graph.)
__global__ void __launch_bounds__(kScanBlock, 4)
k_edge_records_scan(int64_t m, int64_t n, const uint32_t *__restrict__ skey, const uint32_t *__restrict__ sval,
                    const int2 *__restrict__ row_span, const int2 *__restrict__ row_upper,
                    const int32_t *__restrict__ ccol, EdgeRec *rec, u64 *status, ScanState<U64x2> st,
                    uint64_t *ptau, uint64_t *plam) {
    __shared__ U64x2 s_w[kRecScanItems * kScanBlock];
    const int64_t tile = scan_ticket(st);
    const int64_t wbase = scan_wbase<kScanBlock, kRecScanItems>(tile);
    bool asym = false;
#pragma unroll
    for (int g0 = 0; g0 < kRecScanItems; g0 += kRecItems) {
        U64x2 w[kRecItems];
        edge_group<kRecItems>(wbase + 32 * g0, 32, m, n, skey, sval, row_span, row_upper, ccol, rec, w, asym);
#pragma unroll
        for (int q = 0; q < kRecItems; q++) s_w[(g0 + q) * kScanBlock + threadIdx.x] = w[q];
    }
    if (asym) raise_flag(status, F_ASYM);
    U64x2 v[kRecScanItems];
#pragma unroll
    for (int i = 0; i < kRecScanItems; i++) v[i] = s_w[i * kScanBlock + threadIdx.x];
    scan_tile<U64x2, kScanBlock, kRecScanItems>(tile, wbase, v, m, st, U64x2{0, 0}, OpSum(),
                                                StorePrefix{ptau, plam, status, m});
}

int build_edge_table(ps_graph *g, cudaStream_t s) {
    const Layout &L = g->L;
    const int64_t n = L.n, nnz = L.nnz, m = L.m_cap;
    if (nnz <= 0 || m <= 0) return PS_OK;
    const int sms = g->sm_count;
    char *ws = g->ws;
    // (key, value) buffers of m entries each: the lower arcs are listed into
    // the P_tau region, the passes ping-pong between it and the P_lambda
    // region, and the last pass writes to the G_tau region (at least 8 bytes
    // per edge), which nothing reads before the guide tables are built -- so
    // the prefixes can be written while the sorted list is still being read
    uint32_t *ka = reinterpret_cast<uint32_t *>(ws + L.ptau), *va = ka + m;
    uint32_t *kb = reinterpret_cast<uint32_t *>(ws + L.plam), *vb = kb + m;
    uint32_t *kg = reinterpret_cast<uint32_t *>(ws + L.gtau), *vg = kg + m;
    int bits = 0;
    while (bits < 31 && (static_cast<uint64_t>(n > 0 ? n - 1 : 0) >> bits) != 0) bits++;
    const int passes = bits > 0 ? (bits + 7) / 8 : 1;
    const EdgeFilter F{g->filt, static_cast<uint32_t>(L.filt_words), static_cast<int32_t>(L.hub_bit_base)};
    if (n > 0) {
        // few rows: a warp each for the short ones too (5,000 rows: 16 -> 4 us;
        // 32 short rows are up to 32 steps for one warp)
        const bool few = n < kFewRows;
        if (!few) {
            int64_t blocks = (n + 255) / 256;  // a warp per 32 rows
            if (blocks > (int64_t)sms * 16) blocks = (int64_t)sms * 16;
            k_lower_arcs<<<(unsigned)blocks, 256, 0, s>>>(n, g->off, g->col, g->ubase, ka, va, m, g->status, F);
            PS_LAUNCH_CHECK();
        }
        if (few) {
            k_lower_arcs_mid<true><<<(unsigned)(sms * 8), 256, 0, s>>>(g->off, g->col, g->lowcnt, g->ubase, ka, va, m,
                                                                       g->status, n, F);
            PS_LAUNCH_CHECK();
        } else if (g->d_max > kLongRow) {
            k_lower_arcs_mid<false><<<(unsigned)(sms * 6), 256, 0, s>>>(g->off, g->col, g->lowcnt, g->ubase, ka, va, m,
                                                                        g->status, n, F);
            PS_LAUNCH_CHECK();
        }
        if (g->d_max > kTierC) {
            k_lower_arcs_long<<<(unsigned)(sms * 4), 256, 0, s>>>(n, g->off, g->col, g->lowcnt, g->ubase, ka, va, m,
                                                                   g->status, F);
            PS_LAUNCH_CHECK();
        }
    }
    SortPass sort[kMaxPasses];
    for (int pass = 0; pass < passes; pass++) {
        const int shift = 8 * pass;
        const bool last = pass == passes - 1;
        uint32_t *ko = last ? kg : kb, *vo = last ? vg : vb;
        sort[pass] = {m, nullptr, ka, va, ko, vo, shift, std::max(1, std::min(8, bits - shift)), 0,
                      reinterpret_cast<uint32_t *>(ws + L.counts)};
        kb = ka;
        vb = va;
        ka = ko;
        va = vo;
    }
    auto take = [g](int64_t tiles, ScanState<uint32_t> *scan) { return take_scan(g, tiles, scan); };
    int rc = sort_passes(sort, passes, take, s);
    if (rc) return rc;
    // ka/va: the sorted list, in the G_tau region
    const int64_t stiles = (m + kScanBlock * kRecScanItems - 1) / (kScanBlock * kRecScanItems);
    ScanState<U64x2> scan;
    rc = take_scan(g, stiles, &scan);
    if (rc) return rc;
    k_edge_records_scan<<<(unsigned)stiles, kScanBlock, 0, s>>>(
        m, n, ka, va, g->row_span, g->row_upper, g->col, g->rec, g->status, scan, g->ptau, g->plam);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

}  // namespace ps
