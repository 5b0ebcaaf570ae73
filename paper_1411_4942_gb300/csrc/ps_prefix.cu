// ps_prefix.cu -- the guide tables that shorten the inverse-CDF search over
// the prefixes of tau (Section 3) and lambda (Section 4), and the hub bitmaps
// of the adjacency test, both queued by the load step; ps_tau_prefix, which
// publishes the totals; and the per-vertex tables of one adjacency variant.
#include <algorithm>

#include "ps_internal.h"

namespace ps {

// Guide table: bucket b holds r in [b << shift, (b + 1) << shift), and G[b]
// is the edge that the first r of bucket b selects.  Edge j covers r in
// [P[j-1], P[j] - 1], so it owns the buckets whose first r falls in that
// range -- a contiguous run, and every bucket has exactly one owner.  Each
// lane writes its own short run; a warp writes long runs together.  A warp
// takes kGuideGroups groups of 32 edges per step with all their prefix loads
// issued first.
// The heavy edges, with the long runs, are the last ones: on small graphs a
// warp takes one group, so more warps share them (49k edges: 20 -> 6 us for
// both tables).
constexpr int kGuideGroups = 4;

// Table blockIdx.y: 0 = tau, 1 = lambda, its total from the status words.
// Nothing is written when the load has found the input invalid or a sum too
// large (the prefixes need not ascend then).
template <int GROUPS>
__global__ void __launch_bounds__(256)
k_guide_fill(int64_t m, const uint64_t *__restrict__ ptau, const uint64_t *__restrict__ plam, int64_t gcap,
             int32_t *gtau, int32_t *glam, const u64 *__restrict__ status) {
    const uint64_t *P = blockIdx.y ? plam : ptau;
    int32_t *G = blockIdx.y ? glam : gtau;
    const uint64_t total = status[blockIdx.y ? ST_L_LO : ST_W_LO];
    if (status[ST_FLAGS] != 0 || status[ST_M_UPPER] != static_cast<u64>(m) || total == 0) return;
    const int shift = guide_shift(total, gcap);
    const int64_t B = static_cast<int64_t>(((total - 1) >> shift) + 1);
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * blockDim.x / 32;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    if (blockIdx.x == 0 && threadIdx.x == 0) G[B] = static_cast<int32_t>(m - 1);
    for (int64_t g0 = wid * GROUPS; g0 * 32 < m; g0 += nw * GROUPS) {
        uint64_t prev[GROUPS], cur[GROUPS];
#pragma unroll
        for (int u = 0; u < GROUPS; u++) {
            const int64_t j = (g0 + u) * 32 + lane;
            prev[u] = (j >= 1 && j <= m) ? __ldg(P + j - 1) : 0ull;
            cur[u] = j < m ? __ldg(P + j) : 0ull;
        }
        // bucket numbers are below B + 1 <= 2^31, so after the shift the runs
        // are handled in 32 bits
#pragma unroll
        for (int u = 0; u < GROUPS; u++) {
            const int64_t j = (g0 + u) * 32 + lane;
            uint32_t bstart = 0, len = 0;
            if (j < m && cur[u] != prev[u]) {
                bstart = prev[u] ? static_cast<uint32_t>((prev[u] - 1) >> shift) + 1u : 0u;
                const uint32_t bend = static_cast<uint32_t>((cur[u] - 1) >> shift);
                len = bstart <= bend ? bend - bstart + 1u : 0u;
            }
            if (len <= 8) {
                for (uint32_t q = 0; q < len; q++) G[bstart + q] = static_cast<int32_t>(j);
            }
            uint32_t longs = __ballot_sync(0xffffffffu, len > 8);
            while (longs) {
                const int l = __ffs(longs) - 1;
                longs &= longs - 1;
                const uint32_t bs = __shfl_sync(0xffffffffu, bstart, l);
                const uint32_t ln = __shfl_sync(0xffffffffu, len, l);
                const int32_t jj = static_cast<int32_t>((g0 + u) * 32 + l);
                for (uint32_t q = lane; q < ln; q += 32) G[bs + q] = jj;
            }
        }
    }
}

// Hub bitmap rows, a block per (hub, chunk of labels) at a time: the block sets
// bit x for every neighbour x inside its chunk in shared memory, then writes
// the chunk out whole (coalesced), so no clearing pass and no global atomics.
// Bound by the rows' bytes (512 MB on R-MAT 20); blocks of 512 with 32 KB, four
// per SM, so that one writes while another clears or sets bits.
constexpr int kHubThreads = 512;
constexpr int64_t kHubChunkWords = 1 << 13;

__global__ void __launch_bounds__(kHubThreads, 4)
k_hub_rows(int64_t n, int64_t bit_base, const int64_t *__restrict__ coff, const int32_t *__restrict__ ccol,
           uint32_t *bits, int64_t words, const u64 *__restrict__ status) {
    __shared__ __align__(16) uint32_t s_row[kHubChunkWords];
    const int64_t hubs = static_cast<int64_t>(status[ST_HUBS]);
    const int64_t chunks = (words + kHubChunkWords - 1) / kHubChunkWords;
    for (int64_t b = blockIdx.x; b < hubs * chunks; b += gridDim.x) {
        const int64_t h = b / chunks, w0 = (b % chunks) * kHubChunkWords;
        const int nw = static_cast<int>(min(kHubChunkWords, words - w0));
        for (int w = threadIdx.x; w < (nw + 3) / 4; w += kHubThreads)
            reinterpret_cast<uint4 *>(s_row)[w] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const int64_t r = n - hubs + h;
        const int64_t o = ldg_i64(coff + r), e = ldg_i64(coff + r + 1);
        const int64_t lo = bit_base + w0 * 32;  // bit_base % 32 == 0
        const uint32_t span = static_cast<uint32_t>(nw) * 32;
        for (int64_t i = o + threadIdx.x; i < e; i += kHubThreads) {
            const uint32_t x = static_cast<uint32_t>(ldg_i32(ccol + i) - lo);  // below lo: wraps past the span
            if (x < span) atomicOr(s_row + (x >> 5), 1u << (x & 31));
        }
        __syncthreads();
        uint32_t *row = bits + h * words + w0;
        for (int w = threadIdx.x; w < nw; w += kHubThreads) row[w] = s_row[w];
        __syncthreads();
    }
}

// Inserts every arc (x -> y) into the table of x with compare-and-swap; the
// tables' contents are deterministic, their slot layout is not.
constexpr int kVtabItems = 8;
__global__ void __launch_bounds__(256)
k_vtab_build(int64_t n, int64_t nnz, const int64_t *__restrict__ coff, const int32_t *__restrict__ ccol,
             int32_t *vtab, u64 *status) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool failed = false;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c * kVtabItems < nnz; c += stride) {
        const int64_t i0 = c * kVtabItems;
        int64_t lo = 0, hi = n;  // last row r with coff[r] <= i0
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (ldg_i64(coff + mid) <= i0) lo = mid;
            else hi = mid - 1;
        }
        int64_t r = lo;
        int64_t ro = ldg_i64(coff + r), rend = ldg_i64(coff + r + 1);
        for (int t = 0; t < kVtabItems; t++) {
            const int64_t i = i0 + t;
            if (i >= nnz) break;
            while (rend <= i) {
                r++;
                ro = rend;
                rend = ldg_i64(coff + r + 1);
            }
            const int32_t y = ldg_i32(ccol + i);
            const uint64_t size = static_cast<uint64_t>(2 * (rend - ro));
            int32_t *tab = vtab + 2 * ro;
            uint64_t s = vtab_start(y, size);
            bool done = false;
            for (uint64_t probe = 0; probe < size; probe++) {
                const int32_t old = atomicCAS(tab + s, kEmptyLabel, y);
                if (old == kEmptyLabel || old == y) {
                    done = true;
                    break;
                }
                s = (s + 1 == size) ? 0 : s + 1;
            }
            failed |= !done;
        }
    }
    if (failed) raise_flag(status, F_OVERFLOW);
}

int launch_guides(ps_graph *g, cudaStream_t s) {
    const int64_t m = g->L.m_cap;
    if (m <= 0) return PS_OK;
    // one resident wave (the loop strides over the edges)
    const bool small = m < (int64_t{1} << 22);
    auto kernel = small ? k_guide_fill<1> : k_guide_fill<kGuideGroups>;
    const int64_t per_block = 256 * (small ? 1 : kGuideGroups);
    const int64_t blocks = std::min<int64_t>((m + per_block - 1) / per_block, (int64_t)g->sm_count * 8);
    kernel<<<dim3((unsigned)blocks, 2), 256, 0, s>>>(m, g->ptau, g->plam, g->L.gcap, g->gtau, g->glam, g->status);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

int launch_hub_rows(ps_graph *g, cudaStream_t s) {
    const int64_t words = g->L.hub_words, rows = std::min(g->L.hub_cap, g->L.n);
    if (rows <= 0 || words <= 0) return PS_OK;
    const int64_t blocks = rows * ((words + kHubChunkWords - 1) / kHubChunkWords);
    k_hub_rows<<<(unsigned)std::min<int64_t>(blocks, (int64_t)g->sm_count * 4), kHubThreads, 0, s>>>(
        g->L.n, g->L.hub_bit_base, g->off, g->col, g->hub, words, g->status);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

int prefix_graph(ps_graph *g, cudaStream_t s) {
    const int64_t n = g->n, m = g->m;
    const int sms = g->sm_count;
    // the prefixes P_tau, P_lambda and their totals W, Lambda were written
    // by the load step's edge-table kernel (with F_OVERFLOW if a sum passed
    // 2^64), N_1 and the hub count by its vertex pass; all were read back at
    // its end
    const uint64_t flags = g->load_flags;
    if (flags & F_TIMEOUT) return PS_ERR_TIMEOUT;
    ps_stats &S = g->stats;
    S.W = g->load_totals[0];
    S.Lambda = g->load_totals[1];
    S.N1_lo = g->load_totals[2];
    S.N1_hi = g->load_totals[3];
    S.n = n;
    S.m = m;
    S.d_max = g->d_max;
    if (flags & F_OVERFLOW) return PS_ERR_OVERFLOW;

    // the guide tables (with guides off they have at most 2 buckets) and the
    // hub rows were queued by the load step
    const int tshift = S.W > 0 ? guide_shift(S.W, g->L.gcap) : 0;
    const int lshift = S.Lambda > 0 ? guide_shift(S.Lambda, g->L.gcap) : 0;
    S.tau_shift = tshift;
    S.lambda_shift = lshift;

    // per-vertex hash tables
    if (g->vtab) {
        PS_CUDA_TRY(cudaMemsetAsync(g->vtab, 0xFF, sizeof(int32_t) * g->L.vtab_slots, s));
        if (g->nnz > 0) {
            int64_t chunks = (g->nnz + kVtabItems - 1) / kVtabItems;
            int64_t blocks = (chunks + 255) / 256;
            if (blocks > (int64_t)sms * 64) blocks = (int64_t)sms * 64;
            k_vtab_build<<<(unsigned)blocks, 256, 0, s>>>(n, g->nnz, g->off, g->col, g->vtab, g->status);
            PS_LAUNCH_CHECK();
        }
    }

    const int64_t hubs = static_cast<int64_t>(g->load_totals[4]);
    S.hubs = hubs;
    // The kernels queued after the load's synchronisation cannot fail on
    // valid state; later calls on `stream` are ordered after them.

    GraphDev &D = g->dev;
    D.filt_off = g->filt ? static_cast<uint64_t>(g->filt - g->hub) : 0;
    D.filt_words = static_cast<uint32_t>(g->L.filt_words);
    D.vtab = g->vtab;
    D.adj_mode = g->vtab ? kAdjVtab : (g->filt ? kAdjHash : kAdjSearch);
    D.hub_bit_base = static_cast<int32_t>(g->L.hub_bit_base);
    D.off = g->off;
    D.col = g->col;
    D.rec = g->rec;
    D.ptau = g->ptau;
    D.plam = g->plam;
    D.gtau = g->gtau;
    D.glam = g->glam;
    D.hub = g->hub;
    D.W = S.W;
    D.Lambda = S.Lambda;
    D.n = n;
    D.m = m;
    D.hub_start = static_cast<int32_t>(n - hubs);
    D.hub_words = static_cast<int32_t>(g->L.hub_words);
    D.tau_shift = tshift;
    D.lam_shift = lshift;
    g->prefixed = true;
    return (S.W == 0 || S.Lambda == 0) ? PS_NO_PATHS : PS_OK;
}

}  // namespace ps
