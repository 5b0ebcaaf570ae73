// ps_ingest.cu -- ps_csr_from_edges: the undirected simple graph of Section 2
// from a raw edge list, on the device.  The paper's experiments read SNAP edge
// lists and time the whole run from them (Section 6); this turns such a list
// -- either direction, repeats, self-loops -- into the sorted symmetric CSR
// that ps_load_csr takes: self-loops dropped, both arcs of every remaining
// pair, each arc once, rows ascending.
//
// Every edge becomes its pair (lo, hi), lo <= hi, sorted by (lo, hi): e pairs
// instead of 2e arcs.  The first copies of the proper pairs (lo < hi), in that
// order, are every row's neighbours above it; a stable sort of them by hi
// gives every row's neighbours below it, in order too.  So row r is its part
// of the second list followed by its part of the first, and the columns are
// written in two streaming passes.  (Sorting 2e arcs by column, then by row,
// marking and compacting them took 3.95 ms for R-MAT 20's 16.8M drawn edges.)
#include <algorithm>
#include <utility>

#include "ps_internal.h"

namespace ps {

namespace {

enum : int {
    IS_FLAGS = 0,     // F_ARG: an id outside [0, n)
    IS_PAIRS = 1,     // proper pairs kept (half the arcs)
    IS_WORDS = 8,
};

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

int id_bits(int64_t n) {
    int bits = 1;
    while (bits < 31 && (static_cast<uint64_t>(n > 0 ? n - 1 : 0) >> bits) != 0) bits++;
    return bits;
}

constexpr int kPairLists = 3;

struct IngestLayout {
    int64_t scan_words;
    size_t status, scan, spans, clear_end, k[kPairLists], v[kPairLists], counts, total;
};

bool ingest_layout(int64_t n, int64_t n_edges, IngestLayout *L) {
    if (n < 0 || n >= INT32_MAX || n_edges < 0 || n_edges > (INT32_MAX - 1) / 2) return false;
    IngestLayout l{};
    const int64_t n_tiles = (n + kScanTile - 1) / kScanTile, e_tiles = (n_edges + kScanTile - 1) / kScanTile;
    const int64_t es = sort_scan_tiles(n_edges);
    // up to 8 passes by (lo, hi) and 4 by hi, the compaction and the offsets
    l.scan_words = 12 * scan_words<uint32_t>(es) + scan_words<uint32_t>(e_tiles) + scan_words<int64_t>(n_tiles);
    const size_t e1 = static_cast<size_t>(n_edges > 0 ? n_edges : 1), n1 = static_cast<size_t>(n > 0 ? n : 1);
    size_t p = 0;
    auto take = [&](size_t bytes) {
        const size_t at = p;
        p = align256(p + (bytes > 0 ? bytes : 1));
        return at;
    };
    l.status = take(IS_WORDS * sizeof(uint64_t));
    l.scan = take(static_cast<size_t>(l.scan_words) * sizeof(uint64_t));
    l.spans = take(2 * n1 * sizeof(int2));
    l.clear_end = p;
    for (int i = 0; i < kPairLists; i++) {
        l.k[i] = take(e1 * sizeof(uint32_t));
        l.v[i] = take(e1 * sizeof(uint32_t));
    }
    l.counts = take(static_cast<size_t>(256) * sort_tiles(n_edges) * sizeof(uint32_t));
    l.total = p;
    *L = l;
    return true;
}

// Edge i as (hi, lo); a pair with an id out of range becomes (0, 0), which
// like every self-loop is no proper pair.
__global__ void k_ingest_pairs(int64_t n, int64_t n_edges, const int32_t *__restrict__ src,
                               const int32_t *__restrict__ dst, uint32_t *__restrict__ hi, uint32_t *__restrict__ lo,
                               u64 *status) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_edges; i += stride) {
        int32_t u = __ldg(src + i), v = __ldg(dst + i);
        if (u < 0 || u >= n || v < 0 || v >= n) {
            bad = true;
            u = v = 0;
        }
        hi[i] = static_cast<uint32_t>(max(u, v));
        lo[i] = static_cast<uint32_t>(min(u, v));
    }
    if (bad) raise_flag(status + IS_FLAGS, F_ARG);
}

// 1 for the first copy of each proper pair of the sorted list.
struct LoadFirst {
    const uint32_t *hi, *lo;
    __device__ uint32_t operator()(int64_t i) const {
        const uint32_t h = __ldg(hi + i), l = __ldg(lo + i);
        return h != l && (i == 0 || __ldg(hi + i - 1) != h || __ldg(lo + i - 1) != l) ? 1u : 0u;
    }
};
// The kept pairs, compacted, and each row's part of them.  A row's part spans
// the kept pairs of its whole run of the sorted list, so its ends are known
// at the run's first and last pair whether those are kept or not.
struct StoreKept {
    const uint32_t *hi, *lo;
    uint32_t *hi_out, *lo_out;
    int2 *span;
    u64 *status;
    int64_t n_edges;
    __device__ void operator()(int64_t i, uint32_t exc, uint32_t inc) const {
        const uint32_t l = __ldg(lo + i);
        if (inc != exc) {
            hi_out[exc] = __ldg(hi + i);
            lo_out[exc] = l;
        }
        if (i == 0 || __ldg(lo + i - 1) != l) span[l].x = static_cast<int32_t>(exc);
        if (i == n_edges - 1) {
            span[l].y = static_cast<int32_t>(inc);
            status[IS_PAIRS] = inc;
        } else if (__ldg(lo + i + 1) != l) {
            span[l].y = static_cast<int32_t>(inc);
        }
    }
};

// Each row's part of the list sorted by hi.
__global__ void __launch_bounds__(256)
k_ingest_spans(const u64 *__restrict__ pairs, const uint32_t *__restrict__ hi, int2 *span) {
    const int64_t m = static_cast<int64_t>(*pairs);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
        const uint32_t h = __ldg(hi + j);
        if (j == 0 || __ldg(hi + j - 1) != h) span[h].x = static_cast<int32_t>(j);
        if (j == m - 1 || __ldg(hi + j + 1) != h) span[h].y = static_cast<int32_t>(j + 1);
    }
}

struct LoadDegree {
    const int2 *below, *above;
    __device__ int64_t operator()(int64_t r) const {
        const int2 b = below[r], a = above[r];
        return static_cast<int64_t>(b.y - b.x) + (a.y - a.x);
    }
};
struct StoreRowOffsets {
    int64_t *off;
    int64_t n;
    __device__ void operator()(int64_t i, int64_t exc, int64_t inc) const {
        off[i] = exc;
        if (i == n - 1) off[n] = inc;
    }
};

// The columns: entry j of the list sorted by hi is the (j - below.x)-th of row
// hi; entry j of the list sorted by (lo, hi) comes (j - above.x)-th after the
// entries below lo.
__global__ void __launch_bounds__(256)
k_ingest_columns(const u64 *__restrict__ pairs, const uint32_t *__restrict__ bhi, const uint32_t *__restrict__ blo,
                 const uint32_t *__restrict__ ahi, const uint32_t *__restrict__ alo, const int2 *__restrict__ below,
                 const int2 *__restrict__ above, const int64_t *__restrict__ off, int32_t *__restrict__ col) {
    const int64_t m = static_cast<int64_t>(*pairs);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < m; j += stride) {
        const uint32_t r = __ldg(bhi + j), s = __ldg(alo + j);
        const uint32_t x = __ldg(blo + j), y = __ldg(ahi + j);
        const int2 b = __ldg(below + s);
        col[ldg_i64(off + r) + (j - __ldg(&below[r].x))] = static_cast<int32_t>(x);
        col[ldg_i64(off + s) + (b.y - b.x) + (j - __ldg(&above[s].x))] = static_cast<int32_t>(y);
    }
}

// Takes a scan's counter and slots from the cleared region.
template <typename T>
ScanState<T> ingest_scan_state(char *ws, const IngestLayout &L, int64_t tiles, int64_t *used) {
    u64 *at = reinterpret_cast<u64 *>(ws + L.scan) + *used;
    *used += scan_words<T>(tiles);
    return ScanState<T>{at + 2, reinterpret_cast<uint32_t *>(at), reinterpret_cast<u64 *>(ws + L.status) + IS_FLAGS};
}

}  // namespace

}  // namespace ps

using namespace ps;

extern "C" size_t ps_ingest_workspace_bytes(int64_t n, int64_t n_edges) {
    IngestLayout L;
    return ingest_layout(n, n_edges, &L) ? L.total : 0;
}

extern "C" int ps_csr_from_edges(int64_t n, int64_t n_edges, const int32_t *d_src, const int32_t *d_dst,
                                 void *d_workspace, size_t ws_bytes, int64_t *d_off, int32_t *d_col,
                                 int64_t *nnz, ps_stream_t stream) {
    if (!nnz || !d_off || n_edges < 0 || (n_edges > 0 && (!d_src || !d_dst || !d_col))) return PS_ERR_ARG;
    *nnz = 0;
    IngestLayout L;
    if (!ingest_layout(n, n_edges, &L)) return PS_ERR_ARG;
    if (!d_workspace || (reinterpret_cast<uintptr_t>(d_workspace) & 255u) != 0 || ws_bytes < L.total)
        return PS_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    char *ws = static_cast<char *>(d_workspace);
    u64 *status = reinterpret_cast<u64 *>(ws + L.status);
    int2 *above = reinterpret_cast<int2 *>(ws + L.spans), *below = above + (n > 0 ? n : 1);
    uint32_t *k[kPairLists], *v[kPairLists];
    for (int i = 0; i < kPairLists; i++) {
        k[i] = reinterpret_cast<uint32_t *>(ws + L.k[i]);
        v[i] = reinterpret_cast<uint32_t *>(ws + L.v[i]);
    }
    uint32_t *counts = reinterpret_cast<uint32_t *>(ws + L.counts);
    const int sms = sm_count_of_current_device();
    int64_t used = 0;
    // the status words, the scans' counters and slots, and the rows' spans
    PS_CUDA_TRY(cudaMemsetAsync(ws, 0, L.clear_end, s));
    if (n_edges > 0) {
        auto blocks = [&](int64_t items) { return static_cast<unsigned>(std::min<int64_t>((items + 255) / 256, (int64_t)sms * 16)); };
        k_ingest_pairs<<<blocks(n_edges), 256, 0, s>>>(n, n_edges, d_src, d_dst, k[0], v[0], status);
        PS_LAUNCH_CHECK();
        const int bits = id_bits(n);
        auto take = [&](int64_t tiles, ScanState<uint32_t> *scan) {
            *scan = ingest_scan_state<uint32_t>(ws, L, tiles, &used);
            return PS_OK;
        };
        // (hi, lo) pairs by lo * 2^bits + hi, 8 bits at a time
        SortPass sort[kMaxPasses];
        int passes = 0, a = 0, b = 1, rc;
        for (int shift = 0; shift < 2 * bits; shift += 8) {
            const int nbits = std::min(8, 2 * bits - shift);
            SortPass &p = sort[passes++];
            if (shift >= bits) p = {n_edges, nullptr, v[a], k[a], v[b], k[b], shift - bits, nbits, 0, counts};
            else p = {n_edges, nullptr, k[a], v[a], k[b], v[b], shift, nbits, shift + nbits <= bits ? 0 : bits - shift, counts};
            std::swap(a, b);
        }
        rc = sort_passes(sort, passes, take, s);
        if (rc) return rc;
        // the kept pairs into list b
        const int64_t tiles = (n_edges + kScanTile - 1) / kScanTile;
        k_scan<uint32_t, kScanBlock, kScanItems><<<(unsigned)tiles, kScanBlock, 0, s>>>(
            n_edges, ingest_scan_state<uint32_t>(ws, L, tiles, &used), 0u, OpSum(), LoadFirst{k[a], v[a]},
            StoreKept{k[a], v[a], k[b], v[b], above, status, n_edges});
        PS_LAUNCH_CHECK();
        // the same pairs sorted by hi: from list b between the other two
        const u64 *kept = status + IS_PAIRS;
        int from = b, to = a, spare = kPairLists - 1;
        passes = 0;
        for (int shift = 0; shift < bits; shift += 8) {
            sort[passes++] = {n_edges, kept, k[from], v[from], k[to], v[to], shift, std::min(8, bits - shift), 0, counts};
            from = to;
            std::swap(to, spare);
        }
        rc = sort_passes(sort, passes, take, s);
        if (rc) return rc;
        k_ingest_spans<<<blocks(n_edges), 256, 0, s>>>(kept, k[from], below);
        PS_LAUNCH_CHECK();
        if (n > 0) {
            const int64_t n_tiles = (n + kScanTile - 1) / kScanTile;
            k_scan<int64_t, kScanBlock, kScanItems><<<(unsigned)n_tiles, kScanBlock, 0, s>>>(
                n, ingest_scan_state<int64_t>(ws, L, n_tiles, &used), (int64_t)0, OpSum(), LoadDegree{below, above},
                StoreRowOffsets{d_off, n});
            PS_LAUNCH_CHECK();
        }
        k_ingest_columns<<<blocks(n_edges), 256, 0, s>>>(kept, k[from], v[from], k[b], v[b], below, above, d_off, d_col);
        PS_LAUNCH_CHECK();
    } else {
        PS_CUDA_TRY(cudaMemsetAsync(d_off, 0, static_cast<size_t>(n + 1) * sizeof(int64_t), s));
    }
    static_assert(IS_WORDS <= Readback::kWords, "the words fit a read-back");
    Readback r;
    const int rc = r.queue(status, IS_WORDS, nullptr, 0, s);
    if (rc) return rc;
    PS_CUDA_TRY(cudaStreamSynchronize(s));
    const uint64_t *st = r.words;
    const int status_code = flags_to_status(st[IS_FLAGS]);
    if (status_code != PS_OK) return status_code;
    *nnz = 2 * static_cast<int64_t>(st[IS_PAIRS]);
    return PS_OK;
}
