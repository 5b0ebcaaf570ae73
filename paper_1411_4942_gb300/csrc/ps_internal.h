// ps_internal.h -- host-side internals shared by the library's translation
// units: the graph handle, the workspace layout and error helpers.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/pathsample.h"
#include "ps_device.cuh"
#include "ps_scan.cuh"

namespace ps {

// Sort tiers of the row relabel-and-sort step, by row length.
constexpr int kTierA = 32;      // one warp, one key per lane
constexpr int kTierB = 1024;    // one warp, up to 32 keys per lane in registers
// (512 on graphs below kSmallArcs arcs: there one warp's 1024-entry row is the
// load's tail.  Loads with rows of up to 512 / 1024 entries here: 1.8M arcs
// 260 / 269 us, 4M 382 / 386, 15.5M 856 / 865 and 930 / 944 (but R-MAT 18, 7.6M
// arcs, 593 / 572), 31M 1511 / 1501 and 1570 / 1580, 54M 2345 / 2309, 64M
// 3003 / 2867, 128M 5489 / 5358, 233M 9174 / 9025.)
constexpr int kTierBSmall = 512;
constexpr int64_t kSmallArcs = int64_t{1} << 24;
inline int tier_b(int64_t nnz) { return nnz < kSmallArcs ? kTierBSmall : kTierB; }
constexpr int kTierC = 4096;    // one block, registers + 16 KB shared; above: block radix sort
// Rows longer than this have their lower arcs listed a warp or a block per
// row; shorter rows by a warp per 32 rows.
constexpr int kLongRow = 128;
// Hub rows are only worth a bitmap above this degree (default of the tuning
// field hub_min_degree).
constexpr int kHubMinDegree = 64;
constexpr int kHubSpanLog2 = 19;   // default hub-row span beside the edge filter
constexpr int kHubRowsMax = 8192;  // default hub-row cap beside the edge filter
constexpr int64_t kCoarseGuideEdges = int64_t{1} << 25;  // default guide of m/4 buckets from here
// Items per tile of every scan.
constexpr int kScanBlock = 256;
constexpr int kScanItems = 8;
constexpr int64_t kScanTile = kScanBlock * kScanItems;

struct Tuning {
    int block_size;
    int blocks_per_sm;
    int guide_log2_ratio;  // >= 1: m << r buckets; -1: no guide; <= -2: m >> -r buckets
    int hub_count;         // 0: none
    int samples_per_thread;  // batched launch: 1 or 2
    int hub_min_degree;
    int hub_span_log2;     // hub rows cover the top 2^span labels; 0: all labels
    int adj_mode;          // kAdjHash or kAdjSearch
    int draw_order;        // ordered samplers: 0 by size, > 0 always, -1 never
};
Tuning resolve_tuning(const ps_tuning *t, int64_t n, int64_t nnz);
struct Layout {
    int64_t n, nnz, m_cap, gcap, hub_cap, hub_words, hub_bit_base;
    int64_t scan_words;    // 64-bit words of one load's scans (tile counters and slots)
    int64_t filt_words;    // 32-bit words of the edge filter; 0 without it
    int64_t vtab_slots;    // 0 without the per-vertex tables
    size_t status, off, col, rank, lowcnt, ubase, dnew, row_span, row_upper, rec, ptau, plam, gtau, glam, hub, filt, vtab;
    size_t keys0, keys1, vals0, vals1, inv, counts, scan;
    size_t total;
};
bool make_layout(int64_t n, int64_t nnz, const Tuning &t, Layout *L);

}  // namespace ps

struct ps_graph {
    ps::Layout L;
    ps::Tuning tune;
    char *ws;
    int device;
    int sm_count;
    int64_t n, nnz, m, d_max;
    int64_t scan_used;  // words of the scan region taken by this load's scans
    // device arrays (inside ws)
    ps::u64 *status;
    int64_t *off;
    int32_t *col;
    int32_t *rank;
    int32_t *lowcnt;
    int64_t *ubase;
    int2 *row_span, *row_upper;  // of each row: (offset, degree) and (lower arcs, first edge)
    int32_t *dnew;
    ps::EdgeRec *rec;
    uint64_t *ptau, *plam;
    int32_t *gtau, *glam;
    uint32_t *hub;
    uint32_t *filt;
    int32_t *vtab;
    bool prefixed;
    // read back at the end of ps_load_csr: W, Lambda, N_1 (lo, hi), the hub
    // count and the flags, so ps_tau_prefix needs no synchronisation
    uint64_t load_totals[5] = {0, 0, 0, 0, 0};
    uint64_t load_flags = 0;
    ps_stats stats;
    ps::GraphDev dev;
    // fork / join events of this graph's calls
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    ~ps_graph() {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
    }
};

namespace ps {

#define PS_CUDA_TRY(call)                         \
    do {                                          \
        cudaError_t e_ = (call);                  \
        if (e_ != cudaSuccess) return PS_ERR_CUDA; \
    } while (0)

int sm_count_of_current_device();
int flags_to_status(uint64_t flags);
// Two non-blocking streams of `device` for independent kernels within one
// call, which has them to itself while this object lives: with streams shared
// by the calls of a device, a call that joins them, or reads from them, stands
// behind everything that another call's stream still has before its own.
// The caller joins them to its stream and synchronises that before the end.
// stream[0] null: none free.
class SideStreams {
  public:
    explicit SideStreams(int device);
    ~SideStreams();
    SideStreams(const SideStreams &) = delete;
    SideStreams &operator=(const SideStreams &) = delete;
    cudaStream_t stream[2] = {nullptr, nullptr};

  private:
    int dev_, pair_ = -1, generation_ = 0;
};

// Id of the context current on this thread; 0 when there is none or the
// driver cannot say.  (Unlike context handles, ids are never reused.)
unsigned long long current_context_id();

// Device words brought to the host (ps_readback.cu): `words` holds them once
// the stream they were queued on has been synchronised, which the caller does
// before this object ends.
class Readback {
  public:
    static constexpr int kWords = 64;
    Readback();
    ~Readback();
    Readback(const Readback &) = delete;
    Readback &operator=(const Readback &) = delete;
    // words[0, na) = a[0, na), words[na, na + nb) = b[0, nb) (device, 8-byte words)
    int queue(const void *a, int na, const void *b, int nb, cudaStream_t s);

  private:
    uint64_t own_[kWords];
    int dev_ = -1, slot_ = -1, generation_ = 0;

  public:
    uint64_t *words = own_;
};

// Every kernel launch is followed by this: counts the launch (reported by
// ps_kernel_launches) and checks the launch error.
void count_launch();
#define PS_LAUNCH_CHECK()                       \
    do {                                        \
        ::ps::count_launch();                   \
        PS_CUDA_TRY(cudaGetLastError());        \
    } while (0)

// One stable pass of a radix sort (ps_sort.cu) by `bits` (at most 8) bits of
// the key from `shift` on; keys have no bits above those of the sort's last
// pass.  vin null: the values are the items' indices.  vshift > 0: the digit
// goes on with the value's lowest bits, vshift of its bits being the key's.
// dcount (device, may be null) bounds the items at run time.  counts: 256
// words per tile.  max_key (device, may be null): the largest key; a pass
// after the first that sorts by higher bits only does nothing.
struct SortPass {
    int64_t count;
    const u64 *dcount;
    const uint32_t *kin, *vin;
    uint32_t *kout, *vout;
    int shift, bits, vshift;
    uint32_t *counts;
    const u64 *max_key = nullptr;
};
int64_t sort_tiles(int64_t count);
// tiles of the pass's scan (0: it needs none and `scan` is not touched)
int64_t sort_scan_tiles(int64_t count);
int sort_pass(const SortPass &p, const ScanState<uint32_t> &scan, cudaStream_t s);

// All passes of a sort of at most kClusterItems items in one launch; *done is
// left false where the device has no room for such a cluster.
constexpr int64_t kClusterItems = 1 << 17;
constexpr int kMaxPasses = 8;
int sort_cluster(const SortPass *p, int n, cudaStream_t s, bool *done);

// A sort's passes (at most kMaxPasses) in order; `take(tiles, &scan)` supplies
// the scan of a pass that needs one.  Short lists go to one cluster: up to its
// 131,072 items it is the faster way (ingest of 1,000 pairs 150 -> 121 us,
// of 40,000 190 -> 142, of 131,072 211 -> 166), and it holds no more.
template <typename Take>
inline int sort_passes(const SortPass *p, int n, Take take, cudaStream_t s) {
    if (n > 0 && p[0].count <= kClusterItems) {
        bool done = false;
        const int rc = sort_cluster(p, n, s, &done);
        if (rc || done) return rc;
    }
    for (int i = 0; i < n; i++) {
        ScanState<uint32_t> scan{};
        int rc = sort_scan_tiles(p[i].count) ? take(sort_scan_tiles(p[i].count), &scan) : PS_OK;
        if (rc == PS_OK) rc = sort_pass(p[i], scan, s);
        if (rc) return rc;
    }
    return PS_OK;
}

// The scans of a load take their tile counter and slots from a region of
// 64-bit words that the load clears once.
template <typename T>
inline int64_t scan_words(int64_t tiles) { return 2 + ((SlotOf<T>::kWords * tiles + 1) & ~int64_t{1}); }
template <typename T>
inline int take_scan(ps_graph *g, int64_t tiles, ScanState<T> *st) {
    const int64_t words = scan_words<T>(tiles);
    if (g->scan_used + words > g->L.scan_words) return PS_ERR_WORKSPACE;
    u64 *at = reinterpret_cast<u64 *>(g->ws + g->L.scan) + g->scan_used;
    st->counter = reinterpret_cast<uint32_t *>(at);
    st->slots = at + 2;
    st->status = g->status;
    g->scan_used += words;
    return PS_OK;
}
template <typename T, typename Op, typename Load, typename Store>
inline int run_scan(ps_graph *g, int64_t count, T identity, Op op, Load load, Store store, cudaStream_t s) {
    if (count <= 0) return PS_OK;
    const int64_t tiles = (count + kScanTile - 1) / kScanTile;
    ScanState<T> st;
    const int rc = take_scan(g, tiles, &st);
    if (rc) return rc;
    k_scan<T, kScanBlock, kScanItems><<<(unsigned)tiles, kScanBlock, 0, s>>>(count, st, identity, op, load, store);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

// The guide tables and the hub rows (ps_prefix.cu), queued by the load step:
// both take their sizes (the totals W and Lambda, the hub count) from the
// status words on the device.  The guide tables are left alone when the input
// has turned out invalid.
int launch_guides(ps_graph *g, cudaStream_t s);
int launch_hub_rows(ps_graph *g, cudaStream_t s);
// Guide bucket of r is r >> guide_shift(total, buckets).
__host__ __device__ inline int guide_shift(uint64_t total, int64_t gcap) {
    int s = 0;
    while (s < 63 && ((total - 1) >> s) >= static_cast<uint64_t>(gcap)) s++;
    return s;
}

// The edge table (ps_edges.cu): after the rows are relabelled and sorted and
// ubase is known, writes every edge record and prefix, sets every edge's bits
// in the edge filter (cleared before), and raises F_ASYM for an asymmetric
// input.
int build_edge_table(ps_graph *g, cudaStream_t s);
// steps (one translation unit each)
int load_graph(ps_graph *g, const int64_t *d_off, const int32_t *d_col, cudaStream_t s);
int prefix_graph(ps_graph *g, cudaStream_t s);
int launch_sampler(const ps_graph *g, int sampler, uint64_t k, uint64_t seed, uint64_t first_id,
                   uint64_t *d_hist, cudaStream_t s);
// Both samplers over ids first_id ..; one without anything to draw is left out.
int launch_samplers(const ps_graph *g, uint64_t k3, uint64_t *d_hist6, uint64_t kc, uint64_t *d_hist4, uint64_t seed,
                    uint64_t first_id, cudaStream_t s);
// Samples in the order of their edge draws (ps_order.cu), in chunks of what the
// scratch holds and at most 2^27; the largest k_chunk that a scratch can be
// asked for is kOrderMaxChunk.
constexpr uint64_t kOrderMaxChunk = 1ull << 31;
size_t ordered_scratch_bytes(uint64_t k_chunk);
bool order_never(const ps_graph *g);  // every number of samples of this graph is drawn plainly
int launch_ordered(const ps_graph *g, int sampler, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *d_hist,
                   void *d_scratch, size_t scratch_bytes, cudaStream_t s);
int launch_batch(const void *d_table, int32_t n_graphs, const ps_work *d_items, int64_t n_items,
                 uint64_t *d_hist, uint32_t *d_counter, const Tuning &t, cudaStream_t s);
// Records the adjacency variant shared by a descriptor table's graphs (0: mixed).
void note_table_adjacency(const void *d_table, int adj);

}  // namespace ps
