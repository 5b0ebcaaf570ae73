// ps_batch.cu -- ps_batch_sample: one persistent launch over a queue of work
// items drawn from many loaded graphs.  Each block takes an item (a range of
// sample ids of one graph and one sampler), runs it with the same per-sample
// code as the plain launches and adds its class counts to the item's slot.
//
// When every graph of a descriptor table uses the same adjacency variant
// (recorded on the host by ps_batch_prepare), the launch uses a kernel
// compiled for that variant alone, which needs fewer registers and so keeps
// more warps resident; mixed tables use the kernel that handles all of them.
#include <mutex>
#include <unordered_map>

#include "ps_internal.h"
#include "ps_sample.cuh"

namespace ps {

namespace {
std::mutex g_table_mutex;
std::unordered_map<const void *, int> g_table_adj;  // d_table -> common variant (0: mixed)
}  // namespace

void note_table_adjacency(const void *d_table, int adj) {
    std::lock_guard<std::mutex> lock(g_table_mutex);
    g_table_adj[d_table] = adj;
}

static int table_adjacency(const void *d_table) {
    std::lock_guard<std::mutex> lock(g_table_mutex);
    auto it = g_table_adj.find(d_table);
    return it == g_table_adj.end() ? 0 : it->second;
}

template <int ADJ>
__device__ __forceinline__ int batch_sample(const GraphDev &g, int sampler, uint64_t seed, uint64_t id) {
    return sampler == 0 ? sample_3path<ADJ>(g, seed, id) : sample_centred<ADJ>(g, seed, id);
}

// Two samples of one thread with the filter adjacency, their steps
// interleaved: both draws (edge, record, neighbours) as straight-line code,
// then both samples' tests, so the two dependent chains overlap.  The same
// counts as two calls of batch_sample.
__device__ __forceinline__ void batch_sample2_hash(const GraphDev &g, int sampler, uint64_t seed, uint64_t id0,
                                                   uint64_t id1, int &c0, int &c1) {
    EdgeRec e0, e1;
    int32_t a0, b0, a1, b1;
    if (sampler == 0) {
        path3_draw(g, seed, id0, e0, a0, b0);
        path3_draw(g, seed, id1, e1, a1, b1);
        const int32_t x[6] = {a0, e0.u, a0, a1, e1.u, a1}, y[6] = {e0.v, b0, b0, e1.v, b1, b1};
        const PairRow none[6] = {{0, -1}, {0, -1}, {0, -1}, {0, -1}, {0, -1}, {0, -1}};
        bool r[6];
        pair_tests<6>(g, x, y, none, r);
        c0 = a0 == b0 ? 0 : class3(r[0], r[1], r[2]);
        c1 = a1 == b1 ? 0 : class3(r[3], r[4], r[5]);
    } else {
        centred_draw(g, seed, id0, e0, a0, b0);
        centred_draw(g, seed, id1, e1, a1, b1);
        // the chords only for centred paths (u' == v' is not one)
        const int32_t x[2] = {a0, a1}, y[2] = {b0, b1};
        const PairRow none[2] = {{0, -1}, {0, -1}};
        bool k[2];
        pair_tests<2>(g, x, y, none, k);
        c0 = c1 = 0;
        bool r[2];
        if (k[0] && a0 != b0) {
            const int32_t p[2] = {a0, e0.u}, q[2] = {e0.v, b0};
            const PairRow row[2] = {{e0.ov, e0.dv}, {e0.ou, e0.du}};
            pair_tests<2>(g, p, q, row, r);
            c0 = 1 + (int)r[0] + (int)r[1];
        }
        if (k[1] && a1 != b1) {
            const int32_t p[2] = {a1, e1.u}, q[2] = {e1.v, b1};
            const PairRow row[2] = {{e1.ov, e1.dv}, {e1.ou, e1.du}};
            pair_tests<2>(g, p, q, row, r);
            c1 = 1 + (int)r[0] + (int)r[1];
        }
    }
}

constexpr int kAheadItems = 4;

// ADJ = 0: any variant, chosen per item; otherwise the table's only variant.
// counter[0] hands out items; counter[1] counts items skipped because their
// graph does not use the variant this kernel was compiled for.  Registers
// are capped for 1024 resident threads per SM with one sample per thread in
// flight (SPT = 1), 512 with two (SPT = 2, graphs with an edge filter; other variants
// take their two samples one after the other), 640 in blocks of 128: capped for
// 512 those took up to 108 registers, so that a fifth block did not fit (36
// R-MAT graphs, all by filter 886 -> 752 us, of mixed variants 2038 -> 1866).
template <int BLOCK, int ADJ, int SPT>
__global__ void __launch_bounds__(BLOCK, (SPT == 1 ? 1024 : 640) / BLOCK)
k_batch(const GraphDev *__restrict__ table, int32_t n_graphs, const ps_work *__restrict__ items,
        int64_t n_items, uint64_t *hist, uint32_t *counter) {
    // The next item is copied, and the one after it claimed, while this one
    // runs, so a block does not stand still for the queue's three round trips
    // (claim, item, graph); items come grouped by graph, so the graph is mostly
    // in place: 96 R-MAT graphs, 4096-sample items, 6.29 -> 5.29 ms.  Only
    // while kAheadItems items per block are left: near the end of the queue a
    // claimed item would wait for its block while others idle (200 served
    // requests in items of 65536 samples took 12.4 ms claiming ahead to the
    // end, 11.0 ms so).
    __shared__ ps_work s_w[2];
    __shared__ uint32_t s_item[2];
    __shared__ GraphDev s_g;
    static_assert(sizeof(ps_work) == 32 && sizeof(GraphDev) % 4 == 0, "copied by words");
    constexpr uint32_t kNone = ~0u;
    const int64_t ahead_end = n_items - static_cast<int64_t>(kAheadItems) * gridDim.x;
    uint32_t claim = kNone;  // thread 0: the item after the current one
    if (threadIdx.x == 0) {
        const uint32_t it = atomicAdd(counter, 1u);
        if (it < ahead_end) claim = atomicAdd(counter, 1u);
        s_item[0] = it;
        if (it < n_items) s_w[0] = items[it];
    }
    __syncthreads();
    uint32_t graph = kNone;  // of s_g; n_graphs: the empty one
    for (int at = 0; s_item[at] < n_items; at ^= 1) {
        if (threadIdx.x == 0) {
            s_item[at ^ 1] = claim;
            if (claim < n_items) {
                const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(&s_w[at ^ 1]));
                const char *src = reinterpret_cast<const char *>(items + claim);  // 8-byte aligned
#pragma unroll
                for (int i = 0; i < 32; i += 8)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + i), "l"(src + i) : "memory");
                claim = claim < ahead_end ? atomicAdd(counter, 1u) : kNone;
            }
        }
        const ps_work w = s_w[at];
        // an item that names no graph, whatever number stands there (kNone too),
        // takes the empty one: nothing to sample
        const uint32_t named = min(w.graph, static_cast<uint32_t>(n_graphs));
        if (named != graph) {
            graph = named;
            if (graph < static_cast<uint32_t>(n_graphs)) {
                for (int i = threadIdx.x; i < static_cast<int>(sizeof(GraphDev) / 4); i += BLOCK)
                    reinterpret_cast<uint32_t *>(&s_g)[i] = __ldg(reinterpret_cast<const uint32_t *>(table + graph) + i);
            } else if (threadIdx.x == 0) {
                s_g.W = s_g.Lambda = 0;
                s_g.adj_mode = ADJ;
            }
            __syncthreads();
        }
        const bool skip = ADJ != 0 && s_g.adj_mode != ADJ;
        if (skip && threadIdx.x == 0) atomicAdd(counter + 1, 1u);
        Counts6 cnt;
        cnt.zero();
        const int sampler = static_cast<int>(w.sampler);
        const bool any = !skip && (sampler == 0 ? s_g.W > 0 : s_g.Lambda > 0);
        if (any && SPT == 2 && (ADJ == kAdjHash || (ADJ == 0 && s_g.adj_mode == kAdjHash))) {
            for (uint32_t s = threadIdx.x; s < w.count; s += 2 * BLOCK) {
                // a lone last sample repeats its own id as the second, whose class is dropped
                const uint32_t s1 = s + BLOCK < w.count ? s + BLOCK : s;
                int c0, c1;
                batch_sample2_hash(s_g, sampler, w.seed, w.first_id + s, w.first_id + s1, c0, c1);
                cnt.add(c0);
                if (s1 != s) cnt.add(c1);
            }
        } else if (any) {
            for (uint32_t s = threadIdx.x; s < w.count; s += BLOCK) {
                if (ADJ != 0) {
                    cnt.add(batch_sample<ADJ>(s_g, sampler, w.seed, w.first_id + s));
                } else {
                    const int adj = s_g.adj_mode;
                    cnt.add(adj == kAdjVtab   ? batch_sample<kAdjVtab>(s_g, sampler, w.seed, w.first_id + s)
                            : adj == kAdjHash ? batch_sample<kAdjHash>(s_g, sampler, w.seed, w.first_id + s)
                                              : batch_sample<kAdjSearch>(s_g, sampler, w.seed, w.first_id + s));
                }
            }
        }
        if (threadIdx.x == 0) {
            if (s_item[at ^ 1] == kNone) {
                const uint32_t it = atomicAdd(counter, 1u);
                s_item[at ^ 1] = it;
                if (it < n_items) s_w[at ^ 1] = items[it];
            } else {
                asm volatile("cp.async.wait_all;" ::: "memory");
            }
        }
        // its barriers also publish the next item and free this one and s_g
        flush_counts<BLOCK>(cnt, sampler == 0 ? 6 : 4, hist + 6ull * w.slot);
    }
}

template <int BLOCK, int ADJ, int SPT>
static int launch_batch_t(const void *d_table, int32_t n_graphs, const ps_work *d_items, int64_t n_items,
                          uint64_t *d_hist, uint32_t *d_counter, const Tuning &t, cudaStream_t s) {
    int per_sm = t.blocks_per_sm;
    if (per_sm <= 0) {
        int occ = 0;
        PS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch<BLOCK, ADJ, SPT>, BLOCK, 0));
        per_sm = occ > 0 ? occ : 1;
    }
    int64_t blocks = (int64_t)sm_count_of_current_device() * per_sm;
    if (blocks > n_items) blocks = n_items;
    PS_CUDA_TRY(cudaMemsetAsync(d_counter, 0, 2 * sizeof(uint32_t), s));
    k_batch<BLOCK, ADJ, SPT><<<(unsigned)blocks, BLOCK, 0, s>>>(static_cast<const GraphDev *>(d_table), n_graphs,
                                                                d_items, n_items, d_hist, d_counter);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

template <int BLOCK, int ADJ>
static int launch_batch_s(const void *d_table, int32_t n_graphs, const ps_work *d_items, int64_t n_items,
                          uint64_t *d_hist, uint32_t *d_counter, const Tuning &t, cudaStream_t s) {
    return t.samples_per_thread >= 2
               ? launch_batch_t<BLOCK, ADJ, 2>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s)
               : launch_batch_t<BLOCK, ADJ, 1>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
}

template <int BLOCK>
static int launch_batch_b(const void *d_table, int32_t n_graphs, const ps_work *d_items, int64_t n_items,
                          uint64_t *d_hist, uint32_t *d_counter, const Tuning &t, cudaStream_t s) {
    switch (table_adjacency(d_table)) {
        case kAdjHash:
            return launch_batch_s<BLOCK, kAdjHash>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        case kAdjSearch:
            return launch_batch_s<BLOCK, kAdjSearch>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        case kAdjVtab:
            return launch_batch_s<BLOCK, kAdjVtab>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        default:
            return launch_batch_s<BLOCK, 0>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
    }
}

int launch_batch(const void *d_table, int32_t n_graphs, const ps_work *d_items, int64_t n_items,
                 uint64_t *d_hist, uint32_t *d_counter, const Tuning &t, cudaStream_t s) {
    if (n_items <= 0) return PS_OK;
    switch (t.block_size) {
        case 128: return launch_batch_b<128>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        case 256: return launch_batch_b<256>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        case 512: return launch_batch_b<512>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        case 1024: return launch_batch_b<1024>(d_table, n_graphs, d_items, n_items, d_hist, d_counter, t, s);
        default: return PS_ERR_ARG;
    }
}

}  // namespace ps
