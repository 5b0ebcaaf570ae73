// ps_sample.cu -- ps_sample_3paths / ps_sample_centered: persistent
// grid-stride kernels over sample ids, each thread drawing and classifying
// samples independently and counting classes in registers.
#include "ps_internal.h"
#include "ps_sample.cuh"

namespace ps {

template <int SAMPLER, int BLOCK, int ADJ>
__global__ void __launch_bounds__(BLOCK, sample_min_blocks<BLOCK>())
k_sample(GraphDev g, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *hist) {
    Counts6 cnt;
    cnt.zero();
    const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
    for (uint64_t s = (uint64_t)blockIdx.x * BLOCK + threadIdx.x; s < k; s += stride) {
        const uint64_t id = first_id + s;
        cnt.add(SAMPLER == 0 ? sample_3path<ADJ>(g, seed, id) : sample_centred<ADJ>(g, seed, id));
    }
    flush_counts<BLOCK>(cnt, SAMPLER == 0 ? 6 : 4, hist);
}

// Both samplers in one launch, ids first_id .. of each: the threads that run out
// of 3-path samples go on with centred ones, so the second kernel's launch and
// the first one's last wave cost nothing, and short calls (fewer samples than
// resident threads) draw both kinds side by side.  Adaptive run on a 1M-edge
// graph, nine looks of 2^16 to 2^24 samples: 1248 -> 1182 us.
template <int BLOCK, int ADJ>
__global__ void __launch_bounds__(BLOCK, sample_min_blocks<BLOCK>())
k_sample_both(GraphDev g, uint64_t k3, uint64_t kc, uint64_t seed, uint64_t first_id, uint64_t *hist6, uint64_t *hist4) {
    Counts6 cnt;
    cnt.zero();
    const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
    uint64_t s = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
    for (; s < k3; s += stride) cnt.add(sample_3path<ADJ>(g, seed, first_id + s));
    flush_counts<BLOCK>(cnt, 6, hist6);
    cnt.zero();
    for (s -= k3; s < kc; s += stride) cnt.add(sample_centred<ADJ>(g, seed, first_id + s));
    flush_counts<BLOCK>(cnt, 4, hist4);
}

// From these many edges the plain samplers run 768 threads per SM instead of
// 1024 (in blocks that divide it): where the records, rows and tables no longer
// stay in L2, a quarter more threads evict more of each other's lines than the
// latency they hide is worth.  Ids drawn in order (ps_order.cu) share their
// lines and keep 1024.  2^23 samples, 1024 / 768 threads, 3-path and centred:
//   filter   7.7M edges 541 / 522 and 380 / 416 us, 10M 677 / 628 and 579 / 543,
//            R-MAT 20 (15.7M) 812 / 786 and 608 / 566, 117M 1261 / 1176 and 1009 / 974;
//   tables   15.7M 953 / 992 and 1002 / 957, 10M centred 856 / 823, 7.7M centred
//            692 / 734; 2^22 3-path, unskewed graphs of 20M: 719 / 660, 700 / 660;
//   search   47M 2093 / 2107 and 1217 / 1342, 64M 2957 / 2897 and 2009 / 1985.
// On clustered graphs of that size the filter's centred samples wait for their
// confirmed hits and would rather keep 1024 (2^22 on random cliques over
// Chung-Lu graphs of 21M and 102M edges 364 / 383 and 399 / 405 us).
template <int ADJ>
static int64_t few_threads_from(int sampler) {
    if (ADJ == kAdjSearch) return int64_t{3} << 24;
    return ADJ == kAdjVtab && sampler == 0 ? int64_t{1} << 24 : int64_t{1} << 23;
}

template <int BLOCK, int ADJ>
static int resident_blocks(const ps_graph *g, int sampler, int occupancy) {
    if (768 % BLOCK == 0 && occupancy > 768 / BLOCK && g->m >= few_threads_from<ADJ>(sampler)) return 768 / BLOCK;
    return occupancy > 0 ? occupancy : 1;
}

template <int SAMPLER, int BLOCK, int ADJ>
static int launch_t(const ps_graph *g, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *hist,
                    cudaStream_t s) {
    int per_sm = g->tune.blocks_per_sm;
    if (per_sm <= 0) {
        int occ = 0;
        PS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sample<SAMPLER, BLOCK, ADJ>, BLOCK, 0));
        per_sm = resident_blocks<BLOCK, ADJ>(g, SAMPLER, occ);
    }
    const uint64_t full = (uint64_t)g->sm_count * per_sm;
    // per-thread counters are 32-bit: keep every thread under 2^30 samples per launch
    const uint64_t max_chunk = full * BLOCK * (1ull << 30);
    while (k > 0) {
        const uint64_t kk = k < max_chunk ? k : max_chunk;
        uint64_t blocks = (kk + BLOCK - 1) / BLOCK;
        if (blocks > full) blocks = full;
        k_sample<SAMPLER, BLOCK, ADJ><<<(unsigned)blocks, BLOCK, 0, s>>>(g->dev, kk, seed, first_id, hist);
        PS_LAUNCH_CHECK();
        k -= kk;
        first_id += kk;
    }
    return PS_OK;
}

template <int BLOCK>
static int launch_b(const ps_graph *g, int sampler, uint64_t k, uint64_t seed, uint64_t first_id,
                    uint64_t *hist, cudaStream_t s) {
    if (g->tune.adj_mode == kAdjVtab)
        return sampler == 0 ? launch_t<0, BLOCK, kAdjVtab>(g, k, seed, first_id, hist, s)
                            : launch_t<1, BLOCK, kAdjVtab>(g, k, seed, first_id, hist, s);
    if (g->tune.adj_mode == kAdjHash)
        return sampler == 0 ? launch_t<0, BLOCK, kAdjHash>(g, k, seed, first_id, hist, s)
                            : launch_t<1, BLOCK, kAdjHash>(g, k, seed, first_id, hist, s);
    return sampler == 0 ? launch_t<0, BLOCK, kAdjSearch>(g, k, seed, first_id, hist, s)
                        : launch_t<1, BLOCK, kAdjSearch>(g, k, seed, first_id, hist, s);
}

template <int BLOCK, int ADJ>
static int launch_both_t(const ps_graph *g, uint64_t k3, uint64_t kc, uint64_t seed, uint64_t first_id, uint64_t *hist6,
                         uint64_t *hist4, cudaStream_t s) {
    int per_sm = g->tune.blocks_per_sm;
    if (per_sm <= 0) {
        int occ = 0;
        PS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sample_both<BLOCK, ADJ>, BLOCK, 0));
        per_sm = resident_blocks<BLOCK, ADJ>(g, 1, occ);
    }
    const uint64_t full = (uint64_t)g->sm_count * per_sm;
    uint64_t blocks = (k3 + kc + BLOCK - 1) / BLOCK;
    if (blocks > full) blocks = full;
    k_sample_both<BLOCK, ADJ><<<(unsigned)blocks, BLOCK, 0, s>>>(g->dev, k3, kc, seed, first_id, hist6, hist4);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

template <int BLOCK>
static int launch_both_b(const ps_graph *g, uint64_t k3, uint64_t kc, uint64_t seed, uint64_t first_id, uint64_t *hist6,
                         uint64_t *hist4, cudaStream_t s) {
    if (g->tune.adj_mode == kAdjVtab) return launch_both_t<BLOCK, kAdjVtab>(g, k3, kc, seed, first_id, hist6, hist4, s);
    if (g->tune.adj_mode == kAdjHash) return launch_both_t<BLOCK, kAdjHash>(g, k3, kc, seed, first_id, hist6, hist4, s);
    return launch_both_t<BLOCK, kAdjSearch>(g, k3, kc, seed, first_id, hist6, hist4, s);
}

int launch_sampler(const ps_graph *g, int sampler, uint64_t k, uint64_t seed, uint64_t first_id,
                   uint64_t *d_hist, cudaStream_t s) {
    switch (g->tune.block_size) {
        case 128: return launch_b<128>(g, sampler, k, seed, first_id, d_hist, s);
        case 256: return launch_b<256>(g, sampler, k, seed, first_id, d_hist, s);
        case 512: return launch_b<512>(g, sampler, k, seed, first_id, d_hist, s);
        case 1024: return launch_b<1024>(g, sampler, k, seed, first_id, d_hist, s);
        default: return PS_ERR_ARG;
    }
}

int launch_samplers(const ps_graph *g, uint64_t k3, uint64_t *d_hist6, uint64_t kc, uint64_t *d_hist4, uint64_t seed,
                    uint64_t first_id, cudaStream_t s) {
    if (g->stats.W == 0) k3 = 0;
    if (g->stats.Lambda == 0) kc = 0;
    // one launch where there is something of both; beyond 2^30 samples apiece
    // the counters of a thread might overflow, so those go in chunks
    if (k3 > 0 && kc > 0 && k3 < (1ull << 30) && kc < (1ull << 30)) {
        switch (g->tune.block_size) {
            case 128: return launch_both_b<128>(g, k3, kc, seed, first_id, d_hist6, d_hist4, s);
            case 256: return launch_both_b<256>(g, k3, kc, seed, first_id, d_hist6, d_hist4, s);
            case 512: return launch_both_b<512>(g, k3, kc, seed, first_id, d_hist6, d_hist4, s);
            case 1024: return launch_both_b<1024>(g, k3, kc, seed, first_id, d_hist6, d_hist4, s);
            default: return PS_ERR_ARG;
        }
    }
    int rc = k3 > 0 ? launch_sampler(g, 0, k3, seed, first_id, d_hist6, s) : PS_OK;
    if (rc == PS_OK && kc > 0) rc = launch_sampler(g, 1, kc, seed, first_id, d_hist4, s);
    return rc;
}

}  // namespace ps
