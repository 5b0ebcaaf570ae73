// ps_order.cu -- ps_sample_3paths_ordered / ps_sample_centered_ordered: the
// samplers of Alg. 1 and Alg. 3 with the samples taken in the order of their
// edge draws.
//
// Every sample is independent (Claim 3.1: each draw is a fresh r), and the
// histograms are sums, so the order in which ids are classified changes no
// count.  In id order, consecutive samples draw unrelated edges: the guide
// entry, the prefix probe, the edge record and the row N(u) of every sample
// are separate random reads of HBM.  Here the ids of a chunk are first sorted
// by the leading bits of the 64-bit word their edge draw is made from (r grows
// with it); the sampling grid then walks the sorted ids, so the samples in
// flight at any time draw from a narrow band of consecutive edges, the samples
// of a warp mostly from a few edges, and those reads hit L1 and L2 or are one
// read for several lanes.  Only the second endpoint's row and the adjacency
// tests stay random.
//
// The sort is two kernels.  The word is uniform, so equal-width ranges of it
// hold nearly equal numbers of ids: the first kernel draws each id's word once
// and puts the ids into up to kOrderBuckets buckets of a fixed capacity (8
// standard deviations above the mean), reserving room tile by tile, with no
// counting pass before it.  The second sorts every bucket by the next
// kLocalBits bits in one block's shared memory and writes the ids out densely.
// Should a bucket ever run over, the sampling kernel takes the ids in their
// own order instead.
//
// The finer the order, the more the lanes of a warp share: on the 3M-vertex
// graph (115M edges, 2^27 ids) the 3-path sampling kernel took 10.6 / 9.4 / 8.5
// / 7.9 / 7.8 ms with the ids in order of 12 / 16 / 20 / 24 / 32 bits; on R-MAT
// 20 (2^24 ids) 710 / 568 / 527 / 522 us with 8 / 16 / 20 / 24.  This sort
// gives 24 and 21 bits; a sort by 16 bits in two passes of counting,
// offsets and scatter took 1.91 ms on the former, this one 1.70.
#include "ps_internal.h"
#include "ps_sample.cuh"

namespace ps {

constexpr int kOrderBuckets = 4096;              // of the first kernel, at most
// A bucket is one block of the second kernel: 1024 threads with up to 34 ids
// each.  (Smaller buckets for short chunks, a block of 512 with 18 each, left
// fewer SMs idle but cost the first kernel more: 3M ids 179 / 169 against 172 /
// 162 us on a 10M-edge graph.)
constexpr int kLocalThreads = 1024;
constexpr int kLocalItems = 34;
constexpr int kLocalBits = 12;                   // four counters per thread
constexpr int kMeanBits = 15;                    // ids per bucket: 2^14 to 2^15 on average
constexpr uint64_t kOrderMaxSorted = static_cast<uint64_t>(kOrderBuckets) << kMeanBits;  // ids sorted at once
constexpr int kOrderItems = 16;                  // ids per thread and tile of the first kernel
constexpr int kCursorStride = 8;                 // cursors in sectors of their own
// Scratch: the cursors and the overflow flag in a header, then per sample of a
// chunk its id (uint32) in the final order, and per place of the buckets an id
// (uint32) and its key's next bits (uint16): at most 10.4 bytes per sample.
constexpr size_t kOrderHeader = (1u << 20) + 1024;
constexpr size_t kOrderPerSample = 11;
static_assert((kOrderBuckets * kCursorStride + 1) * sizeof(uint32_t) <= kOrderHeader, "cursors and flag");
// By default (tuning draw_order 0) small graphs, whose records and rows stay
// in L2 anyway, and short chunks take the plain sampler: there the sort costs
// more than it saves.  The counts are the same either way.  Measured, ordered
// against plain, 3-path / centred (Chung-Lu; R-MAT crosses a little earlier):
//   2.5M edges: 2^23 ids 285 / 272 against 287 / 266 us;
//   5M edges: 2^21 ids 121 / 115 against 113 / 107, 2^22 184 / 174 against 204 / 192;
//   10M edges: 2^20 ids 101 / 102 against 83 / 82, 2^21 138 / 137 against 150 / 153;
//   40M edges: 2^20 ids 120 / 117 against 116 / 113, 2^24 971 / 777 against 1493 / 1506.
constexpr int64_t kOrderMinEdges = 1ll << 22;
static uint64_t order_min_chunk(int64_t m) { return m >= (1ll << 23) ? 1ull << 21 : 1ull << 22; }

// Buckets for kk ids (a power of two) and the room of each: the whole chunk
// in one bucket, or 8 standard deviations above the mean.
struct OrderPlan {
    int bits;          // log2 of the buckets
    uint32_t room;     // ids per bucket
};
static OrderPlan order_plan(uint64_t kk) {
    OrderPlan p{0, static_cast<uint32_t>(kk)};
    while (((kk - 1) >> kMeanBits) >> p.bits) p.bits++;
    if (p.bits) {
        const uint32_t mean = static_cast<uint32_t>((kk >> p.bits) + 1);
        uint32_t root = 1;
        while (root * root < mean) root++;
        p.room = mean + 8 * root + 64;
    }
    return p;
}

template <int THREADS>
struct PartSmem {
    uint32_t id[THREADS * kOrderItems];
    uint32_t key[THREADS * kOrderItems];
    uint32_t cnt[THREADS * 4];   // counts, then first tile-local places
    uint32_t base[THREADS * 4];  // place in the bucket of the tile-local place 0
    uint32_t warp[32];
};

// Exclusive prefix of v over the block (s_warp: 32 words of scratch).
template <int THREADS>
__device__ __forceinline__ uint32_t block_excl_sum(uint32_t v, uint32_t *s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t w = lane < THREADS / 32 ? s_warp[lane] : 0u;
    uint32_t before = lane < warp ? w : 0u;
    before = __reduce_add_sync(0xffffffffu, before);
    return before + x - v;
}

// The first kernel.  A tile of THREADS * kOrderItems ids per block and turn:
// each id's key is the high word its edge draw starts from; the tile is
// counting-sorted by bucket in shared memory, room for its runs is reserved
// with one atomic per bucket, and each run is written as one piece.  At most
// 4 * THREADS buckets.  2^27 ids into 4096 buckets take 1.22 ms, 0.47 of them
// the Philox rounds; the rest is the short runs (4 ids) of so many buckets --
// 2^24 ids into 512 buckets take 98 us.
template <int SAMPLER, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
k_order_partition(uint64_t kk, uint64_t seed, uint64_t first_id, int bits, uint32_t room, uint32_t *cursor,
                  uint32_t *spilled, uint32_t *__restrict__ ids, uint16_t *__restrict__ keys) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    PartSmem<THREADS> &S = *reinterpret_cast<PartSmem<THREADS> *>(s_raw);
    constexpr int kTile = THREADS * kOrderItems;
    const int t = threadIdx.x;
    const uint32_t buckets = 1u << bits;
    const int down = 32 - bits;  // 20..32
    for (uint64_t t0 = (uint64_t)blockIdx.x * kTile; t0 < kk; t0 += (uint64_t)gridDim.x * kTile) {
        const int n = kk - t0 < kTile ? static_cast<int>(kk - t0) : kTile;
#pragma unroll
        for (int q = 0; q < 4; q++) S.cnt[q * THREADS + t] = 0;
        __syncthreads();
        uint32_t key[kOrderItems];
        uint32_t rank2[kOrderItems / 2];
#pragma unroll
        for (int i = 0; i < kOrderItems; i++) {
            const int q = i * THREADS + t;
            key[i] = sample_block(seed, first_id + t0 + q, 0, SAMPLER).y;
            const uint32_t b = bits ? key[i] >> down : 0u;
            const uint32_t r = q < n ? atomicAdd(&S.cnt[b], 1u) : 0u;  // below kTile <= 2^16
            if (i & 1) rank2[i / 2] |= r << 16;
            else rank2[i / 2] = r;
        }
        __syncthreads();
        // thread t: buckets 4 t .. 4 t + 3
        uint32_t c[4], sum = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            c[q] = S.cnt[4 * t + q];
            sum += c[q];
        }
        uint32_t run = block_excl_sum<THREADS>(sum, S.warp);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t b = 4 * t + q;
            const uint32_t at = c[q] && b < buckets ? atomicAdd(cursor + b * kCursorStride, c[q]) : 0u;
            S.cnt[b] = run;
            S.base[b] = at - run;
            run += c[q];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kOrderItems; i++) {
            const int q = i * THREADS + t;
            if (q < n) {
                const uint32_t b = bits ? key[i] >> down : 0u;
                const uint32_t p = S.cnt[b] + ((rank2[i / 2] >> (16 * (i & 1))) & 0xffffu);
                S.id[p] = static_cast<uint32_t>(t0) + q;
                S.key[p] = key[i];
            }
        }
        __syncthreads();
        bool over = false;
        for (int p = t; p < n; p += THREADS) {
            const uint32_t k = S.key[p];
            const uint32_t b = bits ? k >> down : 0u;
            const uint32_t at = S.base[b] + p;
            if (at < room) {
                const uint32_t dst = b * room + at;
                ids[dst] = S.id[p];
                keys[dst] = static_cast<uint16_t>((k << bits) >> 16);
            } else {
                over = true;
            }
        }
        if (over) *spilled = 1u;
        __syncthreads();
    }
}

// The second kernel, a block per bucket: its ids by the next kLocalBits bits,
// behind the ids of the buckets before it.
struct LocalSmem {
    uint32_t id[kLocalThreads * kLocalItems];
    uint32_t cnt[1 << kLocalBits];
    uint32_t warp[32];
};
static_assert((1 << kLocalBits) == 4 * kLocalThreads, "four counters per thread");

__global__ void __launch_bounds__(kLocalThreads, 1)
k_order_local(uint32_t room, const uint32_t *__restrict__ cursor, const uint32_t *__restrict__ spilled,
              const uint32_t *__restrict__ ids, const uint16_t *__restrict__ keys, uint32_t *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    LocalSmem &S = *reinterpret_cast<LocalSmem *>(s_raw);
    if (*spilled) return;
    const int t = threadIdx.x;
    const uint32_t n = __ldg(cursor + blockIdx.x * kCursorStride);  // at most room
    ids += static_cast<size_t>(blockIdx.x) * room;
    keys += static_cast<size_t>(blockIdx.x) * room;
#pragma unroll
    for (int q = 0; q < 4; q++) S.cnt[q * kLocalThreads + t] = 0;
    // ids in the buckets before this one
    uint32_t before = 0;
    for (uint32_t b = t; b < blockIdx.x; b += kLocalThreads) before += __ldg(cursor + b * kCursorStride);
    __syncthreads();
    uint32_t place[kLocalItems];  // key << 16 | rank among the bucket's ids of that key
#pragma unroll
    for (int i = 0; i < kLocalItems; i++) {
        const uint32_t q = i * kLocalThreads + t;
        place[i] = q < n ? static_cast<uint32_t>(__ldg(keys + q)) >> (16 - kLocalBits) : 0u;
    }
#pragma unroll
    for (int i = 0; i < kLocalItems; i++)
        if (i * kLocalThreads + t < n) place[i] = place[i] << 16 | atomicAdd(&S.cnt[place[i]], 1u);
    before = __reduce_add_sync(0xffffffffu, before);
    __syncthreads();
    uint32_t c[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        c[q] = S.cnt[4 * t + q];
        sum += c[q];
    }
    uint32_t run = block_excl_sum<kLocalThreads>(sum, S.warp);
#pragma unroll
    for (int q = 0; q < 4; q++) {
        S.cnt[4 * t + q] = run;
        run += c[q];
    }
    __syncthreads();
    if ((t & 31) == 0) S.warp[t >> 5] = before;
#pragma unroll
    for (int i = 0; i < kLocalItems; i++) {
        const uint32_t q = i * kLocalThreads + t;
        if (q < n) S.id[S.cnt[place[i] >> 16] + (place[i] & 0xffffu)] = __ldg(ids + q);
    }
    __syncthreads();
    out += __reduce_add_sync(0xffffffffu, S.warp[t & 31]);
    for (uint32_t p = t; p < n; p += kLocalThreads) out[p] = S.id[p];
}

template <int SAMPLER, int BLOCK, int ADJ>
__global__ void __launch_bounds__(BLOCK, sample_min_blocks<BLOCK>())
k_sample_ordered(GraphDev g, uint64_t kk, uint64_t seed, uint64_t first_id, const uint32_t *__restrict__ ids,
                 const uint32_t *__restrict__ spilled, uint64_t *hist) {
    const bool sorted = __ldg(spilled) == 0u;
    Counts6 cnt;
    cnt.zero();
    const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
    for (uint64_t p = (uint64_t)blockIdx.x * BLOCK + threadIdx.x; p < kk; p += stride) {
        const uint64_t id = first_id + (sorted ? __ldg(ids + p) : p);
        cnt.add(SAMPLER == 0 ? sample_3path<ADJ>(g, seed, id) : sample_centred<ADJ>(g, seed, id));
    }
    flush_counts<BLOCK>(cnt, SAMPLER == 0 ? 6 : 4, hist);
}

template <int SAMPLER, int THREADS>
static int launch_partition(const ps_graph *g, uint64_t kk, uint64_t seed, uint64_t first_id, const OrderPlan &plan,
                            uint32_t *cursor, uint32_t *spilled, uint32_t *ids, uint16_t *keys, cudaStream_t s) {
    constexpr uint64_t kTile = THREADS * kOrderItems;
    const int smem = static_cast<int>(sizeof(PartSmem<THREADS>));
    PS_CUDA_TRY(cudaFuncSetAttribute(k_order_partition<SAMPLER, THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    const uint64_t tiles = (kk + kTile - 1) / kTile, full = (uint64_t)g->sm_count * (1024 / THREADS);
    k_order_partition<SAMPLER, THREADS><<<(unsigned)(tiles < full ? tiles : full), THREADS, smem, s>>>(
        kk, seed, first_id, plan.bits, plan.room, cursor, spilled, ids, keys);
    PS_LAUNCH_CHECK();
    return PS_OK;
}

template <int SAMPLER, int BLOCK, int ADJ>
static int ordered_t(const ps_graph *g, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *hist,
                     char *scratch, uint64_t chunk, cudaStream_t s) {
    uint32_t *cursor = reinterpret_cast<uint32_t *>(scratch);
    uint32_t *spilled = cursor + kOrderBuckets * kCursorStride;
    uint32_t *sorted = reinterpret_cast<uint32_t *>(scratch + kOrderHeader);
    int per_sm = g->tune.blocks_per_sm;
    if (per_sm <= 0) {
        int occ = 0;
        PS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sample_ordered<SAMPLER, BLOCK, ADJ>,
                                                                  BLOCK, 0));
        per_sm = occ > 0 ? occ : 1;
    }
    const uint64_t full = (uint64_t)g->sm_count * per_sm;
    while (k > 0) {
        const uint64_t kk = k < chunk ? k : chunk;
        if (kk < order_min_chunk(g->m) && g->tune.draw_order == 0) {
            const int rc = launch_sampler(g, SAMPLER, kk, seed, first_id, hist, s);
            if (rc) return rc;
        } else {
            const OrderPlan plan = order_plan(kk);
            const uint64_t places = static_cast<uint64_t>(plan.room) << plan.bits;
            uint32_t *ids = sorted + kk;
            uint16_t *keys = reinterpret_cast<uint16_t *>(ids + places);
            PS_CUDA_TRY(cudaMemsetAsync(cursor, 0, (kOrderBuckets * kCursorStride + 1) * sizeof(uint32_t), s));
            int rc;
            // up to 2048 buckets two smaller blocks per SM overlap their phases;
            // above, longer tiles keep the runs of a bucket from getting too short
            if (plan.bits <= 11) rc = launch_partition<SAMPLER, 512>(g, kk, seed, first_id, plan, cursor, spilled, ids, keys, s);
            else rc = launch_partition<SAMPLER, 1024>(g, kk, seed, first_id, plan, cursor, spilled, ids, keys, s);
            if (rc) return rc;
            const int smem = static_cast<int>(sizeof(LocalSmem));
            PS_CUDA_TRY(cudaFuncSetAttribute(k_order_local, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            k_order_local<<<1u << plan.bits, kLocalThreads, smem, s>>>(plan.room, cursor, spilled, ids, keys, sorted);
            PS_LAUNCH_CHECK();
            uint64_t blocks = (kk + BLOCK - 1) / BLOCK;
            if (blocks > full) blocks = full;
            k_sample_ordered<SAMPLER, BLOCK, ADJ><<<(unsigned)blocks, BLOCK, 0, s>>>(g->dev, kk, seed, first_id, sorted,
                                                                                    spilled, hist);
            PS_LAUNCH_CHECK();
        }
        k -= kk;
        first_id += kk;
    }
    return PS_OK;
}

template <int SAMPLER, int BLOCK>
static int ordered_b(const ps_graph *g, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *hist,
                     char *scratch, uint64_t chunk, cudaStream_t s) {
    switch (g->tune.adj_mode) {
        case kAdjVtab: return ordered_t<SAMPLER, BLOCK, kAdjVtab>(g, k, seed, first_id, hist, scratch, chunk, s);
        case kAdjHash: return ordered_t<SAMPLER, BLOCK, kAdjHash>(g, k, seed, first_id, hist, scratch, chunk, s);
        default: return ordered_t<SAMPLER, BLOCK, kAdjSearch>(g, k, seed, first_id, hist, scratch, chunk, s);
    }
}

template <int SAMPLER>
static int ordered_s(const ps_graph *g, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *hist,
                     char *scratch, uint64_t chunk, cudaStream_t s) {
    switch (g->tune.block_size) {
        case 128: return ordered_b<SAMPLER, 128>(g, k, seed, first_id, hist, scratch, chunk, s);
        case 256: return ordered_b<SAMPLER, 256>(g, k, seed, first_id, hist, scratch, chunk, s);
        case 512: return ordered_b<SAMPLER, 512>(g, k, seed, first_id, hist, scratch, chunk, s);
        case 1024: return ordered_b<SAMPLER, 1024>(g, k, seed, first_id, hist, scratch, chunk, s);
        default: return PS_ERR_ARG;
    }
}

size_t ordered_scratch_bytes(uint64_t k_chunk) {
    if (k_chunk == 0 || k_chunk > kOrderMaxChunk) return 0;
    return kOrderHeader + static_cast<size_t>(k_chunk) * kOrderPerSample;
}

bool order_never(const ps_graph *g) {
    return g->tune.draw_order < 0 || (g->tune.draw_order == 0 && g->m < kOrderMinEdges);
}

int launch_ordered(const ps_graph *g, int sampler, uint64_t k, uint64_t seed, uint64_t first_id, uint64_t *d_hist,
                   void *d_scratch, size_t scratch_bytes, cudaStream_t s) {
    if (scratch_bytes < ordered_scratch_bytes(1)) return PS_ERR_WORKSPACE;
    uint64_t chunk = (scratch_bytes - kOrderHeader) / kOrderPerSample;
    if (chunk > kOrderMaxSorted) chunk = kOrderMaxSorted;
    if (order_never(g)) return launch_sampler(g, sampler, k, seed, first_id, d_hist, s);
    char *scratch = static_cast<char *>(d_scratch);
    return sampler == 0 ? ordered_s<0>(g, k, seed, first_id, d_hist, scratch, chunk, s)
                        : ordered_s<1>(g, k, seed, first_id, d_hist, scratch, chunk, s);
}

}  // namespace ps
