// ps_sort.cu -- one pass of a stable LSD radix sort of (uint32 key, uint32
// value) pairs by a digit of up to 8 bits: used by the degree order (Section
// 4), the transposition that builds the edge table, and edge-list ingest.
//
// A pass counts the digits of every tile (digit-major), turns the counts into
// run offsets, and scatters: every tile ranks its items stably in shared
// memory -- each warp its own contiguous slice, warps in order -- and writes
// each digit's run contiguously.
//
// The lanes of a row that share a digit are found by one ballot per digit
// bit.  __match_any_sync takes longer the more different values a warp holds
// (with random 8-bit digits the scatter waited on it most of the time): 115M
// pairs took 0.79 ms per scatter with it.
//
// A sort by (value, key) -- the value as the more significant half -- can take
// its digits over the boundary of the two (`vshift`): 40 bits of an R-MAT 20
// edge in 5 passes instead of 6.
//
// Lists of up to kClusterItems items are sorted in one launch (at the end of
// this file).  Above that and up to kDirectTiles tiles every scatter block adds up the raw counts it needs
// itself, which saves the scan's launch (small graphs are bound by the number
// of launches); above that one look-back scan makes the offsets.
#include "ps_internal.h"

namespace ps {

constexpr int kSortBlock = 256;
constexpr int kSortItems = 14;
constexpr int kSortWarps = kSortBlock / 32;
constexpr int64_t kSortTile = static_cast<int64_t>(kSortBlock) * kSortItems;
constexpr int64_t kDirectTiles = 64;

int64_t sort_tiles(int64_t count) { return count > 0 ? (count + kSortTile - 1) / kSortTile : 1; }

int64_t sort_scan_tiles(int64_t count) {
    const int64_t tiles = sort_tiles(count);
    return tiles <= kDirectTiles ? 0 : (256 * tiles + kScanTile - 1) / kScanTile;
}

__device__ __forceinline__ int64_t live_count(int64_t count, const u64 *dcount) {
    return dcount && static_cast<int64_t>(*dcount) < count ? static_cast<int64_t>(*dcount) : count;
}

// A pass whose digit is zero in every key leaves the order as it is: with the
// largest key known on the device only, such passes are launched and skipped
// (the keys then stay where they are; the sort's user looks there).
__device__ __forceinline__ bool skip_pass(const u64 *max_key, int shift) {
    return max_key && shift > 0 && (*max_key >> shift) == 0;
}

// Digit of (key, value): the key's bits from `shift` on and, with CROSS, the
// value's lowest bits above them (vshift = the key's bits left of shift).
template <bool CROSS>
__device__ __forceinline__ uint32_t digit_of(uint32_t k, uint32_t v, int shift, int vshift, uint32_t mask) {
    return (CROSS ? (k >> shift) | (v << vshift) : k >> shift) & mask;
}

// Digit counts of every tile: counts[digit * tiles + tile].
template <bool CROSS>
__global__ void __launch_bounds__(kSortBlock)
k_sort_hist(int64_t count, const u64 *dcount, const u64 *max_key, const uint32_t *__restrict__ key, const uint32_t *__restrict__ val,
            int shift, int vshift, uint32_t mask, uint32_t *counts, int64_t tiles) {
    if (skip_pass(max_key, shift)) return;
    count = live_count(count, dcount);
    __shared__ uint32_t s_h[kSortWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < kSortWarps * 256; d += kSortBlock) (&s_h[0][0])[d] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * (32 * kSortItems) + lane;
    // all of a thread's keys in flight at once, then the counts
    uint32_t k[kSortItems];
#pragma unroll
    for (int q = 0; q < kSortItems; q++) {
        const int64_t idx = base + 32 * q;
        k[q] = idx < count ? digit_of<CROSS>(__ldg(key + idx), CROSS ? __ldg(val + idx) : 0u, shift, vshift, mask) : 0u;
    }
#pragma unroll
    for (int q = 0; q < kSortItems; q++)
        if (base + 32 * q < count) atomicAdd(&s_h[warp][k[q]], 1u);
    __syncthreads();
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) c += s_h[w][threadIdx.x];
    counts[(int64_t)threadIdx.x * tiles + blockIdx.x] = c;
}

struct LoadCounts {
    const uint32_t *p;
    __device__ uint32_t operator()(int64_t i) const { return p[i]; }
};
struct StoreCountsExcl {
    uint32_t *p;
    __device__ void operator()(int64_t i, uint32_t exc, uint32_t) const { p[i] = exc; }
};

// Exclusive prefix of v over the block's 256 threads (s_wsum: scratch).
__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t *s_wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_wsum[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; w++) before += (w < warp) ? s_wsum[w] : 0u;
    return before + x - v;
}

// Stable scatter of one tile.  Item order within a tile: warp w owns the w-th
// slice of 32 * kSortItems items and walks it in rows of 32 lanes, so (warp,
// row, lane) is index order.  Only the keys and their ranks stay in registers
// (values are read when placed), which keeps four blocks resident per SM: what
// bounds the kernel is the latency of the ranking, with ballots and shared
// memory each busy about half the time.  Ingest of 15.7M pairs, whole: three
// blocks of the same tile 1.81 ms, four 1.38, five with spills 1.58; tiles of
// 12, 14, 16 and 18 rows per warp 1.47, 1.36, 1.40 and 1.41 (shorter tiles write
// shorter runs).  Warp bases that include the digit's start and items moved
// as 8 bytes take two shared-memory accesses per item fewer: 1.45 -> 1.39 ms.
// (At 64 registers the crossing digits spill nothing, read values 24 bytes a
// thread above kDirectTiles tiles, indices up to 56.)
// DIRECT: `offsets` holds the raw counts; otherwise offsets[digit * tiles +
// tile] is where the tile's run of that digit starts.  VAL: values read from
// vin, or the items' indices, or read and part of the digit.
enum { kValRead = 0, kValIota = 1, kValCross = 2 };

template <int BITS, bool DIRECT, int VAL>
__global__ void __launch_bounds__(kSortBlock, 4)
k_sort_scatter(int64_t count, const u64 *dcount, const u64 *max_key, const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin,
               uint32_t *__restrict__ kout, uint32_t *__restrict__ vout, int shift, int vshift,
               const uint32_t *__restrict__ offsets, int64_t tiles) {
    constexpr uint32_t kMask = (1u << BITS) - 1;
    constexpr bool CROSS = VAL == kValCross;
    if (skip_pass(max_key, shift)) return;
    count = live_count(count, dcount);
    __shared__ uint2 s_item[kSortTile];          // (key, value) in the tile's order
    __shared__ uint32_t s_cnt[kSortWarps][256];  // per-warp counts, then per-warp bases
    __shared__ uint32_t s_glob[256];             // global start of the tile's run of each digit
    __shared__ uint32_t s_wsum[2 * kSortWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // positions within the tile are 32-bit; a tile past a run-time count is empty
    const int64_t tile0 = (int64_t)blockIdx.x * kSortTile;
    const int n_tile = static_cast<int>(count - tile0 < kSortTile ? count - tile0 : kSortTile);
    if (n_tile <= 0) return;
    kin += tile0;
    if (VAL != kValIota) vin += tile0;
    const int base = warp * (32 * kSortItems) + lane;
    for (int d = threadIdx.x; d < kSortWarps * 256; d += kSortBlock) (&s_cnt[0][0])[d] = 0u;
    uint32_t k[kSortItems];
#pragma unroll
    for (int q = 0; q < kSortItems; q++) k[q] = base + 32 * q < n_tile ? __ldg(kin + base + 32 * q) : 0u;
    if (DIRECT) {
        const uint32_t *mine = offsets + (int64_t)threadIdx.x * tiles;
        uint32_t before = 0, all = 0;
        for (int i = 0; i < static_cast<int>(tiles); i++) {
            const uint32_t c = __ldg(mine + i);
            before += i < static_cast<int>(blockIdx.x) ? c : 0u;
            all += c;
        }
        s_glob[threadIdx.x] = block_excl(all, s_wsum + kSortWarps) + before;
    } else {
        s_glob[threadIdx.x] = offsets[(int64_t)threadIdx.x * tiles + blockIdx.x];
    }
    __syncthreads();
    // stable rank of every item among its warp's items of the same digit
    // (below 32 * kSortItems, two to a register)
    static_assert(32 * kSortItems <= 65536 && kSortItems % 2 == 0, "ranks packed in 16 bits");
    uint32_t rank2[kSortItems / 2];
    // (a crossing digit reads the value here and again when placing it)
    auto digit_at = [&](int q) {
        const bool read = CROSS && base + 32 * q < n_tile;
        return digit_of<CROSS>(k[q], read ? __ldg(vin + base + 32 * q) : 0u, shift, vshift, kMask);
    };
#pragma unroll
    for (int q0 = 0; q0 < kSortItems; q0 += 2) {  // two rows' ballots in flight
        uint32_t peers[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t d = digit_at(q0 + h);
            peers[h] = __ballot_sync(0xffffffffu, base + 32 * (q0 + h) < n_tile);
#pragma unroll
            for (int b = 0; b < BITS; b++) {
                const bool bit = (d >> b) & 1u;
                const uint32_t v = __ballot_sync(0xffffffffu, bit);
                peers[h] &= bit ? v : ~v;
            }
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t d = digit_at(q0 + h), before = s_cnt[warp][d];
            const uint32_t r = before + __popc(peers[h] & lanemask_lt());
            if (h) rank2[q0 / 2] |= r << 16;
            else rank2[q0 / 2] = r;
            __syncwarp();
            if (base + 32 * (q0 + h) < n_tile && lane == __ffs(peers[h]) - 1) s_cnt[warp][d] = before + __popc(peers[h]);
            __syncwarp();
        }
    }
    __syncthreads();
    // thread t = digit t: the digits' tile-local starts (a block scan of the
    // digit totals), from there the warps' bases, and how far the tile's run of
    // the digit lies from its place in the tile
    {
        const int d = threadIdx.x;
        uint32_t c[kSortWarps], run = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; w++) {
            c[w] = s_cnt[w][d];
            run += c[w];
        }
        run = block_excl(run, s_wsum);
        s_glob[d] -= run;
#pragma unroll
        for (int w = 0; w < kSortWarps; w++) {
            s_cnt[w][d] = run;
            run += c[w];
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSortItems; q++) {
        if (base + 32 * q < n_tile) {
            const uint32_t v = VAL == kValIota ? static_cast<uint32_t>(tile0) + base + 32 * q : __ldg(vin + base + 32 * q);
            const uint32_t d = digit_of<CROSS>(k[q], v, shift, vshift, kMask);
            s_item[s_cnt[warp][d] + ((rank2[q / 2] >> (16 * (q & 1))) & 0xFFFFu)] = make_uint2(k[q], v);
        }
    }
    __syncthreads();
    for (int p = threadIdx.x; p < n_tile; p += kSortBlock) {
        const uint2 x = s_item[p];
        const uint32_t g = s_glob[digit_of<CROSS>(x.x, x.y, shift, vshift, kMask)] + p;
        kout[g] = x.x;
        vout[g] = x.y;
    }
}

template <int BITS, int VAL>
static void launch_scatter(const SortPass &p, int64_t tiles, cudaStream_t s) {
    const unsigned blocks = static_cast<unsigned>(tiles);
    if (tiles <= kDirectTiles)
        k_sort_scatter<BITS, true, VAL><<<blocks, kSortBlock, 0, s>>>(p.count, p.dcount, p.max_key, p.kin, p.vin, p.kout, p.vout,
                                                                      p.shift, p.vshift, p.counts, tiles);
    else
        k_sort_scatter<BITS, false, VAL><<<blocks, kSortBlock, 0, s>>>(p.count, p.dcount, p.max_key, p.kin, p.vin, p.kout, p.vout,
                                                                       p.shift, p.vshift, p.counts, tiles);
}

template <int BITS>
static void launch_scatter(const SortPass &p, int64_t tiles, cudaStream_t s) {
    if (p.vshift) launch_scatter<BITS, kValCross>(p, tiles, s);
    else if (p.vin) launch_scatter<BITS, kValRead>(p, tiles, s);
    else launch_scatter<BITS, kValIota>(p, tiles, s);
}

int sort_pass(const SortPass &p, const ScanState<uint32_t> &scan, cudaStream_t s) {
    if (p.count <= 0) return PS_OK;
    if (p.bits < 1 || p.bits > 8 || (p.vshift && !p.vin)) return PS_ERR_ARG;
    const int64_t tiles = sort_tiles(p.count);
    const int bits = (p.bits + 1) & ~1;  // the keys have no bits above the sort's last digit
    const uint32_t mask = (1u << bits) - 1u;
    if (p.vshift)
        k_sort_hist<true><<<static_cast<unsigned>(tiles), kSortBlock, 0, s>>>(p.count, p.dcount, p.max_key, p.kin, p.vin, p.shift,
                                                                              p.vshift, mask, p.counts, tiles);
    else
        k_sort_hist<false><<<static_cast<unsigned>(tiles), kSortBlock, 0, s>>>(p.count, p.dcount, p.max_key, p.kin, nullptr,
                                                                               p.shift, 0, mask, p.counts, tiles);
    PS_LAUNCH_CHECK();
    if (tiles > kDirectTiles) {
        k_scan<uint32_t, kScanBlock, kScanItems><<<static_cast<unsigned>(sort_scan_tiles(p.count)), kScanBlock, 0, s>>>(
            256 * tiles, scan, 0u, OpSum(), LoadCounts{p.counts}, StoreCountsExcl{p.counts});
        PS_LAUNCH_CHECK();
    }
    switch (bits) {  // ballots for the digit's own bits only
        case 2: launch_scatter<2>(p, tiles, s); break;
        case 4: launch_scatter<4>(p, tiles, s); break;
        case 6: launch_scatter<6>(p, tiles, s); break;
        default: launch_scatter<8>(p, tiles, s); break;
    }
    PS_LAUNCH_CHECK();
    return PS_OK;
}

// ------------------------------------------------------- one cluster's sort

// Lists of at most kClusterItems items: all passes in one launch of one
// cluster (up to 16 blocks of 1024, `rows` rows of 32 items per warp).  What
// bounds a small sort is the launches, not the items: a pass is two of them
// (counting, scattering), each waiting for the one before.  Here a pass is two
// cluster barriers.  Every block ranks its slice as the scatter above does,
// reads the other blocks' digit totals through distributed shared memory, and
// writes its runs -- ordered in shared memory first, so that they are written
// contiguously -- to the pass's output in global memory, from which the
// next pass reads past L1.  Measured: 6 passes over 40,000 pairs 58 us in 14
// launches -> 40 us in 2; with 8 blocks 43 us.
//
// The lanes of a row that share a digit are found by or-ing lane bits into a
// word per warp and digit: 7.2 us a pass against 8.0 with ballots.  (The
// scatter above, with four blocks per SM to hide the ballots, is the faster
// with them: 87 against 103 us for 15.7M pairs.)
constexpr int kClusterBlock = 1024;
constexpr int kClusterWarps = kClusterBlock / 32;
constexpr int kClusterRows = 8;
constexpr int kClusterBlocks = 16;
static_assert(kClusterItems == kClusterBlock * kClusterRows * kClusterBlocks, "the cluster's items");

struct ClusterSmem {
    uint2 item[kClusterBlock * kClusterRows];  // the block's slice in the pass's order: (key, value)
    uint32_t cnt[kClusterWarps][256];  // per-warp counts, then per-warp bases
    uint32_t mask[kClusterWarps][256];  // lanes of a row by digit
    uint32_t total[256];               // digit totals, read by the whole cluster
    uint32_t start[256];               // first slot of each digit in the block's slice
    uint32_t shift[256];               // from there to its place in the output
    uint32_t wsum[2][8];
};

struct ClusterSort {
    SortPass pass[kMaxPasses];
    int n, rows;
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Word of block `rank`'s shared memory that lies where `p` does in this one's.
__device__ __forceinline__ uint32_t cluster_load(const uint32_t *p, uint32_t rank) {
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), v;
    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// Exclusive prefix over the first 256 threads (v = 0 in the others).
__device__ __forceinline__ uint32_t excl256(uint32_t v, uint32_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31 && warp < 8) wsum[warp] = x;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int w = 0; w < 8; w++) before += (w < warp) ? wsum[w] : 0u;
    return before + x - v;
}

__device__ __forceinline__ uint32_t digit(const SortPass &p, uint32_t k, uint32_t v) {
    return ((k >> p.shift) | (p.vshift ? v << p.vshift : 0u)) & ((1u << p.bits) - 1u);
}

__global__ void __launch_bounds__(kClusterBlock, 1) k_sort_cluster(const __grid_constant__ ClusterSort job) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    ClusterSmem &S = *reinterpret_cast<ClusterSmem *>(s_raw);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rows = job.rows, blocks = static_cast<int>(gridDim.x), me = static_cast<int>(blockIdx.x);  // one cluster
    const int tile0 = me * rows * kClusterBlock;
    const int base = warp * (32 * rows) + lane;
    for (int i = 0; i < job.n; i++) {
        const SortPass &p = job.pass[i];
        if (skip_pass(p.max_key, p.shift)) continue;  // the same for the whole cluster
        const int left = static_cast<int>(live_count(p.count, p.dcount)) - tile0;
        const int n_tile = left < 0 ? 0 : (left < rows * kClusterBlock ? left : rows * kClusterBlock);
        uint32_t k[kClusterRows], v[kClusterRows], rank[kClusterRows];
#pragma unroll
        for (int q = 0; q < kClusterRows; q++) {
            const bool ok = q < rows && base + 32 * q < n_tile;
            const int64_t at = tile0 + base + 32 * q;
            k[q] = ok ? __ldcg(p.kin + at) : 0u;
            v[q] = ok ? (p.vin ? __ldcg(p.vin + at) : static_cast<uint32_t>(at)) : 0u;
        }
        for (int d = t; d < kClusterWarps * 256; d += kClusterBlock) (&S.cnt[0][0])[d] = (&S.mask[0][0])[d] = 0u;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kClusterRows; q++) {
            if (q < rows) {
                const uint32_t d = digit(p, k[q], v[q]);
                const bool ok = base + 32 * q < n_tile;
                if (ok) atomicOr(&S.mask[warp][d], 1u << lane);
                __syncwarp();
                const uint32_t peers = S.mask[warp][d], before = S.cnt[warp][d];
                rank[q] = before + __popc(peers & lanemask_lt());
                __syncwarp();
                if (ok && lane == __ffs(peers) - 1) {
                    S.cnt[warp][d] = before + __popc(peers);
                    S.mask[warp][d] = 0u;
                }
                __syncwarp();
            }
        }
        __syncthreads();
        uint32_t run = 0;
        if (t < 256) {
#pragma unroll
            for (int w = 0; w < kClusterWarps; w++) {
                const uint32_t c = S.cnt[w][t];
                S.cnt[w][t] = run;
                run += c;
            }
            S.total[t] = run;
        }
        const uint32_t start = excl256(run, S.wsum[0]);
        if (t < 256) S.start[t] = start;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kClusterRows; q++) {
            if (q < rows && base + 32 * q < n_tile) {
                const uint32_t d = digit(p, k[q], v[q]);
                S.item[S.start[d] + S.cnt[warp][d] + rank[q]] = make_uint2(k[q], v[q]);
            }
        }
        cluster_barrier();  // every block's totals are there, and its items read
        uint32_t all = 0, before = 0;
        if (t < 256) {
#pragma unroll
            for (int b = 0; b < kClusterBlocks; b++) {
                if (b < blocks) {
                    const uint32_t c = cluster_load(S.total + t, b);
                    before += b < me ? c : 0u;
                    all += c;
                }
            }
        }
        const uint32_t glob = excl256(all, S.wsum[1]) + before;
        if (t < 256) S.shift[t] = glob - start;
        __syncthreads();
        for (int at = t; at < n_tile; at += kClusterBlock) {
            const uint2 x = S.item[at];
            const uint32_t to = at + S.shift[digit(p, x.x, x.y)];
            p.kout[to] = x.x;
            p.vout[to] = x.y;
        }
        cluster_barrier();  // the output is there, and nobody reads the totals any more
    }
}

int sort_cluster(const SortPass *p, int n, cudaStream_t s, bool *done) {
    *done = true;
    if (n <= 0 || p[0].count <= 0) return PS_OK;
    if (n > kMaxPasses || p[0].count > kClusterItems) return PS_ERR_ARG;
    ClusterSort job{};
    for (int i = 0; i < n; i++) {
        if (p[i].count != p[0].count || p[i].bits < 1 || p[i].bits > 8 || (p[i].vshift && !p[i].vin)) return PS_ERR_ARG;
        job.pass[i] = p[i];
    }
    job.n = n;
    int blocks = 1;
    while (blocks < kClusterBlocks && static_cast<int64_t>(blocks) * kClusterBlock < p[0].count) blocks *= 2;
    job.rows = static_cast<int>((p[0].count + blocks * kClusterBlock - 1) / (blocks * kClusterBlock));
    const int smem = static_cast<int>(sizeof(ClusterSmem));
    PS_CUDA_TRY(cudaFuncSetAttribute(k_sort_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    PS_CUDA_TRY(cudaFuncSetAttribute(k_sort_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kClusterBlock);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // 16 blocks are more than every device is bound to place in one cluster
    // (a partition of one may be too small): the caller then sorts pass by pass
    if (cudaLaunchKernelEx(&cfg, k_sort_cluster, job) != cudaSuccess) {
        cudaGetLastError();
        *done = false;
        return PS_OK;
    }
    PS_LAUNCH_CHECK();
    return PS_OK;
}

}  // namespace ps
