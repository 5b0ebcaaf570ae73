// ps_load.cu -- ps_load_csr: validation of the input graph (Section 2), the
// degree order of Section 4 made the integer order by relabelling, sorted
// adjacency lists, and the edge table (u < v, row-major) with the position of
// each edge in both endpoint lists.
#include <algorithm>
#include <climits>
#include <utility>

#include "ps_internal.h"

namespace ps {

// ------------------------------------------------------------------ degrees

__global__ void k_degrees(int64_t n, int64_t nnz, const int64_t *__restrict__ off,
                          uint32_t *__restrict__ keys, u64 *status) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 == 0) {
        if (ldg_i64(off) != 0 || ldg_i64(off + n) != nnz) raise_flag(status, F_ARG);
    }
    uint32_t dmax = 0;
    bool bad = false, longrow = false;
    for (int64_t v = t0; v < n; v += stride) {
        const int64_t a = ldg_i64(off + v), b = ldg_i64(off + v + 1);
        int64_t d = b - a;
        if (d < 0 || a < 0 || b > nnz) {
            bad = true;
            d = 0;
        }
        if (d > n - 1) longrow = true;  // cannot be a simple row; the load ends early
        keys[v] = static_cast<uint32_t>(d);
        dmax = max(dmax, static_cast<uint32_t>(d));
    }
    if (bad) raise_flag(status, F_ARG);
    if (longrow) raise_flag(status, F_NOT_SIMPLE);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_down_sync(0xffffffffu, dmax, o));
    if ((threadIdx.x & 31) == 0 && dmax)
        atomicMax(reinterpret_cast<unsigned long long *>(status + ST_DMAX), (unsigned long long)dmax);
}

// F_ARG for a column out of range (when the rows themselves are not walked).
__global__ void __launch_bounds__(256) k_check_columns(int64_t n, int64_t nnz, const int32_t *__restrict__ col, u64 *status) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += stride) {
        const int32_t c = ldg_i32(col + i);
        bad |= c < 0 || c >= n;
    }
    if (bad) raise_flag(status, F_ARG);
}

// The sorted (degree, vertex) pairs, position r = label r: rank[v] = the label
// of v, inv[r] = v, dnew[r] = its degree, lowcnt[r] = 0.  The pairs are in the
// first or the second buffers, by how many sort passes the largest degree
// needed.  Also the first label whose degree
// exceeds each row-length limit; N_1 = sum_v C(d_v, 3) (128-bit); and the
// number of hub rows: the top `hub_cap` labels whose degree is at least
// `hub_min`.
__global__ void __launch_bounds__(256)
k_rank(int64_t n, int bits, const uint32_t *__restrict__ k0, const uint32_t *__restrict__ v0,
       const uint32_t *__restrict__ k1, const uint32_t *__restrict__ v1, int32_t *rank, uint32_t *inv, int32_t *dnew,
       int32_t *lowcnt, uint32_t tier_b_end, int64_t hub_cap, int64_t hub_min, u64 *status) {
    const uint32_t lim[5] = {0, kTierA, tier_b_end, kTierC, kLongRow};
    const int slot[5] = {ST_TIER, ST_TIER + 1, ST_TIER + 2, ST_TIER + 3, ST_LONG};
    bool second = true;  // the first pass moves the pairs to the second buffers, and so on
    for (int shift = 8; shift < bits && (status[ST_DMAX] >> shift) != 0; shift += 8) second = !second;
    const uint32_t *skeys = second ? k1 : k0, *svals = second ? v1 : v0;
    uint64_t lo = 0, hi = 0;
    unsigned long long hubs = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride) {
        const uint32_t d = __ldg(skeys + r);
        const uint32_t v = __ldg(svals + r);
        rank[v] = static_cast<int32_t>(r);
        inv[r] = v;
        dnew[r] = static_cast<int32_t>(d);
        lowcnt[r] = 0;
        const uint32_t before = r ? __ldg(skeys + r - 1) : 0u;
#pragma unroll
        for (int t = 0; t < 5; t++) {
            if (d > lim[t] && (r == 0 || before <= lim[t])) status[slot[t]] = static_cast<u64>(r);
            if (r == n - 1 && d <= lim[t]) status[slot[t]] = static_cast<u64>(n);
        }
        if (r == n - 1) status[ST_TIER + 4] = static_cast<u64>(n);
        add_stars(lo, hi, d);
        hubs += r >= n - hub_cap && d >= static_cast<uint64_t>(hub_min);
    }
    warp_add128(lo, hi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) hubs += __shfl_down_sync(0xffffffffu, hubs, o);
    if ((threadIdx.x & 31) == 0) {
        if (lo | hi) atomic_add128(status + ST_N1_LO, lo, hi);
        if (hubs) atomicAdd(reinterpret_cast<unsigned long long *>(status + ST_HUBS), hubs);
    }
}

struct LoadDeg {
    const int32_t *d;
    __device__ int64_t operator()(int64_t i) const { return d[i]; }
};
struct StoreOffsets {
    int64_t *off;
    int64_t n;
    __device__ void operator()(int64_t i, int64_t exc, int64_t inc) const {
        off[i] = exc;
        if (i == n - 1) off[n] = inc;
    }
};

// ------------------------------------------------------- row relabel + sort

struct RowIn {
    const int64_t *off;
    const int32_t *col;
    const uint32_t *inv;   // row r of the new graph is input vertex inv[r]
    const int32_t *rank;
    const int64_t *coff;
    int32_t *ccol;
    int32_t *lowcnt;
    int64_t n;
    u64 *status;
};

// Relabelled neighbour, with range and self-loop checks (the bad column is
// replaced by the row itself so no access leaves the arrays).
__device__ __forceinline__ int32_t relabel(const RowIn &R, int64_t i, uint32_t v, int32_t r,
                                          bool &bad_arg, bool &self) {
    const int32_t c = ldg_i32(R.col + i);
    if (c < 0 || c >= R.n) {
        bad_arg = true;
        return r;
    }
    if (c == static_cast<int32_t>(v)) self = true;
    return ldg_i32(R.rank + c);
}

__device__ __forceinline__ void report(const RowIn &R, bool bad_arg, bool not_simple) {
    if (bad_arg) raise_flag(R.status, F_ARG);
    if (not_simple) raise_flag(R.status, F_NOT_SIMPLE);
}

// 32 / G rows of at most G entries from row r on, G lanes each, bitonic
// network in registers.
template <int G>
__device__ __forceinline__ void sort_rows_short(const RowIn &R, int64_t r, int64_t r_end, bool &bad, bool &nsimple) {
    const int lane = threadIdx.x & 31, at = lane % G;
    r += lane / G;
    int64_t dst = 0;
    int d = 0;
    int32_t x = INT_MAX;
    if (r < r_end) {
        const uint32_t v = R.inv[r];
        dst = R.coff[r];
        d = static_cast<int>(R.coff[r + 1] - dst);
        if (at < d) x = relabel(R, ldg_i64(R.off + v) + at, v, static_cast<int32_t>(r), bad, nsimple);
    }
#pragma unroll
    for (int k = 2; k <= G; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const int32_t y = __shfl_xor_sync(0xffffffffu, x, j);
            const bool asc = (at & k) == 0, lower = (at & j) == 0;
            x = (lower == asc) ? min(x, y) : max(x, y);
        }
    }
    const int32_t nx = __shfl_down_sync(0xffffffffu, x, 1);
    if (at + 1 < d && nx == x) nsimple = true;
    const uint32_t below = __ballot_sync(0xffffffffu, at < d && x < static_cast<int32_t>(r)) >> (lane - at);
    if (at < d) R.ccol[dst + at] = x;
    if (at == 0 && r < r_end) R.lowcnt[r] = __popc(G == 32 ? below : below & ((1u << (G & 31)) - 1u));
}

// Tier A: rows of 1..32 entries.  What bounds a row is the chain inv -> offset
// -> column -> label.  With more rows than warps a warp takes four rows, which
// in degree order are about as long as each other, and rows of at most 8 or 16
// entries share its lanes: R-MAT 20 97 -> 50 us, 150k rows 25 -> 17 us, the
// 3M-vertex graph, whose rows are longer, 390 -> 383 us.  (40 registers, six
// blocks per SM: 48 registers were 20 us slower on R-MAT 20.)  With fewer rows
// a warp each.
__global__ void __launch_bounds__(256, 6) k_sort_tier_a(RowIn R) {
    const int64_t r0 = static_cast<int64_t>(R.status[ST_TIER + 0]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_TIER + 1]);
    const int64_t nw = (int64_t)gridDim.x * blockDim.x / 32;
    const int64_t group = r1 - r0 > nw ? 4 : 1;
    bool bad = false, nsimple = false;
    for (int64_t r = r0 + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32 * group; r < r1; r += group * nw) {
        const int64_t end = min(r + group, r1);
        const int64_t longest = R.coff[end] - R.coff[end - 1];
        if (longest <= 8) {
            sort_rows_short<8>(R, r, end, bad, nsimple);
        } else if (longest <= 16) {
            for (int64_t q = r; q < end; q += 2) sort_rows_short<16>(R, q, end, bad, nsimple);
        } else {
            for (int64_t q = r; q < end; q++) sort_rows_short<32>(R, q, end, bad, nsimple);
        }
    }
    report(R, bad, nsimple);
}

// Bitonic sort, ascending, of N = E * THREADS keys held E per thread in
// blocked order (thread t holds keys t*E .. t*E + E - 1).  A compare-exchange
// stage whose partner key sits in the same thread works on registers, one
// whose partner sits in the same warp exchanges by shuffle, and only the
// stages that cross warps go through shared memory (smem: N keys; unused
// when THREADS == 32).  Fully unrolled, so every register index is static.
template <int E, int THREADS>
__device__ __forceinline__ void bitonic_blocked(int32_t (&x)[E], int32_t *smem) {
    constexpr int N = E * THREADS;
    const int lane = threadIdx.x & 31;
    const int base = (THREADS == 32 ? lane : static_cast<int>(threadIdx.x)) * E;
#pragma unroll
    for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j < E) {
#pragma unroll
                for (int i = 0; i < E; i++)
                    if ((i & j) == 0) {
                        const bool asc = ((base | i) & k) == 0;
                        const int32_t a = x[i], b = x[i | j];
                        x[i] = asc ? min(a, b) : max(a, b);
                        x[i | j] = asc ? max(a, b) : min(a, b);
                    }
            } else if (j < 32 * E) {
                const int lm = j / E;
                const bool keep_min = ((lane & lm) == 0) == ((base & k) == 0);
#pragma unroll
                for (int i = 0; i < E; i++) {
                    const int32_t y = __shfl_xor_sync(0xffffffffu, x[i], lm);
                    x[i] = keep_min ? min(x[i], y) : max(x[i], y);
                }
            } else if (THREADS > 32) {
                __syncthreads();  // the previous stage's readers are done
#pragma unroll
                for (int i = 0; i < E; i++) smem[base + i] = x[i];
                __syncthreads();
                const bool keep_min = ((base & j) == 0) == ((base & k) == 0);
#pragma unroll
                for (int i = 0; i < E; i++) {
                    const int32_t y = smem[(base + i) ^ j];
                    x[i] = keep_min ? min(x[i], y) : max(x[i], y);
                }
            }
        }
    }
}

// One row of tier B with P = 32 * E slots: relabel, sort in registers, write
// the row and its lower count.
template <int E>
__device__ __forceinline__ void sort_row_warp(const RowIn &R, int64_t r, uint32_t v, int64_t o, int d,
                                              bool &bad, bool &nsimple) {
    const int lane = threadIdx.x & 31;
    int32_t x[E];
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = lane * E + i;
        x[i] = idx < d ? relabel(R, o + idx, v, static_cast<int32_t>(r), bad, nsimple) : INT_MAX;
    }
    bitonic_blocked<E, 32>(x, nullptr);
    const int32_t after = __shfl_down_sync(0xffffffffu, x[0], 1);  // first key of the next lane
    int32_t *dst = R.ccol + R.coff[r];
    int low = 0;
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = lane * E + i;
        if (idx < d) {
            dst[idx] = x[i];
            low += x[i] < static_cast<int32_t>(r);
            const int32_t nx = (i + 1 < E) ? x[i + 1] : after;
            if (idx + 1 < d && nx == x[i]) nsimple = true;
        }
    }
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) low += __shfl_down_sync(0xffffffffu, low, o2);
    if (lane == 0) R.lowcnt[r] = low;
}

// Tier B: rows of 33..1024 (or 512, tier_b) entries, one warp, bitonic network in registers,
// in two kernels: rows up to kLongRow entries (two or four keys per lane)
// at 32 registers and full occupancy, the longer ones capped at 64
// registers (four blocks per SM beat the spill-free 105-register build; the
// same holds for tier C at three blocks).
__global__ void __launch_bounds__(256, 8) k_sort_tier_b(RowIn R) {
    const int64_t r0 = static_cast<int64_t>(R.status[ST_TIER + 1]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_LONG]);
    const int64_t nw = (int64_t)gridDim.x * blockDim.x / 32;
    bool bad = false, nsimple = false;
    for (int64_t r = r0 + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; r < r1; r += nw) {
        const uint32_t v = R.inv[r];
        const int64_t o = ldg_i64(R.off + v);
        const int d = static_cast<int>(ldg_i64(R.off + v + 1) - o);
        if (d <= 64) sort_row_warp<2>(R, r, v, o, d, bad, nsimple);
        else sort_row_warp<4>(R, r, v, o, d, bad, nsimple);
    }
    report(R, bad, nsimple);
}
static_assert(kLongRow == 128 && kLongRow < kTierB, "tier B's first kernel sorts rows of at most 4 keys per lane");

__global__ void __launch_bounds__(256, 4) k_sort_tier_b2(RowIn R) {
    const int64_t r0 = static_cast<int64_t>(R.status[ST_LONG]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_TIER + 2]);
    const int64_t nw = (int64_t)gridDim.x * blockDim.x / 32;
    bool bad = false, nsimple = false;
    for (int64_t r = r0 + ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; r < r1; r += nw) {
        const uint32_t v = R.inv[r];
        const int64_t o = ldg_i64(R.off + v);
        const int d = static_cast<int>(ldg_i64(R.off + v + 1) - o);
        if (d <= 256) sort_row_warp<8>(R, r, v, o, d, bad, nsimple);
        else if (d <= 512) sort_row_warp<16>(R, r, v, o, d, bad, nsimple);
        else sort_row_warp<32>(R, r, v, o, d, bad, nsimple);
    }
    report(R, bad, nsimple);
}

// Tier C: rows from there to 4096 entries, one block of 512, bitonic network in
// registers with the cross-warp stages in shared memory (16 KB, several
// blocks per SM).
template <int E>
__device__ __forceinline__ void sort_row_block(const RowIn &R, int64_t r, uint32_t v, int64_t o, int d,
                                               int32_t *smem, int *s_low, bool &bad, bool &nsimple) {
    constexpr int kThreads = 512;
    const int base = static_cast<int>(threadIdx.x) * E;
    int32_t x[E];
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = base + i;
        x[i] = idx < d ? relabel(R, o + idx, v, static_cast<int32_t>(r), bad, nsimple) : INT_MAX;
    }
    if (threadIdx.x == 0) *s_low = 0;
    bitonic_blocked<E, kThreads>(x, smem);
    __syncthreads();  // the sort's last shared-memory readers are done
#pragma unroll
    for (int i = 0; i < E; i++) smem[base + i] = x[i];
    __syncthreads();
    int32_t *dst = R.ccol + R.coff[r];
    int low = 0;
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = base + i;
        if (idx < d) {
            dst[idx] = x[i];
            low += x[i] < static_cast<int32_t>(r);
            if (idx + 1 < d && smem[idx + 1] == x[i]) nsimple = true;
        }
    }
#pragma unroll
    for (int o2 = 16; o2 > 0; o2 >>= 1) low += __shfl_down_sync(0xffffffffu, low, o2);
    if ((threadIdx.x & 31) == 0) atomicAdd(s_low, low);
    __syncthreads();
    if (threadIdx.x == 0) R.lowcnt[r] = *s_low;
    __syncthreads();  // s_low and smem are free for the next row
}

// Bucket of label x for the bucketed row sort: 256 buckets in label order,
// fine near the top labels and coarse far from them -- a float-like code
// (exponent and three mantissa bits) of the distance n - 1 - x from the
// top.  In degree order a long row's neighbours crowd the top labels (their
// density falls roughly as a power of that distance), which this spreads
// evenly: on the 3M-vertex graph a 1025..4096-entry row's largest bucket
// holds at most ~100 entries, against ~900 for the top 8 label bits.
__device__ __forceinline__ int row_bucket(int32_t x, int32_t top) {
    const uint32_t y1 = static_cast<uint32_t>(top - x) + 1u;  // 1 .. n
    const int e = 31 - __clz(y1);
    const uint32_t m = e >= 3 ? (y1 >> (e - 3)) & 7u : (y1 << (3 - e)) & 7u;
    return 255 - (e * 8 + static_cast<int>(m));
}

// One warp sorts the run p[0, s) of shared memory (s <= 32 E).
template <int E>
__device__ __forceinline__ void sort_run_warp(int32_t *p, int s) {
    const int lane = threadIdx.x & 31;
    int32_t x[E];
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = lane * E + i;
        x[i] = idx < s ? p[idx] : INT_MAX;
    }
    bitonic_blocked<E, 32>(x, nullptr);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int idx = lane * E + i;
        if (idx < s) p[idx] = x[i];
    }
}

// Tier C by buckets: the row relabelled into shared memory, counted and
// scattered into its 256 buckets (row_bucket), each bucket sorted by one
// warp, the row written out.  A row with a bucket above 256 entries (none on
// the benchmark graphs) takes the block-wide bitonic sort above instead.
constexpr int kBucketRun = 256;

__global__ void __launch_bounds__(512, 3) k_sort_tier_c(RowIn R) {
    __shared__ int32_t s_a[kTierC];
    __shared__ int32_t s_b[kTierC];
    __shared__ uint32_t s_cnt[256], s_start[257];
    __shared__ int s_low, s_big;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t r0 = static_cast<int64_t>(R.status[ST_TIER + 2]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_TIER + 3]);
    const int32_t top = static_cast<int32_t>(R.n - 1);
    bool bad = false, nsimple = false;
    for (int64_t r = r0 + blockIdx.x; r < r1; r += gridDim.x) {
        const uint32_t v = R.inv[r];
        const int64_t o = ldg_i64(R.off + v);
        const int d = static_cast<int>(ldg_i64(R.off + v + 1) - o);
        if (t < 256) s_cnt[t] = 0;
        if (t == 0) {
            s_low = 0;
            s_big = 0;
        }
        __syncthreads();
        for (int i = t; i < d; i += 512) {
            const int32_t x = relabel(R, o + i, v, static_cast<int32_t>(r), bad, nsimple);
            s_a[i] = x;
            atomicAdd(&s_cnt[row_bucket(x, top)], 1u);
        }
        __syncthreads();
        if (warp == 0) {
            // exclusive scan of the 256 counts, 8 per lane
            uint32_t c[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                c[j] = s_cnt[lane * 8 + j];
                sum += c[j];
                if (c[j] > kBucketRun) s_big = 1;
            }
            uint32_t x = sum;
#pragma unroll
            for (int off2 = 1; off2 < 32; off2 <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, off2);
                if (lane >= off2) x += y;
            }
            uint32_t run = x - sum;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                s_start[lane * 8 + j] = run;
                s_cnt[lane * 8 + j] = run;  // becomes the scatter cursor
                run += c[j];
            }
            if (lane == 31) s_start[256] = run;
        }
        __syncthreads();
        if (s_big) {
            // every thread reads s_big after the barrier, so the branch is uniform
            __syncthreads();
            sort_row_block<8>(R, r, v, o, d, s_b, &s_low, bad, nsimple);
            continue;
        }
        for (int i = t; i < d; i += 512) {
            const int32_t x = s_a[i];
            s_b[atomicAdd(&s_cnt[row_bucket(x, top)], 1u)] = x;
        }
        __syncthreads();
        for (int b = warp; b < 256; b += 16) {
            const int st = static_cast<int>(s_start[b]);
            const int sz = static_cast<int>(s_start[b + 1]) - st;
            if (sz <= 1) continue;
            if (sz <= 32) sort_run_warp<1>(s_b + st, sz);
            else if (sz <= 64) sort_run_warp<2>(s_b + st, sz);
            else if (sz <= 128) sort_run_warp<4>(s_b + st, sz);
            else sort_run_warp<8>(s_b + st, sz);
        }
        __syncthreads();
        int32_t *dst = R.ccol + R.coff[r];
        int low = 0;
        for (int i = t; i < d; i += 512) {
            const int32_t x = s_b[i];
            dst[i] = x;
            low += x < static_cast<int32_t>(r);
            if (i + 1 < d && s_b[i + 1] == x) nsimple = true;
        }
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) low += __shfl_down_sync(0xffffffffu, low, o2);
        if (lane == 0) atomicAdd(&s_low, low);
        __syncthreads();
        if (t == 0) R.lowcnt[r] = s_low;
        __syncthreads();  // the shared arrays are free for the next row
    }
    report(R, bad, nsimple);
}

// Tier D (graphs with more than 2^20 vertices; smaller ones use the bitmap
// sort below): rows above 4096 entries, one block of 1024, stable LSD radix sort
// (8-bit digits) ping-ponging between the output row and a scratch row.  Each
// pass is a warp-level multisplit: every warp owns a contiguous slice of the
// row, counts its digits, gets per-(digit, warp) offsets from one block-wide
// scan, and scatters its slice in order -- stable without block barriers
// inside the scatter.  Bound by latency: two rows of 32 entries are read at
// once, and the lanes of a digit found by ballots (with one row at a time and
// __match_any_sync 1.12 ms per load on the 3M-vertex graph; 4 rows spill).
// A step there: 22.02 -> 21.90 ms.
constexpr int kRadixBatch = 2;
__global__ void __launch_bounds__(1024, 2) k_sort_tier_d(RowIn R, int32_t *tmp, int bits) {
    __shared__ uint32_t s_tot[256];
    __shared__ uint32_t s_wcnt[32][256];
    __shared__ int s_low;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r0 = static_cast<int64_t>(R.status[ST_TIER + 3]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_TIER + 4]);
    const int64_t tbase = (r0 < r1) ? R.coff[r0] : 0;
    bool bad = false, nsimple = false;
    for (int64_t r = r0 + blockIdx.x; r < r1; r += gridDim.x) {
        const uint32_t v = R.inv[r];
        const int64_t o = ldg_i64(R.off + v);
        const int64_t d = ldg_i64(R.off + v + 1) - o;
        int32_t *out = R.ccol + R.coff[r];
        int32_t *scr = tmp + (R.coff[r] - tbase);
#pragma unroll 4
        for (int64_t i = threadIdx.x; i < d; i += blockDim.x)
            scr[i] = relabel(R, o + i, v, (int32_t)r, bad, nsimple);
        __syncthreads();
        int32_t *src = scr, *dst = out;
        const int64_t slice = (d + 31) / 32;
        const int64_t lo = warp * slice;
        const int64_t hi = (lo + slice < d) ? lo + slice : d;
        for (int shift = 0; shift < bits; shift += 8) {
            // (1) per-warp digit counts of the warp's slice
            if (threadIdx.x < 256)
                for (int w = 0; w < 32; w++) s_wcnt[w][threadIdx.x] = 0;
            __syncthreads();
#pragma unroll 4
            for (int64_t i = lo + lane; i < hi; i += 32)
                atomicAdd(&s_wcnt[warp][(static_cast<uint32_t>(src[i]) >> shift) & 255u], 1u);
            __syncthreads();
            // (2) offsets in (digit, warp) order: digit totals, their
            // exclusive scan, then the warps in order within each digit
            if (threadIdx.x < 256) {
                uint32_t t = 0;
                for (int w = 0; w < 32; w++) t += s_wcnt[w][threadIdx.x];
                s_tot[threadIdx.x] = t;
            }
            __syncthreads();
            if (warp == 0) {
                uint32_t h[8], run = 0;
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    h[q] = s_tot[lane * 8 + q];
                    run += h[q];
                }
                uint32_t x = run;
#pragma unroll
                for (int o2 = 1; o2 < 32; o2 <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o2);
                    if (lane >= o2) x += y;
                }
                uint32_t e = x - run;
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    s_tot[lane * 8 + q] = e;
                    e += h[q];
                }
            }
            __syncthreads();
            if (threadIdx.x < 256) {
                uint32_t base = s_tot[threadIdx.x];
                for (int w = 0; w < 32; w++) {
                    const uint32_t c = s_wcnt[w][threadIdx.x];
                    s_wcnt[w][threadIdx.x] = base;
                    base += c;
                }
            }
            __syncthreads();
            // (3) each warp scatters its slice in order, two rows of 32 read
            // at once
            for (int64_t i0 = lo; i0 < hi; i0 += 32 * kRadixBatch) {
                int32_t x[kRadixBatch];
#pragma unroll
                for (int q = 0; q < kRadixBatch; q++) x[q] = i0 + 32 * q + lane < hi ? src[i0 + 32 * q + lane] : 0;
#pragma unroll
                for (int q = 0; q < kRadixBatch; q++) {
                    const bool valid = i0 + 32 * q + lane < hi;
                    const uint32_t digit = (static_cast<uint32_t>(x[q]) >> shift) & 255u;
                    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
                    for (int b = 0; b < 8; b++) {
                        const bool bit = (digit >> b) & 1u;
                        const uint32_t same = __ballot_sync(0xffffffffu, bit);
                        peers &= bit ? same : ~same;
                    }
                    const uint32_t rank = __popc(peers & lanemask_lt());
                    const uint32_t base = s_wcnt[warp][digit];
                    __syncwarp();
                    if (valid) {
                        dst[base + rank] = x[q];
                        if (lane == __ffs(peers) - 1) s_wcnt[warp][digit] = base + __popc(peers);
                    }
                    __syncwarp();
                }
            }
            __syncthreads();
            int32_t *t = src;
            src = dst;
            dst = t;
        }
        if (src != out) {
            for (int64_t i = threadIdx.x; i < d; i += blockDim.x) out[i] = src[i];
            __syncthreads();
        }
        if (threadIdx.x == 0) s_low = 0;
        __syncthreads();
        int low = 0;
        for (int64_t i = threadIdx.x; i < d; i += blockDim.x) {
            const int32_t x = out[i];
            low += (x < (int32_t)r);
            if (i + 1 < d && out[i + 1] == x) nsimple = true;
        }
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) low += __shfl_down_sync(0xffffffffu, low, o2);
        if (lane == 0) atomicAdd(&s_low, low);
        __syncthreads();
        if (threadIdx.x == 0) R.lowcnt[r] = s_low;
        __syncthreads();
    }
    report(R, bad, nsimple);
}

// Rows above kTierC entries, one block of 1024 per row, sorted through a
// bitmap of labels in shared memory: a relabelled row is a set of distinct
// labels in [0, n), so setting one bit per entry and reading the bits back
// in order sorts it (a repeated entry finds its bit already set).  Labels
// are taken kBitmapBits at a time (one chunk when n <= 2^20).  Warp w owns
// words [1024 w, 1024 (w + 1)) and reads them lane-interleaved (no bank
// conflicts): one pass counts its bits, a block scan of the warp counts
// gives each warp its output base, and a second pass writes the labels in
// order -- positions from warp scans of the words' bit counts -- and clears
// each word behind it, so the bitmap is empty again for the next chunk.
constexpr int kBitmapThreads = 1024;
constexpr int kBitmapWords = 1 << 15;
constexpr int64_t kBitmapBits = 32ll * kBitmapWords;  // 2^20 labels, 128 KB
constexpr int kWarpWords = kBitmapWords / (kBitmapThreads / 32);  // 1024

__global__ void __launch_bounds__(kBitmapThreads, 1) k_sort_bitmap(RowIn R, int32_t *tmp) {
    extern __shared__ uint32_t s_bits[];
    __shared__ int s_warp[32];
    __shared__ int s_low[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t r0 = static_cast<int64_t>(R.status[ST_TIER + 3]);
    const int64_t r1 = static_cast<int64_t>(R.status[ST_TIER + 4]);
    const int64_t tbase = (r0 < r1) ? R.coff[r0] : 0;
    bool bad = false, nsimple = false;
    for (int w = tid; w < kBitmapWords; w += kBitmapThreads) s_bits[w] = 0u;
    __syncthreads();
    uint32_t *mine = s_bits + warp * kWarpWords;
    for (int64_t r = r0 + blockIdx.x; r < r1; r += gridDim.x) {
        const uint32_t v = R.inv[r];
        const int64_t o = ldg_i64(R.off + v);
        const int d = static_cast<int>(ldg_i64(R.off + v + 1) - o);
        int32_t *t = tmp + (R.coff[r] - tbase);
        for (int i = tid; i < d; i += kBitmapThreads)
            t[i] = relabel(R, o + i, v, static_cast<int32_t>(r), bad, nsimple);
        __syncthreads();
        int32_t *dst = R.ccol + R.coff[r];
        int written = 0, low = 0;
        for (int64_t c0 = 0; c0 < R.n; c0 += kBitmapBits) {
            for (int i = tid; i < d; i += kBitmapThreads) {
                const int64_t x = static_cast<int64_t>(t[i]) - c0;
                if (x >= 0 && x < kBitmapBits) {
                    const uint32_t m = 1u << (x & 31);
                    if (atomicOr(s_bits + (x >> 5), m) & m) nsimple = true;
                }
            }
            __syncthreads();
            int cnt = 0;
            for (int k = lane; k < kWarpWords; k += 32) cnt += __popc(mine[k]);
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, q);
            if (lane == 0) s_warp[warp] = cnt;
            __syncthreads();
            if (warp == 0) {
                const int c = s_warp[lane];
                int incl = c;
#pragma unroll
                for (int q = 1; q < 32; q <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, q);
                    if (lane >= q) incl += y;
                }
                s_warp[lane] = incl - c;  // exclusive warp bases
                if (lane == 31) s_low[0] = incl;  // chunk total
            }
            __syncthreads();
            int run = written + s_warp[warp];
            const int total = s_low[0];
            const int64_t wbase = c0 + 32ll * warp * kWarpWords;
            for (int k = lane; k < kWarpWords; k += 32) {
                uint32_t bits = mine[k];
                mine[k] = 0u;
                const int c = __popc(bits);
                int incl = c;
#pragma unroll
                for (int q = 1; q < 32; q <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, q);
                    if (lane >= q) incl += y;
                }
                int pos = run + incl - c;
                while (bits) {
                    const int b = __ffs(bits) - 1;
                    bits &= bits - 1;
                    const int32_t label = static_cast<int32_t>(wbase + 32ll * k + b);
                    dst[pos++] = label;
                    low += label < static_cast<int32_t>(r);
                }
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            written += total;
            __syncthreads();  // s_warp / s_low reused by the next chunk
        }
        // repeated entries leave the row short: later kernels of the load take
        // every column for a label
        for (int i = written + tid; i < d; i += kBitmapThreads) dst[i] = static_cast<int32_t>(r);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) low += __shfl_xor_sync(0xffffffffu, low, q);
        if (lane == 0) s_low[warp] = low;
        __syncthreads();
        if (warp == 0) {
            int c = s_low[lane];
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) c += __shfl_xor_sync(0xffffffffu, c, q);
            if (lane == 0) R.lowcnt[r] = c;
        }
        __syncthreads();
    }
    report(R, bad, nsimple);
}

// ------------------------------------------------------------- edge table

struct LoadUp {
    const int32_t *dnew;
    const int32_t *low;
    __device__ int64_t operator()(int64_t i) const { return (int64_t)dnew[i] - low[i]; }
};
struct StoreUbase {
    int64_t *ubase;
    const int64_t *off;
    const int32_t *dnew, *low;
    int2 *row_span, *row_upper;  // below 2^31 all (nnz < 2^31)
    int64_t n;
    u64 *status;
    __device__ void operator()(int64_t i, int64_t exc, int64_t inc) const {
        ubase[i] = exc;
        row_span[i] = make_int2(static_cast<int32_t>(off[i]), dnew[i]);
        row_upper[i] = make_int2(low[i], static_cast<int32_t>(exc));
        if (i == n - 1) {
            ubase[n] = inc;
            status[ST_M_UPPER] = static_cast<u64>(inc);
        }
    }
};

// ------------------------------------------------------------------- driver

// Runs independent kernels of one call on its side streams: fork()
// makes them wait for the caller's stream, join() makes the caller's stream
// wait for them.  The destructor joins on every return path, so no side work
// outlives a call that failed halfway.  Without side streams every kernel
// runs on the caller's stream.
class SideFork {
  public:
    SideFork(ps_graph *g, const SideStreams &streams, cudaStream_t s) : g_(g), streams_(streams), s_(s) { side_[0] = side_[1] = s; }
    ~SideFork() { join(); }
    SideFork(const SideFork &) = delete;
    SideFork &operator=(const SideFork &) = delete;

    int fork(int count) {
        if (!streams_.stream[0]) return PS_OK;
        PS_CUDA_TRY(cudaEventRecord(g_->ev[0], s_));
        for (int i = 0; i < count; i++) {
            PS_CUDA_TRY(cudaStreamWaitEvent(streams_.stream[i], g_->ev[0], 0));
            side_[i] = streams_.stream[i];
            used_ = i + 1;
        }
        return PS_OK;
    }
    cudaStream_t side(int i) const { return side_[i]; }
    int join() {
        int rc = PS_OK;
        for (int i = 0; i < used_; i++)
            if (cudaEventRecord(g_->ev[1 + i], side_[i]) != cudaSuccess ||
                cudaStreamWaitEvent(s_, g_->ev[1 + i], 0) != cudaSuccess)
                rc = PS_ERR_CUDA;
        used_ = 0;
        return rc;
    }

  private:
    ps_graph *g_;
    const SideStreams &streams_;
    cudaStream_t s_;
    cudaStream_t side_[2];
    int used_ = 0;
};

int load_graph(ps_graph *g, const int64_t *d_off, const int32_t *d_col, cudaStream_t s) {
    const Layout &L = g->L;
    const int64_t n = L.n, nnz = L.nnz;
    char *ws = g->ws;
    const int sms = g->sm_count;
    // the status words and, right behind them, the counters and slots of every
    // scan of this load
    g->scan_used = 0;
    PS_CUDA_TRY(cudaMemsetAsync(g->status, 0, L.scan - L.status + sizeof(uint64_t) * L.scan_words, s));
    uint32_t *k0 = reinterpret_cast<uint32_t *>(ws + L.keys0);
    uint32_t *k1 = reinterpret_cast<uint32_t *>(ws + L.keys1);
    uint32_t *v0 = reinterpret_cast<uint32_t *>(ws + L.vals0);
    uint32_t *v1 = reinterpret_cast<uint32_t *>(ws + L.vals1);

    // (1) degrees and offset validation; nothing else may index with bad offsets
    k_degrees<<<sms * 8, 256, 0, s>>>(n, nnz, d_off, k0, g->status);
    PS_LAUNCH_CHECK();
    SideStreams streams(g->device);
    SideFork read(g, streams, s);
    int rc = read.fork(1);
    if (rc) return rc;

    // (2) stable radix sort of (degree, id): ties keep increasing id.  Queued
    // before the host has seen the largest degree (below n on valid input):
    // passes above its bits do nothing.
    int bits = 1;
    while (bits < 31 && (static_cast<uint64_t>(n > 0 ? n - 1 : 0) >> bits) != 0) bits++;
    SortPass order[kMaxPasses];
    int passes = 0;
    for (int shift = 0; shift < bits && n > 0; shift += 8) {
        const bool even = shift % 16 == 0;
        order[passes++] = {n, nullptr, even ? k0 : k1, shift ? (even ? v0 : v1) : nullptr, even ? k1 : k0,
                           even ? v1 : v0, shift, std::min(8, bits - shift), 0,
                           reinterpret_cast<uint32_t *>(ws + L.counts), g->status + ST_DMAX};
    }
    auto take = [g](int64_t tiles, ScanState<uint32_t> *scan) { return take_scan(g, tiles, scan); };
    rc = sort_passes(order, passes, take, s);
    if (rc) return rc;
    uint32_t *inv = reinterpret_cast<uint32_t *>(ws + L.inv);
    if (n > 0) {
        k_rank<<<sms * 8, 256, 0, s>>>(n, bits, k0, v0, k1, v1, g->rank, inv, g->dnew, g->lowcnt,
                                       static_cast<uint32_t>(tier_b(nnz)), L.hub_cap,
                                       g->tune.hub_min_degree, g->status);
        PS_LAUNCH_CHECK();
    } else {
        PS_CUDA_TRY(cudaMemsetAsync(g->off, 0, sizeof(int64_t), s));
        PS_CUDA_TRY(cudaMemsetAsync(g->ubase, 0, sizeof(int64_t), s));
    }
    rc = run_scan<int64_t>(g, n, (int64_t)0, OpSum(), LoadDeg{g->dnew}, StoreOffsets{g->off, n}, s);
    if (rc) return rc;

    // the offsets' verdict and the largest degree, read on the side while the
    // sort runs
    static_assert(ST_WORDS <= Readback::kWords, "the words fit a read-back");
    Readback back;
    rc = back.queue(g->status, ST_WORDS, nullptr, 0, read.side(0));
    if (rc) return rc;
    PS_CUDA_TRY(cudaStreamSynchronize(read.side(0)));
    const uint64_t *st = back.words;
    rc = read.join();
    if (rc) return rc;
    g->d_max = static_cast<int64_t>(st[ST_DMAX]);
    if ((st[ST_FLAGS] & F_ARG) || g->d_max >= std::max<int64_t>(n, 1)) {
        // bad offsets, or a row too long to be simple (then only a column out
        // of range outranks that)
        if (!(st[ST_FLAGS] & F_ARG)) {
            k_check_columns<<<sms * 8, 256, 0, s>>>(n, nnz, d_col, g->status);
            PS_LAUNCH_CHECK();
        }
        rc = back.queue(g->status, ST_WORDS, nullptr, 0, s);
        if (rc) return rc;
        PS_CUDA_TRY(cudaStreamSynchronize(s));
        return flags_to_status(st[ST_FLAGS] | F_NOT_SIMPLE);
    }

    // (3) relabel + sort every row, by tier; the tiers touch disjoint rows, so
    // the long-row tiers run on side streams next to the short-row ones
    RowIn R{d_off, d_col, inv, g->rank, g->off, g->col, g->lowcnt, n, g->status};
    if (n > 0) {
        SideFork fork(g, streams, s);
        if (g->d_max > tier_b(nnz)) {
            rc = fork.fork(2);
            if (rc) return rc;
        }
        // rows above kTierC: the bitmap sort when all labels fit one chunk
        // (R-MAT 20: 0.11 ms against 0.25 ms for the radix sort), the block
        // radix sort otherwise (3 chunks on the 3M-vertex graph: +0.4 ms)
        const bool bitmap = n <= kBitmapBits;
        if (bitmap && g->d_max > kTierC) {
            const int smem = kBitmapWords * static_cast<int>(sizeof(uint32_t));
            PS_CUDA_TRY(cudaFuncSetAttribute(k_sort_bitmap, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            k_sort_bitmap<<<sms, kBitmapThreads, smem, fork.side(1)>>>(R, reinterpret_cast<int32_t *>(g->rec));
            PS_LAUNCH_CHECK();
        }
        if (!bitmap && g->d_max > kTierC) {
            int vb = 0;
            while (vb < 31 && (static_cast<uint64_t>(n - 1) >> vb) != 0) vb++;
            k_sort_tier_d<<<sms * 2, 1024, 0, fork.side(1)>>>(R, reinterpret_cast<int32_t *>(g->rec), vb);
            PS_LAUNCH_CHECK();
        }
        if (g->d_max > tier_b(nnz)) {
            k_sort_tier_c<<<sms * 3, 512, 0, fork.side(0)>>>(R);
            PS_LAUNCH_CHECK();
        }
        k_sort_tier_b<<<sms * 8, 256, 0, s>>>(R);
        PS_LAUNCH_CHECK();
        if (g->d_max > kLongRow) {
            k_sort_tier_b2<<<sms * 4, 256, 0, s>>>(R);
            PS_LAUNCH_CHECK();
        }
        k_sort_tier_a<<<sms * 16, 256, 0, s>>>(R);
        PS_LAUNCH_CHECK();
        rc = fork.join();
        if (rc) return rc;
    }

    // (4) the edge numbering: ubase[r] = the edges (upper arcs) of the rows before r
    rc = run_scan<int64_t>(g, n, (int64_t)0, OpSum(), LoadUp{g->dnew, g->lowcnt},
                           StoreUbase{g->ubase, g->off, g->dnew, g->lowcnt, g->row_span, g->row_upper, n, g->status}, s);
    if (rc) return rc;

    // (5) on a side stream the hub rows, which need only the sorted rows; here
    // the edge table, the prefixes and the edge filter, then the guide tables
    SideFork hubs(g, streams, s);
    rc = hubs.fork(1);
    if (rc) return rc;
    rc = launch_hub_rows(g, hubs.side(0));
    if (rc) return rc;
    if (g->filt) PS_CUDA_TRY(cudaMemsetAsync(g->filt, 0, sizeof(uint32_t) * L.filt_words, s));
    rc = build_edge_table(g, s);
    if (rc) return rc;
    rc = launch_guides(g, s);
    if (rc) return rc;
    rc = hubs.join();
    if (rc) return rc;

    rc = back.queue(g->status, ST_WORDS, nullptr, 0, s);
    if (rc) return rc;
    PS_CUDA_TRY(cudaStreamSynchronize(s));
    g->load_totals[0] = st[ST_W_LO];
    g->load_totals[1] = st[ST_L_LO];
    g->load_totals[2] = st[ST_N1_LO];
    g->load_totals[3] = st[ST_N1_HI];
    g->load_totals[4] = st[ST_HUBS];
    g->load_flags = st[ST_FLAGS];
    const uint64_t m_upper = st[ST_M_UPPER];
    uint64_t flags = st[ST_FLAGS];
    if (2 * m_upper != static_cast<uint64_t>(nnz)) flags |= F_ASYM;
    // a prefix sum past 2^64 is reported by ps_tau_prefix, as documented
    const int status = flags_to_status(flags & ~static_cast<uint64_t>(F_OVERFLOW));
    if (status != PS_OK) return status;
    g->m = static_cast<int64_t>(m_upper);
    return PS_OK;
}

}  // namespace ps
