// ccs_setup.cu -- expander generation, CSR transpose and y = A x.
//
// Generation follows the Sec. 1.1 footnote of the paper: columns are drawn
// independently, each column's support uniform over the C(m, d) subsets of
// size d.  Every column owns a counter-based SplitMix64 stream, so a column
// is one thread's work and the matrix depends only on (n, m, d, seed).
#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <cstdarg>
#include <cstdio>

#include "ccs_checks.cuh"
#include "ccs_internal.cuh"

namespace ccs {

// ---------------------------------------------------------------------------
// Random numbers
// ---------------------------------------------------------------------------

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014): Weyl increment
// 0x9e3779b97f4a7c15, then the variant-13 mixing function.
__device__ __forceinline__ uint64_t splitmix64(uint64_t &state) {
    state += 0x9e3779b97f4a7c15ull;
    uint64_t z = state;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Lemire's bounded draw (ACM TOMACS 2019): high word of x * range, redrawing
// while the low word is below 2^64 mod range.  The 96-bit product is formed
// from two 32 x 32-bit ones (range has 32 bits).
__device__ __forceinline__ uint32_t draw_below(uint64_t &state, uint32_t range) {
    uint64_t x = splitmix64(state);
    uint64_t p0 = (x & 0xffffffffull) * range, p1 = (x >> 32) * range + (p0 >> 32);
    uint64_t lo = (p1 << 32) | (p0 & 0xffffffffull);
    if (lo < range) {
        const uint64_t floor_mod = (0ull - (uint64_t)range) % (uint64_t)range;
        while (lo < floor_mod) {
            x = splitmix64(state);
            p0 = (x & 0xffffffffull) * range;
            p1 = (x >> 32) * range + (p0 >> 32);
            lo = (p1 << 32) | (p0 & 0xffffffffull);
        }
    }
    return (uint32_t)(p1 >> 32);
}

// Column j's D distinct rows, ascending, in registers.
template <int D>
__device__ __forceinline__ void draw_column(int j, int m, uint64_t seed, int32_t (&rows)[D]) {
    uint64_t state = seed + (uint64_t)(j + 1) * 0xd1b54a32d192ed03ull;
#pragma unroll
    for (int t = 0; t < D; ++t) {
        bool seen;
        do {
            rows[t] = (int32_t)draw_below(state, (uint32_t)m);
            seen = false;
#pragma unroll
            for (int q = 0; q < t; ++q) seen |= (rows[q] == rows[t]);
        } while (seen);
    }
    // compare-exchange rounds of neighbours: D of them sort D values
#pragma unroll
    for (int round = 0; round < D; ++round)
#pragma unroll
        for (int q = round & 1; q + 1 < D; q += 2) {
            const int32_t lo = min(rows[q], rows[q + 1]), hi = max(rows[q], rows[q + 1]);
            rows[q] = lo;
            rows[q + 1] = hi;
        }
}

// A block's columns (their rows laid out one column after another in shared
// memory) to the CSC array by 16-byte stores: `ints` of them from dst, which
// is 16-byte aligned.
__device__ __forceinline__ void store_columns(const int32_t *stage, int32_t *dst, int ints) {
    for (int q = threadIdx.x; q < ints / 4; q += blockDim.x)
        reinterpret_cast<int4 *>(dst)[q] = reinterpret_cast<const int4 *>(stage)[q];
    for (int q = (ints & ~3) + threadIdx.x; q < ints; q += blockDim.x) dst[q] = stage[q];
}

// One thread a column, and one atomic add per entry counts its row.  With
// shift > 0 the add's result, the entry's rank in its row, rides in the bits of
// the row index above `shift` (k_place_ranked takes it out again), so that
// placing the transpose needs no second round of atomics.
//
// Bound by the 64-bit integer work of the draws (~25 instructions each) and
// the atomics; the entries go through shared memory so that the stores are
// whole lines instead of 4 d-byte pieces.
constexpr int kGenBlock = 256;
template <int D>
__global__ void __launch_bounds__(kGenBlock)
k_generate_columns(int n, int m, uint64_t seed, int shift, int32_t *csc_rows, int32_t *deg) {
    __shared__ __align__(16) int32_t stage[kGenBlock * D];
    const int j0 = blockIdx.x * kGenBlock, j = j0 + threadIdx.x;
    if (j < n) {
        int32_t rows[D];
        draw_column<D>(j, m, seed, rows);
        if (shift) {
            int rank[D];
#pragma unroll
            for (int t = 0; t < D; ++t) rank[t] = atomicAdd(deg + rows[t], 1);
#pragma unroll
            for (int t = 0; t < D; ++t)
                stage[threadIdx.x * D + t] = rows[t] | (int32_t)((uint32_t)rank[t] << shift);
        } else {
#pragma unroll
            for (int t = 0; t < D; ++t) {
                atomicAdd(deg + rows[t], 1);
                stage[threadIdx.x * D + t] = rows[t];
            }
        }
    }
    __syncthreads();
    store_columns(stage, csc_rows + (size_t)j0 * D, min(kGenBlock, n - j0) * D);
}

// ---------------------------------------------------------------------------
// CSR transpose: row degrees -> scan -> place -> sort each row
// ---------------------------------------------------------------------------

constexpr int kScanBlock = 1024;
constexpr int kWarpSortCap = 512;   // longest row a warp sorts in registers
// From here on the rows' counters and offsets leave L2, and entries carry their
// ranks from the count to the placing instead of counting again (n = 2^25 + 1:
// m = 2^24, d = 7 18.7 ms against 23.7; m = 2^22, d = 5 10.7 against 10.4; m =
// 2^20, d = 3 5.8 against 4.2).
constexpr int kRankedRows = 1 << 22;
constexpr int kGroupEntries = 36864;  // entries a group of rows has at most, on average
constexpr int kMaxGroups = 8192;      // counted on chip
constexpr int kMaxGroupRowBits = 12;
constexpr int kBucketEntries = 8;
// Matrices measured through the nonzero marks: from 2^24 entries (n = 2^22,
// m = 2^19, d = 7: 112 us against 131 us for gathering every entry; n = 2^24,
// m = 16777, d = 9: 193 against 604), and from 2^22 when rows are long, which
// few warps gather (n = 2^20, m = 10486, d = 7: 25 us against 43 us).  Below,
// x stays in L2 and the second launch costs more than it saves (n = 2^20,
// m = 2^17, d = 7: 45 us against 37 us).
constexpr long long kMarkedMinEntries = 1 << 24;
constexpr long long kMarkedMinLongRows = 1 << 22;
constexpr long long kMarkedLongRow = 128;         // mean columns of a long row
constexpr int kMarkBytes = 128 << 10;             // marks in shared memory
constexpr int kMarkMaxShift = 8;                  // coarsest mark: 256 columns

// Per block of kScanBlock rows: inclusive prefix of deg into ptr[1 + i],
// block total into sums[block], largest degree into *max_deg.
__global__ void __launch_bounds__(kScanBlock)
k_scan_local(int m, const int32_t *deg, int64_t *ptr, int64_t *sums, int *max_deg) {
    __shared__ long long warp_tot[kScanBlock / 32];
    const int i = blockIdx.x * kScanBlock + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long v = (i < m) ? deg[i] : 0;
    int mx = (int)v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0 && mx > 0) atomicMax(max_deg, mx);
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        long long w = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        warp_tot[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    if (warp > 0) inc += warp_tot[warp - 1];
    if (i < m) ptr[i + 1] = inc;
    if (threadIdx.x == kScanBlock - 1) sums[blockIdx.x] = inc;
}

// ptr += the totals of the blocks before.  Up to kScanBlock blocks (m = 2^20)
// each sums them itself, one load a thread; beyond, k_scan_totals has turned
// them into prefixes (`scanned`): the sums would be quadratic in m (33 ms
// more at m = 2^29, 1.8 ms at 2^27).
__global__ void __launch_bounds__(kScanBlock)
k_scan_add(int m, int64_t *ptr, const int64_t *sums, bool scanned) {
    __shared__ unsigned long long before;
    const int i = blockIdx.x * kScanBlock + threadIdx.x;
    if (i == 0) ptr[0] = 0;
    if (scanned) {
        if (i < m) ptr[i + 1] += sums[blockIdx.x];
        return;
    }
    if (threadIdx.x == 0) before = 0;
    __syncthreads();
    const long long v = warp_sum_ll(threadIdx.x < blockIdx.x ? sums[threadIdx.x] : 0);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&before, (unsigned long long)v);
    __syncthreads();
    if (i < m) ptr[i + 1] += (long long)before;
}

// Exclusive prefix of the block totals, in place: one block, each warp a
// stretch of them, 32 consecutive ones at a time.
__global__ void __launch_bounds__(kScanBlock) k_scan_totals(int nblocks, int64_t *sums) {
    constexpr int kU = 8;  // loads in flight
    __shared__ long long warp_tot[kScanBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (nblocks + kScanBlock - 1) / kScanBlock * 32;
    const int b0 = min(nblocks, warp * per), b1 = min(nblocks, b0 + per);
    long long sum = 0;
#pragma unroll kU
    for (int b = b0 + lane; b < b1; b += 32) sum += sums[b];
    sum = warp_sum_ll(sum);
    if (lane == 0) warp_tot[warp] = sum;
    __syncthreads();
    long long run = 0;
    for (int w = 0; w < warp; ++w) run += warp_tot[w];
    for (int b = b0 + lane; b - lane < b1; b += 32 * kU) {
        long long v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = b + 32 * u < b1 ? sums[b + 32 * u] : 0;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            long long inc = v[u];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            if (b + 32 * u < b1) sums[b + 32 * u] = run + inc - v[u];
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
}

// Entries of a k_generate_columns that packed their ranks: each goes to its
// place in its row, and the CSC array gets the plain row index back.  A
// thread takes four entries (one 16-byte load and store of the CSC).
template <int D>
__global__ void k_place_ranked(long long edges, int shift, int32_t *csc_rows, const int64_t *ptr,
                               int32_t *csr_cols) {
    const uint32_t mask = (1u << shift) - 1u;
    const long long quads = edges / 4;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < quads; q += step) {
        int4 v = reinterpret_cast<int4 *>(csc_rows)[q];
        uint32_t e[4] = {(uint32_t)v.x, (uint32_t)v.y, (uint32_t)v.z, (uint32_t)v.w};
        int64_t at[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) at[t] = __ldg(ptr + (e[t] & mask)) + (e[t] >> shift);
        v.x = (int)(e[0] & mask);
        v.y = (int)(e[1] & mask);
        v.z = (int)(e[2] & mask);
        v.w = (int)(e[3] & mask);
        reinterpret_cast<int4 *>(csc_rows)[q] = v;
#pragma unroll
        for (int t = 0; t < 4; ++t) csr_cols[at[t]] = (int32_t)((uint32_t)(4 * q + t) / D);
    }
    const long long r = quads * 4 + blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (r < edges) {
        const uint32_t e = (uint32_t)csc_rows[r];
        csc_rows[r] = (int32_t)(e & mask);
        csr_cols[__ldg(ptr + (e & mask)) + (e >> shift)] = (int32_t)((uint32_t)r / D);
    }
}

__global__ void k_scatter_cols(int n, int d, const int32_t *csc_rows, const int64_t *ptr,
                               int32_t *fill, int32_t *csr_cols) {
    const long long edges = (long long)n * d;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < edges;
         e += (long long)gridDim.x * blockDim.x) {
        const int32_t i = csc_rows[e];
        const int32_t pos = atomicAdd(&fill[i], 1);
        csr_cols[ptr[i] + pos] = (int32_t)(e / d);
    }
}

// One block per row: bucket sort of the row's columns in shared memory.  The
// columns of a row are uniform over [0, n), so buckets of equal width
// (2^shift columns, `buckets` of them cover n) hold a few each (~8), and a
// thread sorts a bucket by insertion.  Any other distribution is sorted too,
// only slower.  Rows longer than `cap` are left alone.
//
// The row is read twice (the second time from cache) and written once; the
// compare-exchange network it replaces took log2(len)^2 / 2 passes over
// shared memory (12.5 ms at n = 2^24, m = 16777, d = 9).
constexpr int kSortBlock = 512;
__global__ void __launch_bounds__(kSortBlock)
k_sort_rows(int m, int cap, int shift, int buckets, const int64_t *ptr, int32_t *csr_cols) {
    extern __shared__ int32_t sm[];
    int32_t *end = sm, *buf = sm + buckets;  // buckets, cap
    __shared__ int warp_tot[kSortBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = blockIdx.x; i < m; i += gridDim.x) {
        const int64_t b = ptr[i];
        const int len = (int)(ptr[i + 1] - b);
        if (len <= 1 || len > cap) continue;
        for (int q = threadIdx.x; q < buckets; q += kSortBlock) end[q] = 0;
        __syncthreads();
        for (int t = threadIdx.x; t < len; t += kSortBlock)
            atomicAdd(end + (csr_cols[b + t] >> shift), 1);
        __syncthreads();
        // exclusive prefix of the counts: a run of buckets a thread
        const int per = (buckets + kSortBlock - 1) / kSortBlock;
        const int q0 = min(buckets, (int)threadIdx.x * per), q1 = min(buckets, q0 + per);
        int sum = 0;
        for (int q = q0; q < q1; ++q) sum += end[q];
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) warp_tot[warp] = inc;
        __syncthreads();
        int run = inc - sum;
        for (int w = 0; w < warp; ++w) run += warp_tot[w];
        for (int q = q0; q < q1; ++q) {
            const int c = end[q];
            end[q] = run;
            run += c;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < len; t += kSortBlock) {
            const int32_t c = csr_cols[b + t];
            buf[atomicAdd(end + (c >> shift), 1)] = c;
        }
        __syncthreads();  // end[q] is now bucket q's end
        for (int q = threadIdx.x; q < buckets; q += kSortBlock) {
            const int lo = q ? end[q - 1] : 0, hi = end[q];
            for (int t = lo + 1; t < hi; ++t) {
                const int32_t c = buf[t];
                int u = t - 1;
                while (u >= lo && buf[u] > c) {
                    buf[u + 1] = buf[u];
                    --u;
                }
                buf[u + 1] = c;
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < len; t += kSortBlock) csr_cols[b + t] = buf[t];
        __syncthreads();
    }
}

// Rows of at most 32 E columns: one warp a row, the row in registers (E per
// lane, element lane * E + e), bitonic sort by register exchanges and warp
// shuffles: no shared memory and no block barriers.  Longer rows are left alone.
template <int E>
__global__ void k_sort_rows_warp(int m, const int64_t *ptr, int32_t *csr_cols) {
    constexpr int kCap = 32 * E;
    const int lane = threadIdx.x & 31;
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long i = w0; i < m; i += nw) {
        const int64_t b = ptr[i];
        const int len = (int)(ptr[i + 1] - b);
        if (len <= 1 || len > kCap) continue;
        int32_t v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int idx = lane * E + e;
            v[e] = idx < len ? csr_cols[b + idx] : 0x7fffffff;
        }
#pragma unroll
        for (int k = 2; k <= kCap; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                if (j < E) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int p = e ^ j;
                        if (p > e) {
                            const bool up = ((lane * E + e) & k) == 0;
                            const int32_t a = v[e], c = v[p];
                            if ((a > c) == up) {
                                v[e] = c;
                                v[p] = a;
                            }
                        }
                    }
                } else {
                    const int lj = j / E;
                    const bool lower = (lane & lj) == 0;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const int32_t o = __shfl_xor_sync(0xffffffffu, v[e], lj);
                        const bool up = ((lane * E + e) & k) == 0;
                        v[e] = (lower == up) ? min(v[e], o) : max(v[e], o);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int idx = lane * E + e;
            if (idx < len) csr_cols[b + idx] = v[e];
        }
    }
}

// ---------------------------------------------------------------------------
// Grouped construction: draw -> partition by group of rows -> sort each group
// ---------------------------------------------------------------------------
//
// Rows are taken in groups of 2^row_bits whose entries fit one CTA's shared
// memory.  The columns are drawn and the groups' sizes counted on chip; a
// second pass deals the entries out to their groups' parts of csr_cols, a
// block's entries ordered by group on chip first so that they leave as runs;
// then a CTA a group sorts its entries by (row, column), which also gives
// the row offsets.  An entry on its way is one word, its row in the group
// above its column, so nothing beyond csr_cols is needed.
//
// What it replaces took two rounds of global atomics per entry, a scattered
// 4-byte store (about 130 G/s each, whatever their size) and a sort of
// log2(len)^2 / 2 passes: 18.2 ms at n = 2^24, m = 16777, d = 9 (2.28 ms
// here: draw 380 us, deal 750 us, sort 1016 us) and 324 us at n = 2^20, m =
// 2^17, d = 7 (146 us: 20, 23 and 66 us and four launches).

// Columns of this block's turn, their CSC entries stored, the entries per
// group added to size[0, groups).
constexpr int kDrawBlock = 512;
template <int D>
__global__ void __launch_bounds__(kDrawBlock)
k_draw_columns(int n, int m, uint64_t seed, int row_bits, int groups, int32_t *csc_rows,
               int32_t *size) {
    extern __shared__ __align__(16) int32_t sm[];
    int32_t *stage = sm, *cnt = sm + kDrawBlock * D;  // kDrawBlock D, groups
    for (int g = threadIdx.x; g < groups; g += kDrawBlock) cnt[g] = 0;
    __syncthreads();
    for (long long j0 = (long long)blockIdx.x * kDrawBlock; j0 < n;
         j0 += (long long)gridDim.x * kDrawBlock) {
        const long long j = j0 + threadIdx.x;
        if (j < n) {
            int32_t rows[D];
            draw_column<D>((int)j, m, seed, rows);
#pragma unroll
            for (int t = 0; t < D; ++t) {
                stage[threadIdx.x * D + t] = rows[t];
                atomicAdd(cnt + (rows[t] >> row_bits), 1);
            }
        }
        __syncthreads();
        store_columns(stage, csc_rows + (size_t)j0 * D, (int)min((long long)kDrawBlock, n - j0) * D);
        __syncthreads();
    }
    for (int g = threadIdx.x; g < groups; g += kDrawBlock)
        if (cnt[g]) atomicAdd(size + g, cnt[g]);
}

// Exclusive prefix of one int per thread over the block (kDealBlock threads).
constexpr int kDealBlock = 1024;
__device__ __forceinline__ int deal_scan(int v) {
    __shared__ int warp_tot[kDealBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    __syncthreads();  // earlier users of warp_tot are done
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    const int w = warp_tot[lane];
    const int before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0);
    return before + inc - v;
}

// Group sizes -> first entries (one block).
__global__ void __launch_bounds__(kDealBlock) k_scan_groups(int groups, int32_t *size) {
    const int per = (groups + kDealBlock - 1) / kDealBlock;
    const int g0 = min(groups, (int)threadIdx.x * per), g1 = min(groups, g0 + per);
    int sum = 0;
    for (int g = g0; g < g1; ++g) sum += size[g];
    int run = deal_scan(sum);
    for (int g = g0; g < g1; ++g) {
        const int c = size[g];
        size[g] = run;
        run += c;
    }
}

// Entries to their groups.  A block takes kDealPer entries a thread at a
// time, ranks them by group with shared-memory atomics, reserves each
// group's run (next[g], which starts as the group's first entry and ends as
// its last), lays the entries out by group on chip and stores them in that
// order: consecutive threads store consecutive words of a run.
constexpr int kDealPer = 24;
template <int D>
__global__ void __launch_bounds__(kDealBlock)
k_deal_entries(uint32_t edges, int row_bits, int col_bits, int groups, int per,
               const int32_t *csc_rows, int32_t *next, int32_t *csr_cols) {
    extern __shared__ __align__(16) int32_t sm[];
    int32_t *cnt = sm, *to = sm + groups;                     // groups each
    uint32_t *val = reinterpret_cast<uint32_t *>(to + groups);  // kDealBlock per
    uint16_t *grp = reinterpret_cast<uint16_t *>(val + kDealBlock * per);
    const uint32_t row_mask = (1u << row_bits) - 1u;
    const uint32_t turn = (uint32_t)(kDealBlock * per);
    for (uint64_t e0 = (uint64_t)blockIdx.x * turn; e0 < edges; e0 += (uint64_t)gridDim.x * turn) {
        const uint32_t len = (uint32_t)min((uint64_t)turn, edges - e0);
        for (int g = threadIdx.x; g < groups; g += kDealBlock) cnt[g] = 0;
        __syncthreads();
        int32_t row[kDealPer];
        uint16_t rank[kDealPer];
#pragma unroll
        for (int k = 0; k < kDealPer; ++k) {
            const uint32_t q = threadIdx.x + k * kDealBlock;
            row[k] = (k < per && q < len) ? __ldcs(csc_rows + e0 + q) : -1;
        }
#pragma unroll
        for (int k = 0; k < kDealPer; ++k)
            if (row[k] >= 0) rank[k] = (uint16_t)atomicAdd(cnt + (row[k] >> row_bits), 1);
        __syncthreads();
        const int gper = (groups + kDealBlock - 1) / kDealBlock;
        const int g0 = min(groups, (int)threadIdx.x * gper), g1 = min(groups, g0 + gper);
        int sum = 0;
        for (int g = g0; g < g1; ++g) {
            const int c = cnt[g];
            to[g] = c ? atomicAdd(next + g, c) : 0;
            sum += c;
        }
        int run = deal_scan(sum);
        for (int g = g0; g < g1; ++g) {
            const int c = cnt[g];
            cnt[g] = run;   // where the group starts on chip
            to[g] -= run;   // and how far its run is from there
            run += c;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kDealPer; ++k)
            if (row[k] >= 0) {
                const int g = row[k] >> row_bits, p = cnt[g] + rank[k];
                const uint32_t e = (uint32_t)e0 + threadIdx.x + k * kDealBlock;
                val[p] = (e / D) | (((uint32_t)row[k] & row_mask) << col_bits);
                grp[p] = (uint16_t)g;
            }
        __syncthreads();
        for (uint32_t p = threadIdx.x; p < len; p += kDealBlock)
            csr_cols[to[grp[p]] + (int)p] = (int32_t)val[p];
        __syncthreads();
    }
}

// One CTA a group: its entries sorted by (row, column), the rows' offsets,
// and the largest degree.  The packed words are dealt to buckets of equal
// width, which hold a few each (columns are uniform; no bucket spans two
// rows); then every entry counts the smaller ones of its bucket and goes
// straight to its place.  Any distribution is sorted, only slower.  The
// entries are read twice, the second time from cache.  end[g] is the
// group's last entry; a group of more than `cap` entries sets *max_deg to
// INT_MAX.
//
// Consecutive threads hold consecutive entries, so the counting reads a
// bucket's words together, without bank conflicts: a thread per bucket
// sorting it by insertion took 1285 us at n = 2^24, m = 16777, d = 9, this
// 1016 us.
constexpr int kGroupBlock = 1024;
__global__ void __launch_bounds__(kGroupBlock)
k_sort_groups(int m, int groups, int row_bits, int col_bits, int shift, int buckets, int cap,
              const int32_t *end, int64_t *csr_ptr, int32_t *csr_cols, int *max_deg) {
    extern __shared__ __align__(16) int32_t sm[];
    int32_t *top = sm;                                       // buckets
    uint32_t *buf = reinterpret_cast<uint32_t *>(sm + buckets);  // cap
    const uint32_t col_mask = (1u << col_bits) - 1u;
    for (int g = blockIdx.x; g < groups; g += gridDim.x) {
        const int b = g ? end[g - 1] : 0, len = end[g] - b;
        const int r0 = g << row_bits, rows = min(1 << row_bits, m - r0);
        if (len > cap) {
            if (threadIdx.x == 0) atomicMax(max_deg, 0x7fffffff);
            continue;
        }
        uint32_t *src = reinterpret_cast<uint32_t *>(csr_cols) + b;
        __syncthreads();  // the previous group's readers are done
        for (int q = threadIdx.x; q < buckets; q += kGroupBlock) top[q] = 0;
        __syncthreads();
#pragma unroll 8
        for (int t = threadIdx.x; t < len; t += kGroupBlock) atomicAdd(top + (src[t] >> shift), 1);
        __syncthreads();
        const int per = (buckets + kGroupBlock - 1) / kGroupBlock;
        const int q0 = min(buckets, (int)threadIdx.x * per), q1 = min(buckets, q0 + per);
        int sum = 0;
        for (int q = q0; q < q1; ++q) sum += top[q];
        int run = deal_scan(sum);
        for (int q = q0; q < q1; ++q) {
            const int c = top[q];
            top[q] = run;
            run += c;
        }
        __syncthreads();
#pragma unroll 8
        for (int t = threadIdx.x; t < len; t += kGroupBlock) {
            const uint32_t v = src[t];
            buf[atomicAdd(top + (v >> shift), 1)] = v;
        }
        __syncthreads();  // top[q] is now bucket q's end
        for (int t = threadIdx.x; t < len; t += kGroupBlock) {
            const uint32_t v = buf[t];
            const int q = (int)(v >> shift);
            const int lo = q ? top[q - 1] : 0, hi = top[q];
            int at = lo;
            for (int u = lo; u < hi; ++u) at += buf[u] < v;
            src[at] = v & col_mask;
        }
        // a row ends with its last bucket
        int mx = 0;
        const int row_shift = col_bits - shift;
        for (int r = threadIdx.x; r < rows; r += kGroupBlock) {
            const int from = r ? top[(r << row_shift) - 1] : 0;
            const int to = top[((r + 1) << row_shift) - 1];
            csr_ptr[(int64_t)r0 + r + 1] = (int64_t)b + to;
            mx = max(mx, to - from);
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((threadIdx.x & 31) == 0 && mx) atomicMax(max_deg, mx);
        if (g == 0 && threadIdx.x == 0) csr_ptr[0] = 0;
    }
}

// ---------------------------------------------------------------------------
// y = A x: one warp per row, ascending column order
// ---------------------------------------------------------------------------

// Sum of v[j] over the row's columns in ascending j, from +0.0, skipping zero
// entries.  The 32 lanes fetch 32 consecutive entries at a time; the nonzero
// ones are then added in lane order, so the addition order is exactly the
// sequential one.  Result valid in every lane.
__device__ __forceinline__ double warp_ordered_row_sum(const int64_t *ptr, const int32_t *cols,
                                                       const double *v, int i, int lane) {
    double s = 0.0;
    const int64_t b = ptr[i], e = ptr[i + 1];
    for (int64_t p0 = b; p0 < e; p0 += 32) {
        const int64_t p = p0 + lane;
        const double vj = (p < e) ? v[cols[p]] : 0.0;
        unsigned nz = __ballot_sync(0xffffffffu, vj != 0.0);
        while (nz) {
            const int src = __ffs(nz) - 1;
            nz &= nz - 1;
            s = __dadd_rn(s, __shfl_sync(0xffffffffu, vj, src));
        }
    }
    return s;
}

// Column scales for signals that are not dissociated (Sec. 4.3.3): one
// i.i.d. scale per column, uniform on [1, 2) to a grid of 2^-20 -- 1 plus the
// top 20 bits of the first draw of the column's SplitMix64 stream, times
// 2^-20 (exact in binary64).
__global__ void k_column_scales(int n, uint64_t seed, double *s) {
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x) {
        uint64_t state = seed + (uint64_t)(j + 1) * 0xd1b54a32d192ed03ull;
        const uint64_t k = splitmix64(state) >> 44;
        s[j] = __dadd_rn(1.0, (double)k * 0x1p-20);
    }
}

// y = A diag(s) x: the row's nonzero products s_j x_j (each rounded once),
// added in ascending j from +0.0 by the whole warp.
__global__ void k_measure_scaled(int m, const int64_t *ptr, const int32_t *cols,
                                 const double *sc, const double *x, double *y) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += warps) {
        double s = 0.0;
        const int64_t b = ptr[i], e = ptr[i + 1];
        for (int64_t p0 = b; p0 < e; p0 += 32) {
            const int64_t p = p0 + lane;
            const int c = (p < e) ? cols[p] : 0;
            const double vj = (p < e) ? __dmul_rn(sc[c], x[c]) : 0.0;
            unsigned nz = __ballot_sync(0xffffffffu, vj != 0.0);
            while (nz) {
                const int src = __ffs(nz) - 1;
                nz &= nz - 1;
                s = __dadd_rn(s, __shfl_sync(0xffffffffu, vj, src));
            }
        }
        if (lane == 0) y[i] = s;
    }
}

// x_j = z_j / s_j (the decode of a column-scaled measurement is z = s . x).
// Most z_j are zero, and a zero over a scale that is neither zero nor NaN is
// the zero whose sign is the product of theirs: no binary64 division (they
// run at a 64th of the integer rate here: 10.1 us instead of 3.6 us at n =
// 200003).
__global__ void k_unscale(int n, const double *sc, const double *z, double *x) {
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n;
         j += (long long)gridDim.x * blockDim.x) {
        const double zj = z[j], sj = sc[j];
        const unsigned long long zb = (unsigned long long)__double_as_longlong(zj),
                                 sb = (unsigned long long)__double_as_longlong(sj);
        const unsigned long long mag = sb << 1;
        if ((zb << 1) == 0ull && mag != 0ull && mag <= 0xffe0000000000000ull)
            x[j] = __longlong_as_double((long long)((zb ^ sb) & 0x8000000000000000ull));
        else
            x[j] = __ddiv_rn(zj, sj);
    }
}

__global__ void k_measure(int m, const int64_t *ptr, const int32_t *cols, const double *x,
                          double *y) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += warps) {
        const double s = warp_ordered_row_sum(ptr, cols, x, i, lane);
        if (lane == 0) y[i] = s;
    }
}

// ---- sparse x -------------------------------------------------------------
//
// The signals measured are sparse (k of n entries), and a row sum skips zero
// entries, so almost every gather of x is for nothing.  k_mark_nonzeros
// first notes which blocks of 2^shift columns hold a nonzero (the product
// s_j x_j for the scaled measurement), a bit each, in y's own memory;
// k_measure_marked brings the bits into shared memory -- every CTA does,
// before any of them stores a row of y (cooperative launch) -- and gathers
// only where they are set.  The columns of the rows then stream at the
// memory's rate: at n = 2^24, m = 16777, d = 9, k = 839 the 151 M gathers of
// 32-byte sectors from 134 MB took 604 us.

// A value of the measured vector: x_j, or s_j x_j rounded once.
template <bool kScaled>
__device__ __forceinline__ double measured_value(const double *sc, const double *x, long long j) {
    return kScaled ? __dmul_rn(__ldg(sc + j), __ldg(x + j)) : __ldg(x + j);
}

// Bit b of `bits`: columns [b 2^shift, (b + 1) 2^shift) hold a nonzero.  A
// warp makes whole words: 32 columns at a time, coalesced.
//
// A dense x is not marked: every block looks at the same sample, eight
// stretches of 32 columns spread over x, and when more than kMarkDense of
// them hold a nonzero the word behind the bits says so and the rows gather
// everything.  The sample decides the way only, never the result.  Marks pay
// below ~2 % of nonzeros; beyond, the lines below hold gathering every entry a
// warp a row, marks, and the unmarked rows here, in us:
//   n = 2^20, m = 10486, d = 7:   1 % 50, 47, -;  5 % 59, 70, 65;  10 % 86, 96, 89
//   n = 2^23, m = 2^16, d = 7:   10 % 511, 543, 522;  100 % 3726, 3803, 3781
//   n = 2^24, m = 16777, d = 9:  10 % 1339, 1321, 1279;  100 % 9697, 9819, 9776
// (the first has no second launch).  Tried: a dense x measured a warp a row by
// the marking blocks, which the GPU holds all at once: 1545 us instead of 1279
// in the last line, its rows being shared out less evenly.  A sample of 1024
// single columns cost every x 3-6 us.
constexpr int kMarkThreads = 256;
constexpr int kMarkDense = 5;
template <bool kScaled>
__global__ void __launch_bounds__(kMarkThreads)
k_mark_nonzeros(int n, int shift, const double *sc, const double *x, unsigned *bits) {
    const int lane = threadIdx.x & 31;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long words = (((long long)n - 1) >> shift) / 32 + 1;
    const long long at =
        (long long)__umulhi((threadIdx.x >> 5) * 0x9e3779b9u, (unsigned)n) + lane;
    const bool dense = __syncthreads_count(at < n && measured_value<kScaled>(sc, x, at) != 0.0) >
                       kMarkDense;
    if (blockIdx.x == 0 && threadIdx.x == 0) bits[words] = dense;
    if (dense) return;
    for (long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < words;
         w += warps) {
        const long long c0 = w << (shift + 5);
        unsigned word = 0;
#pragma unroll 8
        for (int u = 0; u < (1 << shift); ++u) {  // 32 columns each
            const long long j = c0 + 32 * u + lane;
            const bool nz = j < n && measured_value<kScaled>(sc, x, j) != 0.0;
            const unsigned bal = __ballot_sync(0xffffffffu, nz);
            // these 32 columns belong to 32 >> shift bits (one from shift 5 on)
            if (shift == 0) {
                word = bal;
            } else if (bal) {
                const int per = shift < 5 ? 32 >> shift : 1;
                for (int b = 0; b < per; ++b) {
                    const unsigned part =
                        shift < 5 ? (bal >> (b << shift)) & ((1u << (1 << shift)) - 1u) : bal;
                    if (part) word |= 1u << (shift < 5 ? u * per + b : u >> (shift - 5));
                }
            }
        }
        if (lane == 0) bits[w] = word;
    }
}

// A warp takes the CTA's rows a few at a time (`batch` consecutive ones, so
// that short rows fill its loads too) and streams their columns; set bits
// are looked up in order, so a row's nonzero values are added in ascending
// j from +0.0, as in warp_ordered_row_sum.
constexpr int kMarkBlock = 1024;
constexpr int kMarkUnroll = 8;  // (12 and 16: 2 and 13 % slower)
template <bool kScaled>
__global__ void __launch_bounds__(kMarkBlock)
k_measure_marked(int m, int shift, int words, int batch, const int64_t *ptr, const int32_t *cols,
                 const double *sc, const double *x, double *y) {
    extern __shared__ unsigned bits[];
    __shared__ int next;
    const unsigned *src = reinterpret_cast<const unsigned *>(y);
    const bool dense = __ldcg(src + words) != 0;
    for (int w = threadIdx.x; w < words; w += kMarkBlock) bits[w] = dense ? ~0u : __ldcg(src + w);
    const int lane = threadIdx.x & 31;
    const int r0 = (int)((long long)m * blockIdx.x / gridDim.x);
    const int r1 = (int)((long long)m * (blockIdx.x + 1) / gridDim.x);
    if (threadIdx.x == 0) next = r0;
    cooperative_groups::this_grid().sync();
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(&next, batch);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= r1) break;
        const int rows = min(batch, r1 - i);  // at most 32: lane l keeps the end of row i + l
        const int64_t b = __ldg(ptr + i);
        const int64_t mine = __ldg(ptr + i + 1 + min(lane, rows - 1));
        const int64_t e = __shfl_sync(0xffffffffu, mine, rows - 1);
        int row = 0;
        int64_t row_end = __shfl_sync(0xffffffffu, mine, 0);
        double s = 0.0, out = 0.0;  // lane l: the finished sum of row i + l
        int c[kMarkUnroll];
#pragma unroll
        for (int u = 0; u < kMarkUnroll; ++u) {
            const int64_t p = b + 32 * u + lane;
            c[u] = p < e ? __ldcs(cols + p) : -1;
        }
        for (int64_t p0 = b; p0 < e; p0 += 32 * kMarkUnroll) {
            int cn[kMarkUnroll];
#pragma unroll
            for (int u = 0; u < kMarkUnroll; ++u) {
                const int64_t p = p0 + 32 * (kMarkUnroll + u) + lane;
                cn[u] = p < e ? __ldcs(cols + p) : -1;
            }
            unsigned hit = 0;
#pragma unroll
            for (int u = 0; u < kMarkUnroll; ++u) {
                const unsigned blk = (unsigned)max(c[u], 0) >> shift;
                hit |= (c[u] >= 0 ? (bits[blk >> 5] >> (blk & 31)) & 1u : 0u) << u;
            }
            if (__any_sync(0xffffffffu, hit)) {
                constexpr int kV = 4;  // gathers in flight
#pragma unroll
                for (int u0 = 0; u0 < kMarkUnroll; u0 += kV) {
                    double v[kV];
#pragma unroll
                    for (int u = 0; u < kV; ++u)
                        v[u] = (hit >> (u0 + u)) & 1u ? measured_value<kScaled>(sc, x, c[u0 + u])
                                                      : 0.0;
#pragma unroll
                    for (int u = 0; u < kV; ++u) {
                        unsigned nz = __ballot_sync(0xffffffffu, v[u] != 0.0);
                        while (nz) {
                            const int at = __ffs(nz) - 1;
                            nz &= nz - 1;
                            const int64_t p = p0 + 32 * (u0 + u) + at;
                            while (p >= row_end) {  // rows that end before this entry
                                if (lane == row) out = s;
                                s = 0.0;
                                ++row;
                                row_end = __shfl_sync(0xffffffffu, mine, row);
                            }
                            s = __dadd_rn(s, __shfl_sync(0xffffffffu, v[u], at));
                        }
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kMarkUnroll; ++u) c[u] = cn[u];
        }
        if (lane == row) out = s;  // later rows hold no nonzero: 0.0
        if (lane < rows) y[i + lane] = out;
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

static thread_local char g_last_error[512] = "";

void set_last_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_last_error, sizeof(g_last_error), fmt, ap);
    va_end(ap);
}

int cuda_fail(cudaError_t e, const char *what) {
    set_last_error("%s: %s", what, cudaGetErrorString(e));
    return CCS_ECUDA;
}

int check_sizes(int32_t n, int32_t m, int32_t d) {
    if (n < 1 || m < 1 || d < 1 || d > kMaxD || d > m) {
        set_last_error("invalid sizes n=%d m=%d d=%d (need n,m >= 1, 1 <= d <= min(m, %d))",
                       n, m, d, kMaxD);
        return CCS_EINVAL;
    }
    if ((long long)n * d >= (1ll << 31)) {
        set_last_error("n*d = %lld exceeds the int32 edge index range", (long long)n * d);
        return CCS_EINVAL;
    }
    return CCS_OK;
}

int check_aligned(const char *who, const char *what, const void *p, unsigned align) {
    if (reinterpret_cast<uintptr_t>(p) % align) {
        set_last_error("%s: %s is not on a %u-byte boundary", who, what, align);
        return CCS_EINVAL;
    }
    return CCS_OK;
}

int check_problem_arrays(const char *who, const int32_t *csc_rows, const int64_t *csr_ptr,
                         const int32_t *csr_cols, const double *y, const double *x_hat,
                         const double *r, const int64_t *r0_hist) {
    int rc;
    if ((rc = check_aligned(who, "csc_rows", csc_rows, 16))) return rc;
    if ((rc = check_aligned(who, "csr_ptr", csr_ptr, 8))) return rc;
    if ((rc = check_aligned(who, "csr_cols", csr_cols, 4))) return rc;
    if ((rc = check_aligned(who, "y", y, 8))) return rc;
    if ((rc = check_aligned(who, "x_hat", x_hat, 8))) return rc;
    if ((rc = check_aligned(who, "r", r, 8))) return rc;
    return check_aligned(who, "r0_hist", r0_hist, 8);
}

static size_t make_expander_ws(int32_t n, int32_t m) {
    (void)n;
    const size_t nblocks = ((size_t)m + kScanBlock - 1) / kScanBlock;
    return align_up((size_t)m * 4, 256) + align_up(nblocks * 8, 256) + 256;
}

static int grid_for(long long work, int block) {
    long long g = (work + block - 1) / block;
    if (g > 152ll * 32) g = 152ll * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace ccs

using namespace ccs;

extern "C" {

const char *ccs_last_error(void) { return g_last_error; }

int ccs_version(void) { return 10000; }

const char *ccs_status_string(int status) {
    switch (status) {
        case CCS_OK: return "CCS_OK";
        case CCS_EINVAL: return "CCS_EINVAL";
        case CCS_ENOMEM: return "CCS_ENOMEM";
        case CCS_ECUDA: return "CCS_ECUDA";
        case CCS_ETIMEOUT: return "CCS_ETIMEOUT";
        case CCS_EBUDGET: return "CCS_EBUDGET";
        case CCS_EBUSY: return "CCS_EBUSY";
        default: return "CCS_E?";
    }
}

void ccs_params_init(ccs_params *p) {
    if (!p) return;
    p->alpha = 2;
    p->max_iter = 100;
    p->score_mode = CCS_SCORE_L0_DECREASE;
    p->engine = CCS_ENGINE_AUTO;
    p->watchdog_ms = 0;
    p->debug_flags = 0;
    p->schedule = 0;
    p->shifted = 0;
}

size_t ccs_workspace_size(int32_t op, int32_t n, int32_t m, int32_t d) {
    if (check_sizes(n, m, d) != CCS_OK) return 0;
    if (op == CCS_OP_MAKE_EXPANDER) return make_expander_ws(n, m);
    if (op == CCS_OP_DECODE) return engine_header_bytes(1) + decode_ws_layout(n, m, nullptr, nullptr);
    return 0;
}

}  // extern "C"

namespace ccs {

// How (n, m, d) is drawn and transposed.
struct ExpanderPlan {
    int sms;
    int groups;             // > 0: grouped construction
    int row_bits, col_bits;
    int group_cap;          // entries a group is not expected to pass
    int buckets, shift;     // of the group sort
    int deal_per;           // entries a thread of the deal takes at a time
    size_t draw_smem, deal_smem, sort_smem;
    // otherwise:
    int rank_shift;         // > 0: ranks ride above this bit of the row indices
};

// Entries that a row (or a group of rows) with `mean` of them on average is
// not expected to pass in a uniform draw: seven standard deviations more.
static int likely_most(double mean, long long edges) {
    return (int)fmin(fmin(mean + 7.0 * sqrt(mean) + 8.0, (double)edges), 2147483647.0);
}

static int bits_for(long long values) {  // of an index below `values`
    int b = 0;
    while (((values - 1) >> b) != 0) ++b;
    return b;
}

static int expander_plan(int32_t n, int32_t m, int32_t d, ExpanderPlan &pl) {
    const long long edges = (long long)n * d;
    const double mean = (double)edges / m;
    int dev = 0, optin = 0;
    CCS_CUDA_TRY(cudaGetDevice(&dev));
    CCS_CUDA_TRY(cudaDeviceGetAttribute(&pl.sms, cudaDevAttrMultiProcessorCount, dev));
    CCS_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int row_bits = m > 1 ? bits_for(m) : 1;
    const long long likely = std::min(likely_most(mean, edges), kMaxSortRow);
    pl.rank_shift = m > kRankedRows && (likely >> (32 - row_bits)) == 0 ? row_bits : 0;

    // groups of up to kGroupEntries entries, and enough of them for every SM
    pl.groups = 0;
    pl.col_bits = n > 1 ? bits_for(n) : 1;
    const double target = fmin((double)kGroupEntries, fmax((double)edges / (2 * pl.sms), 1024.0));
    int rb = 0;
    while (rb < kMaxGroupRowBits && rb + 1 + pl.col_bits <= 32 && mean * (2 << rb) <= target &&
           (1ll << rb) < m)
        ++rb;
    const long long groups = ((long long)m + (1ll << rb) - 1) >> rb;
    pl.row_bits = rb;
    pl.group_cap = likely_most(mean * (1 << rb), edges);
    const double likely_row = mean + 10.0 * sqrt(mean) + 10.0;
    if (groups > kMaxGroups || likely_row > kMaxSortRow) return CCS_OK;
    pl.buckets = 64;
    while ((pl.buckets < pl.group_cap / kBucketEntries && pl.buckets < 8192) || pl.buckets < 1 << rb)
        pl.buckets <<= 1;
    const uint64_t span = ((uint64_t)1 << pl.col_bits) << rb;
    while ((uint64_t)pl.buckets > span) pl.buckets >>= 1;
    pl.shift = 0;
    while ((span >> pl.shift) > (uint64_t)pl.buckets) ++pl.shift;
    pl.draw_smem = ((size_t)kDrawBlock * d + groups) * 4;
    pl.sort_smem = ((size_t)pl.buckets + pl.group_cap) * 4;
    const long long share = (edges + (long long)pl.sms * kDealBlock - 1) / ((long long)pl.sms * kDealBlock);
    pl.deal_per = (int)(share < 1 ? 1 : (share > kDealPer ? kDealPer : share));
    pl.deal_smem = (size_t)groups * 8 + (size_t)kDealBlock * pl.deal_per * 6;
    if (pl.draw_smem > (size_t)optin || pl.deal_smem + 256 > (size_t)optin ||
        pl.sort_smem + 256 > (size_t)optin)
        return CCS_OK;
    pl.groups = (int)groups;
    return CCS_OK;
}

// Sort every CSR row of at most `cap` columns, enqueued on `s`.  Rows of at
// most kWarpSortCap columns: a warp a row, in registers; longer ones a block
// a row.
static int sort_rows(int32_t n, int32_t m, int cap, const int64_t *csr_ptr, int32_t *csr_cols,
                     cudaStream_t s) {
    if (cap <= kWarpSortCap) {
        int size = 32;
        while (size < cap) size <<= 1;
        const int threads = 256;
        const int grid = grid_for((long long)m * 32, threads);
        switch (size) {
            case 32: k_sort_rows_warp<1><<<grid, threads, 0, s>>>(m, csr_ptr, csr_cols); break;
            case 64: k_sort_rows_warp<2><<<grid, threads, 0, s>>>(m, csr_ptr, csr_cols); break;
            case 128: k_sort_rows_warp<4><<<grid, threads, 0, s>>>(m, csr_ptr, csr_cols); break;
            case 256: k_sort_rows_warp<8><<<grid, threads, 0, s>>>(m, csr_ptr, csr_cols); break;
            default: k_sort_rows_warp<16><<<grid, threads, 0, s>>>(m, csr_ptr, csr_cols); break;
        }
    } else {
        int buckets = 64;
        while (buckets < cap / 8 && buckets < 4096) buckets <<= 1;
        int shift = 0;
        while ((long long)(n - 1) >> shift >= buckets) ++shift;
        const size_t smem = ((size_t)cap + buckets) * 4;
        CCS_CUDA_TRY(cudaFuncSetAttribute(k_sort_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)((kMaxSortRow + 4096) * 4)));
        const int grid = m < 152 * 16 ? m : 152 * 16;
        k_sort_rows<<<grid, kSortBlock, smem, s>>>(m, cap, shift, buckets, csr_ptr, csr_cols);
    }
    CCS_CUDA_TRY(cudaGetLastError());
    return CCS_OK;
}

// The workspace: row degrees, block totals of their scan, the largest degree.
struct ExpanderWs {
    int32_t *deg;
    int64_t *sums;
    int *max_deg;
    int nblocks;
    size_t bytes;
};

static ExpanderWs expander_ws(int32_t m, void *ws) {
    char *base = static_cast<char *>(ws);
    ExpanderWs w;
    w.nblocks = (int)(((long long)m + kScanBlock - 1) / kScanBlock);
    const size_t sums = align_up((size_t)m * 4, 256);
    const size_t top = sums + align_up((size_t)w.nblocks * 8, 256);
    w.deg = reinterpret_cast<int32_t *>(base);
    w.sums = reinterpret_cast<int64_t *>(base + sums);
    w.max_deg = reinterpret_cast<int *>(base + top);
    w.bytes = top + sizeof(int);
    return w;
}

// Lets launches of `fn` use `bytes` of shared memory.  The attribute belongs to
// the kernel, not to the call: it is raised to the device's limit and never
// lowered, so threads drawing matrices of different sizes do not meet.
static int allow_smem(const void *fn, size_t bytes) {
    int dev = 0;
    CCS_CUDA_TRY(cudaGetDevice(&dev));
    if (max_dynamic_smem(dev, fn) >= bytes) return CCS_OK;
    set_last_error("ccs_make_expander: a kernel cannot use %zu bytes of shared memory", bytes);
    return CCS_ECUDA;
}

// The whole construction, for one d.
template <int D>
static int expander_build(int32_t n, int32_t m, uint64_t seed, int32_t *csc_rows,
                          int64_t *csr_ptr, int32_t *csr_cols, const ExpanderWs &w,
                          const ExpanderPlan &pl, cudaStream_t s) {
    const long long edges = (long long)n * D;
    CCS_CUDA_TRY(cudaMemsetAsync(w.deg, 0, w.bytes, s));
    if (pl.groups) {
        int rc;
        if ((rc = allow_smem((const void *)k_draw_columns<D>, pl.draw_smem)) ||
            (rc = allow_smem((const void *)k_deal_entries<D>, pl.deal_smem)) ||
            (rc = allow_smem((const void *)k_sort_groups, pl.sort_smem)))
            return rc;
        const int draw_grid = (int)std::min(((long long)n + kDrawBlock - 1) / kDrawBlock, 3ll * pl.sms);
        k_draw_columns<D><<<draw_grid, kDrawBlock, pl.draw_smem, s>>>(n, m, seed, pl.row_bits,
                                                                     pl.groups, csc_rows, w.deg);
        k_scan_groups<<<1, kDealBlock, 0, s>>>(pl.groups, w.deg);
        const long long turns = (edges + (long long)kDealBlock * pl.deal_per - 1) /
                                ((long long)kDealBlock * pl.deal_per);
        k_deal_entries<D><<<(int)std::min(turns, (long long)pl.sms), kDealBlock, pl.deal_smem, s>>>(
            (uint32_t)edges, pl.row_bits, pl.col_bits, pl.groups, pl.deal_per, csc_rows, w.deg,
            csr_cols);
        k_sort_groups<<<std::min(pl.groups, 4 * pl.sms), kGroupBlock, pl.sort_smem, s>>>(
            m, pl.groups, pl.row_bits, pl.col_bits, pl.shift, pl.buckets, pl.group_cap, w.deg,
            csr_ptr, csr_cols, w.max_deg);
        CCS_CUDA_TRY(cudaGetLastError());
        return CCS_OK;
    }
    k_generate_columns<D><<<(n + kGenBlock - 1) / kGenBlock, kGenBlock, 0, s>>>(
        n, m, seed, pl.rank_shift, csc_rows, w.deg);
    k_scan_local<<<w.nblocks, kScanBlock, 0, s>>>(m, w.deg, csr_ptr, w.sums, w.max_deg);
    const bool scanned = w.nblocks > kScanBlock;
    if (scanned) k_scan_totals<<<1, kScanBlock, 0, s>>>(w.nblocks, w.sums);
    k_scan_add<<<w.nblocks, kScanBlock, 0, s>>>(m, csr_ptr, w.sums, scanned);
    CCS_CUDA_TRY(cudaGetLastError());
    if (pl.rank_shift) {
        k_place_ranked<D><<<grid_for((edges + 3) / 4, 256), 256, 0, s>>>(
            edges, pl.rank_shift, csc_rows, csr_ptr, csr_cols);
    } else {
        CCS_CUDA_TRY(cudaMemsetAsync(w.deg, 0, (size_t)m * 4, s));
        k_scatter_cols<<<grid_for(edges, 256), 256, 0, s>>>(n, D, csc_rows, csr_ptr, w.deg,
                                                            csr_cols);
    }
    CCS_CUDA_TRY(cudaGetLastError());
    return CCS_OK;  // the rows are sorted once the longest one is known
}

typedef int (*build_fn)(int32_t, int32_t, uint64_t, int32_t *, int64_t *, int32_t *,
                        const ExpanderWs &, const ExpanderPlan &, cudaStream_t);
static build_fn expander_builder(int d) {
    static const build_fn fns[kMaxD] = {
        expander_build<1>,  expander_build<2>,  expander_build<3>,  expander_build<4>,
        expander_build<5>,  expander_build<6>,  expander_build<7>,  expander_build<8>,
        expander_build<9>,  expander_build<10>, expander_build<11>, expander_build<12>,
        expander_build<13>, expander_build<14>, expander_build<15>, expander_build<16>};
    return fns[d - 1];
}

// The expander's construction up to the sort of single rows, enqueued on `s`.
// *max_deg_dev receives the device address of the largest row degree, which
// expander_finish needs on the host.
// Arguments already checked.
int expander_build_async(int32_t n, int32_t m, int32_t d, uint64_t seed, int32_t *csc_rows,
                         int64_t *csr_ptr, int32_t *csr_cols, void *ws, cudaStream_t s,
                         int **max_deg_dev) {
    ExpanderPlan pl;
    int rc = expander_plan(n, m, d, pl);
    if (rc) return rc;
    const ExpanderWs w = expander_ws(m, ws);
    *max_deg_dev = w.max_deg;
    return expander_builder(d)(n, m, seed, csc_rows, csr_ptr, csr_cols, w, pl, s);
}

// What is left once the largest row degree is known: nothing after a grouped
// construction, as a rule; else the sort of the rows, sized by the longest
// one (sizing it beforehand by what rows are unlikely to pass took up to twice
// as long: n = 2^25 + 1, m = 2^20, d = 1 0.58 ms against 0.27; and where no
// row holds two columns there is nothing to sort: n = 1003, m = 2^29, d = 3
// 26 ms spared).  CCS_EINVAL when a row is longer than the on-chip sort
// takes.  Enqueued on `s`; *again: whether anything was.
int expander_finish(int32_t n, int32_t m, int32_t d, uint64_t seed, int32_t *csc_rows,
                    int64_t *csr_ptr, int32_t *csr_cols, void *ws, int host_max, cudaStream_t s,
                    bool *again) {
    *again = false;
    ExpanderPlan pl;
    int rc = expander_plan(n, m, d, pl);
    if (rc) return rc;
    if (pl.groups && host_max == 0x7fffffff) {
        // a group that did not fit on chip: build again row by row
        const ExpanderWs w = expander_ws(m, ws);
        pl.groups = 0;
        if ((rc = expander_builder(d)(n, m, seed, csc_rows, csr_ptr, csr_cols, w, pl, s))) return rc;
        CCS_CUDA_TRY(cudaMemcpyAsync(&host_max, w.max_deg, sizeof(int), cudaMemcpyDeviceToHost, s));
        CCS_CUDA_TRY(cudaStreamSynchronize(s));
        *again = true;
    }
    if (host_max > kMaxSortRow) {
        set_last_error("ccs_make_expander: a row has %d columns (limit %d)", host_max,
                       kMaxSortRow);
        return CCS_EINVAL;
    }
    if (pl.groups || host_max <= 1) return CCS_OK;
    *again = true;
    if (pl.rank_shift && ((long long)host_max >> (32 - pl.rank_shift)) != 0) {
        // ranks that did not fit their bits: draw again without them
        pl.rank_shift = 0;
        if ((rc = expander_builder(d)(n, m, seed, csc_rows, csr_ptr, csr_cols,
                                      expander_ws(m, ws), pl, s)))
            return rc;
    }
    return sort_rows(n, m, host_max, csr_ptr, csr_cols, s);
}

// y = A x or y = A diag(sc) x, enqueued on `s`: through the nonzero marks
// when the matrix is large, else by gathering every entry.
template <bool kScaled>
static int measure_rows(int32_t n, int32_t m, int32_t d, const int64_t *csr_ptr,
                        const int32_t *csr_cols, const double *sc, const double *x, double *y,
                        cudaStream_t s) {
    const long long edges = (long long)n * d;
    if (edges >= kMarkedMinEntries ||
        (edges >= kMarkedMinLongRows && edges / m >= kMarkedLongRow)) {
        int dev = 0, sms = 0, coop = 0;
        CCS_CUDA_TRY(cudaGetDevice(&dev));
        CCS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        CCS_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        // as many bits as y (64 m, less a word) and shared memory hold
        const long long room = std::min(64ll * m - 32, (long long)kMarkBytes * 8);
        int shift = 0;
        while (((((long long)n - 1) >> shift) / 32 + 1) * 32 > room) ++shift;
        const int words = (int)((((long long)n - 1) >> shift) / 32 + 1);
        if (coop && shift <= kMarkMaxShift) {
            k_mark_nonzeros<kScaled><<<sms * 8, kMarkThreads, 0, s>>>(n, shift, sc, x,
                                                             reinterpret_cast<unsigned *>(y));
            CCS_CUDA_TRY(cudaGetLastError());
            const size_t smem = (size_t)words * 4;
            CCS_CUDA_TRY(cudaFuncSetAttribute(k_measure_marked<kScaled>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              kMarkBytes));
            int batch = (int)std::max(1ll, std::min(32ll, 512ll * m / edges));
            int words_arg = words, shift_arg = shift;
            void *args[] = {&m, &shift_arg, &words_arg, &batch, &csr_ptr, &csr_cols, &sc, &x, &y};
            CCS_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_measure_marked<kScaled>,
                                                     dim3(sms), dim3(kMarkBlock), args, smem, s));
            return CCS_OK;
        }
    }
    const long long threads = (long long)m * 32;
    if (kScaled)
        k_measure_scaled<<<grid_for(threads, 256), 256, 0, s>>>(m, csr_ptr, csr_cols, sc, x, y);
    else
        k_measure<<<grid_for(threads, 256), 256, 0, s>>>(m, csr_ptr, csr_cols, x, y);
    CCS_CUDA_TRY(cudaGetLastError());
    return CCS_OK;
}

}  // namespace ccs

extern "C" {

int ccs_make_expander(int32_t n, int32_t m, int32_t d, uint64_t seed, int32_t *csc_rows,
                      int64_t *csr_ptr, int32_t *csr_cols, void *ws, size_t ws_bytes,
                      ccs_stream_t stream) {
    int rc = check_sizes(n, m, d);
    if (rc) return rc;
    if (!csc_rows || !csr_ptr || !csr_cols || !ws) {
        set_last_error("ccs_make_expander: null pointer argument");
        return CCS_EINVAL;
    }
    if (ws_bytes < make_expander_ws(n, m)) {
        set_last_error("ccs_make_expander: workspace %zu < %zu bytes", ws_bytes,
                       make_expander_ws(n, m));
        return CCS_ENOMEM;
    }
    if ((rc = check_problem_arrays("ccs_make_expander", csc_rows, csr_ptr, csr_cols, nullptr,
                                   nullptr, nullptr, nullptr)) ||
        (rc = check_aligned("ccs_make_expander", "ws", ws, kWorkspaceAlign)))
        return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int *max_deg = nullptr;
    if ((rc = expander_build_async(n, m, d, seed, csc_rows, csr_ptr, csr_cols, ws, s, &max_deg)))
        return rc;
    int host_max = 0;
    CCS_CUDA_TRY(cudaMemcpyAsync(&host_max, max_deg, sizeof(int), cudaMemcpyDeviceToHost, s));
    CCS_CUDA_TRY(cudaStreamSynchronize(s));
    bool again = false;
    if ((rc = expander_finish(n, m, d, seed, csc_rows, csr_ptr, csr_cols, ws, host_max, s, &again)))
        return rc;
    if (again) CCS_CUDA_TRY(cudaStreamSynchronize(s));
    return CCS_OK;
}

int ccs_measure(int32_t n, int32_t m, int32_t d, const int64_t *csr_ptr,
                const int32_t *csr_cols, const double *x, double *y, ccs_stream_t stream) {
    int rc = check_sizes(n, m, d);
    if (rc) return rc;
    if (!csr_ptr || !csr_cols || !x || !y) {
        set_last_error("ccs_measure: null pointer argument");
        return CCS_EINVAL;
    }
    if ((rc = check_problem_arrays("ccs_measure", nullptr, csr_ptr, csr_cols, y, nullptr,
                                   nullptr, nullptr)) ||
        (rc = check_aligned("ccs_measure", "x", x, 8)))
        return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return measure_rows<false>(n, m, d, csr_ptr, csr_cols, nullptr, x, y, s);
}

int ccs_column_scales(int32_t n, uint64_t seed, double *scales, ccs_stream_t stream) {
    if (n < 1 || !scales) {
        set_last_error("ccs_column_scales: n < 1 or null output");
        return CCS_EINVAL;
    }
    if (int rc = check_aligned("ccs_column_scales", "s", scales, 8)) return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_column_scales<<<grid_for(n, 256), 256, 0, s>>>(n, seed, scales);
    CCS_CUDA_TRY(cudaGetLastError());
    return CCS_OK;
}

int ccs_measure_scaled(int32_t n, int32_t m, int32_t d, const int64_t *csr_ptr,
                       const int32_t *csr_cols, const double *scales, const double *x,
                       double *y, ccs_stream_t stream) {
    int rc = check_sizes(n, m, d);
    if (rc) return rc;
    if (!csr_ptr || !csr_cols || !scales || !x || !y) {
        set_last_error("ccs_measure_scaled: null pointer argument");
        return CCS_EINVAL;
    }
    if ((rc = check_problem_arrays("ccs_measure_scaled", nullptr, csr_ptr, csr_cols, y, nullptr,
                                   nullptr, nullptr)) ||
        (rc = check_aligned("ccs_measure_scaled", "x", x, 8)) ||
        (rc = check_aligned("ccs_measure_scaled", "s", scales, 8)))
        return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return measure_rows<true>(n, m, d, csr_ptr, csr_cols, scales, x, y, s);
}

int ccs_unscale(int32_t n, const double *scales, const double *z, double *x,
                ccs_stream_t stream) {
    if (n < 1 || !scales || !z || !x) {
        set_last_error("ccs_unscale: n < 1 or null pointer argument");
        return CCS_EINVAL;
    }
    int rc;
    if ((rc = check_aligned("ccs_unscale", "s", scales, 8)) ||
        (rc = check_aligned("ccs_unscale", "z", z, 8)) ||
        (rc = check_aligned("ccs_unscale", "x", x, 8)))
        return rc;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_unscale<<<grid_for(n, 256), 256, 0, s>>>(n, scales, z, x);
    CCS_CUDA_TRY(cudaGetLastError());
    return CCS_OK;
}

}  // extern "C"
