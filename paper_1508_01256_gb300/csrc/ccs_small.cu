// ccs_small.cu -- Parallel-l0 (Alg. 2) on problems small enough for the shared
// memory of one thread-block cluster.
//
// A decode's iteration is short on a small problem, and the persistent
// engine (ccs_engine_kernel.cuh) spends it on latency: two barriers across
// the GPU, a copy of the fingerprints into every SM, gathers of r through L2
// (16 us an iteration at n = 4096 as at n = 200000).  Here a cluster of up to
// 8 CTAs keeps the whole state on chip for the length of the decode:
//   - each CTA holds the row indices of its part of the columns (16 bits
//     each, one array per position, so a warp reads consecutive words);
//   - every CTA holds all of r, its fingerprints, the changes of this
//     iteration and the touched flags; an accepted column updates all the
//     cluster's copies (distributed shared memory);
//   - one hardware cluster barrier an iteration, one more under the ordered
//     residual, whose row sums are shared out, and one more when a CTA accepts
//     more columns than its list holds: every CTA then brings its copy of r up
//     to date and evaluates the stop rule by itself, so all copies have to end
//     with the same bits.
// x_hat, the contributor records of the ordered residual and the CSR rows
// stay in global memory; few columns are accepted.
//
// Clusters take the problems of a launch one after another, so a batch's
// small problems run side by side, each at its own pace (a server's rounds of
// two iterations stay with the engine: loading a problem's rows each round
// cost what it gave, 17 problems of n = 10000-30000 1.55 ms against 1.45, 24
// of n = 4096-500000 7.1-8.1 ms against 7.1-7.8).  The method, its
// order of operations and the residual forms are the engine's (see there):
// results are the same bits.
//
// Bound by latency: at n = 6378, m = 64, d = 7 an iteration takes 5.6 us
// (the engine: 15 us), of which the fingerprint test ~1, the exact score of
// the few queued columns with one read of x_hat ~2, the barrier ~1; at n =
// 54797, m = 548, d = 9 14 us, half of it the fingerprint test (two shared
// loads per row index, ~3.5-way bank conflicts in the second).  A decode of
// n = 4096, m = 410, d = 7: 39 us in the engine, 19 us here; 64 mixed
// problems, 8 of them past recovery: 4.3 ms with the engine alone, 2.7 ms.
// Tried: adding each accepted column to every copy with remote binary64
// atomics (60 us instead of 19 us for the first of these: a round trip each).
#include <cooperative_groups.h>
#include <mutex>

#include "ccs_device.cuh"

namespace ccs {

namespace cg = cooperative_groups;

constexpr int kSmallThreads = 1024;
constexpr int kSmallCluster = 8;        // CTAs of a cluster (the portable size)
constexpr int kSmallMaxM = 65535;       // rows fit 16 bits
constexpr size_t kSmallSmem = 216 << 10;  // shared memory a CTA's problem may take
// Entries per CTA below which a smaller cluster is taken.
constexpr long long kSmallPerCta = 4096;
// A problem decoded alone goes to the persistent engine from here on, which
// has 152 SMs for it (n = 15383, m = 4615, d = 11: 46 us against 70 us here;
// n = 35926, m = 1796, d = 11: 42 against 48; n = 12380, m = 124, d = 7: 72
// against 43).  In a batch the clusters run side by side.
constexpr long long kSmallAloneEntries = 300000;
constexpr int kSmallAloneM = 2560;
// Accepted columns a CTA sends to the others in an iteration; when there are
// more, the CTAs read one another's sums instead.
constexpr int kSmallList = 64;

struct SmallArgs {
    ProblemDev single;         // probs == nullptr
    const ProblemDev *probs;
    int P;
    int alpha, mode, max_iter, debug_flags, shifted;
    EngineSync *sync;
    ccs_result *dev_out;       // or null
    unsigned long long *stamps;  // phases of the first problem (or null)
};

// Updates of another CTA's shared memory: `local` is the place in this CTA's,
// `rank` the CTA of the cluster that holds the one meant.
__device__ __forceinline__ uint32_t cluster_addr(const void *local, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;"
        : "=r"(a)
        : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(local))), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_set(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_set(uint32_t a, unsigned long long v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_set(uint32_t a, unsigned v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_set(uint32_t a, uint16_t v) {
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory");
}

// A CTA's share of one problem in shared memory.  What exists once per
// iteration parity has its second half `m` (or the list's length) further on.
struct SmallSmem {
    double *r, *delta;     // m; 2 m: r, and its changes
    double *omega;         // 2 C kSmallList: accepted columns of every CTA: their omega,
    uint16_t *where;       // d times as many: and their d rows each
    uint16_t *fp, *over;   // m; m: rows whose sum needs the whole CSR row
    uint16_t *rows;        // d arrays of `pitch`: the rows of this CTA's columns
    uint16_t *queue;       // pitch: columns that may be accepted
    uint8_t *touched;      // 2 m
};

__host__ __device__ inline int small_pitch(int n, int C) { return ((n + C - 1) / C + 31) / 32 * 32; }

__host__ __device__ inline size_t small_smem(int n, int m, int d, int C, char *base,
                                             SmallSmem *S) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base + off;
        off += (bytes + 15) / 16 * 16;
        return p;
    };
    const size_t list = C > 1 ? 2 * (size_t)kSmallList * C : 0;
    char *r = take(8 * (size_t)m), *delta = take(16 * (size_t)m), *omega = take(8 * list);
    char *where = take(2 * d * list), *fp = take(2 * (size_t)m), *over = take(2 * (size_t)m);
    char *rows = take(2 * (size_t)d * small_pitch(n, C)), *queue = take(2 * (size_t)small_pitch(n, C));
    char *touched = take(2 * (size_t)m);
    if (S) {
        S->r = reinterpret_cast<double *>(r);
        S->delta = reinterpret_cast<double *>(delta);
        S->omega = reinterpret_cast<double *>(omega);
        S->where = reinterpret_cast<uint16_t *>(where);
        S->fp = reinterpret_cast<uint16_t *>(fp);
        S->over = reinterpret_cast<uint16_t *>(over);
        S->rows = reinterpret_cast<uint16_t *>(rows);
        S->queue = reinterpret_cast<uint16_t *>(queue);
        S->touched = reinterpret_cast<uint8_t *>(touched);
    }
    return off;
}

// Exact score of a column's values v, as exact_score_values, each pair of
// values compared once.
template <int DMAX>
__device__ __forceinline__ bool score_pairs(const unsigned long long (&v)[DMAX], int d, int alpha,
                                            int mode, unsigned long long *omega) {
    int cnt[DMAX];
    int c0 = 0;
#pragma unroll
    for (int t = 0; t < DMAX; ++t) {
        cnt[t] = 1;
        c0 += (t < d) & (v[t] == 0ull);
    }
#pragma unroll
    for (int a = 0; a < DMAX; ++a)
#pragma unroll
        for (int b = a + 1; b < DMAX; ++b) {
            const int e = (b < d) & (v[a] == v[b]);
            cnt[a] += e;
            cnt[b] += e;
        }
    int best = 0;
    unsigned long long bits = 0ull, key = ~0ull;
#pragma unroll
    for (int t = 0; t < DMAX; ++t) {
        const unsigned long long k = order_key(v[t]);
        const bool better = (t < d) && v[t] != 0ull && (cnt[t] > best || (cnt[t] == best && k < key));
        best = better ? cnt[t] : best;
        key = better ? k : key;
        bits = better ? v[t] : bits;
    }
    *omega = bits;
    return best > 0 && (mode == CCS_SCORE_COUNT ? best : best - c0) >= alpha;
}

// The exactness certificate of the incremental residual, as in the engine:
// while Y + deg (X + 2 R) < 2^min(e+51, 1023), with Y, X, R the largest
// |y_i|, |x_hat_j|, |r_i| and e the exponent of the lowest set bit over the
// nonzero y_i, every addition of the iteration is exact and none overflows.
// (A sum that overflows in one order and not in another would leave the
// CTAs' copies of r different.)
struct Certificate {
    double Y, deg, limit;  // limit < 0: always holds
};

__device__ __forceinline__ Certificate certificate_from(int grid_b, unsigned long long ymax,
                                                        int deg) {
    const int e = 1100 - grid_b;
    Certificate q;
    q.Y = __longlong_as_double((long long)ymax);
    q.deg = (double)deg;
    // y == 0: nothing is ever added
    q.limit = grid_b == 0 ? -1.0 : ldexp(1.0, min(e + 51, 1023));
    return q;
}

__device__ __forceinline__ bool exact_certified(int debug_flags, const Certificate &q, int it,
                                                unsigned long long xmax, unsigned long long rmax) {
    if ((debug_flags & kFlagOrdered) || ((debug_flags & kFlagSwitch) && it >= 2)) return false;
    const double R = __longlong_as_double((long long)rmax);
    const double X = __longlong_as_double((long long)xmax);
    return q.limit < 0.0 || q.Y + q.deg * (X + 2.0 * R) < q.limit;
}

// Bits of the largest of the warp's values (bits of non-negative doubles), in
// every lane: the high words' maximum, then the low words' among its holders.
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

// Counters shared by the CTA; those of the second group are written by the
// whole cluster.
struct SmallState {
    long long r0;
    unsigned long long rmax;      // max |r_i| (bits) of the current r
    unsigned long long xmax;      // bound of |x_hat| (bits) so far
    int gridb, deg, n_over;
    int it, status, rmode, empty_run, problem;
    Certificate cert;
    int queued;
    unsigned acc;                 // columns this CTA accepted
    unsigned long long xnew;      // largest |x_hat| (bits) it set
    // every CTA's acc and xnew, by iteration parity
    unsigned all_acc[2][kSmallCluster];
    unsigned long long all_xnew[2][kSmallCluster];
};

// One problem by the cluster, from its first iteration to its end.
template <int DMAX>
__device__ __forceinline__ void small_decode(const SmallArgs &a, const ProblemDev &P, SmallState &s,
                                             char *smem) {
    const cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kSmallThreads / 32;
    const int n = P.n, m = P.m, d = P.d;
    DecodeCtrl *const ctrl = P.ctrl;
    const int pitch = small_pitch(n, C);
    const int c0 = min(n, rank * pitch), cols = min(n, c0 + pitch) - c0;
    SmallSmem S;
    small_smem(n, m, d, C, smem, &S);

    // ---- state on chip; Alg. 2, first line ------------------------------
    if (tid == 0) {
        s.r0 = 0;
        s.rmax = 0;
        s.gridb = s.deg = s.n_over = 0;
        s.queued = 0;
        s.acc = 0;
        s.xnew = 0;
    }
    const int32_t *src = P.csc_rows + (size_t)c0 * d;
    for (int e = tid; e < cols * d; e += kSmallThreads) {
        const int j = e / d;
        S.rows[(e - j * d) * pitch + j] = (uint16_t)__ldg(src + e);
    }
    __syncthreads();
    int nz = 0, gridb = 0, deg = 0;
    unsigned long long mx = 0;
    for (int i = tid; i < m; i += kSmallThreads) {
        const double v = __ldg(P.y + i);
        const unsigned long long b = value_bits(v);
        S.r[i] = v;
        S.delta[i] = S.delta[m + i] = 0.0;
        S.touched[i] = S.touched[m + i] = 0;
        S.fp[i] = fingerprint16_of_bits(b);
        const unsigned long long mag = b & 0x7fffffffffffffffull;
        nz += mag != 0;
        mx = mag > mx ? mag : mx;
        if (mag) gridb = max(gridb, 1100 - lowbit_exponent(mag));
        deg = max(deg, (int)(__ldg(P.csr_ptr + i + 1) - __ldg(P.csr_ptr + i)));
        if (i % C == rank) P.slots[(size_t)i * kSlotRec] = 0;
    }
    for (int j = tid; j < cols; j += kSmallThreads) P.x_hat[c0 + j] = 0.0;
    nz = __reduce_add_sync(0xffffffffu, nz);
    mx = warp_max_bits(mx);
    gridb = __reduce_max_sync(0xffffffffu, gridb);
    deg = __reduce_max_sync(0xffffffffu, deg);
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&s.r0), (unsigned long long)nz);
        atomicMax(&s.rmax, mx);
        atomicMax(&s.gridb, gridb);
        atomicMax(&s.deg, deg);
    }
    __syncthreads();
    if (tid == 0) {
        s.it = s.empty_run = s.rmode = 0;
        s.xmax = 0;
        s.status = s.r0 == 0 ? CCS_CONVERGED : (a.max_iter == 0 ? CCS_MAX_ITER : kRunning);
        s.cert = certificate_from(s.gridb, s.rmax, s.deg);
        if (rank == 0 && P.r0_hist) P.r0_hist[0] = s.r0;
    }
    // Thread 0: the residual form of the next iteration.
    auto next_form = [&]() {
        if (s.rmode == 2) s.rmode = 1;
        else if (s.rmode == 0 &&
                 !exact_certified(a.debug_flags, s.cert, s.it, s.xmax, s.rmax))
            s.rmode = 2;
    };
    if (tid == 0 && s.status == kRunning) next_form();
    cl.sync();  // every CTA's copy is ready for the others' updates
    auto stamp = [&](int at) {
        if (a.stamps && tid == 0 && rank == 0 && s.problem == 0 && s.it < kMaxStampIters)
            a.stamps[at] = globaltimer();
    };
    stamp(0);

    while (s.status == kRunning) {
        const int it = s.it, par = it & 1;
        double *const delta = S.delta + (par ? m : 0);
        uint8_t *const touched = S.touched + (par ? m : 0);
        const int list = par * C * kSmallList;  // this parity's half of the lists
        const bool exact = s.rmode == 0;
        const int spos = a.shifted ? it % d : -1;
        if (s.rmode == 2) {
            // the columns already nonzero enter their rows' records
            for (int j = tid; j < cols; j += kSmallThreads) {
                const bool on = __ldcg(P.x_hat + c0 + j) != 0.0;
                P.in_slots[c0 + j] = on;
                if (on) {
                    int32_t rows[DMAX];
#pragma unroll
                    for (int t = 0; t < DMAX; ++t)
                        rows[t] = t < d ? S.rows[t * pitch + j] : 0;
                    enter_slots<DMAX>(P, c0 + j, rows, d);
                }
            }
        }

        stamp(kSubBase + 3 * it);

        // ---- score: the columns the fingerprints let through are queued, ----
        // then scored exactly on full warps
        for (int j0 = warp * 32; j0 < cols; j0 += kSmallThreads) {
            const int j = j0 + lane;
            const bool live = j < cols;
            unsigned f[DMAX];
            int nonzero = 0;
#pragma unroll
            for (int t = 0; t < DMAX; ++t) {
                f[t] = t < d && live ? S.fp[S.rows[t * pitch + j]] : 0u;
                nonzero += f[t] != 0u;
            }
            // no value occurs more often than its fingerprint
            const int need = a.mode == CCS_SCORE_COUNT ? a.alpha : a.alpha + (d - nonzero);
            bool pass = live && nonzero >= need;
            if (__any_sync(0xffffffffu, pass))
                pass = pass && (spos >= 0 || fp_pair_exists<DMAX>(f, d));
            const unsigned bal = __ballot_sync(0xffffffffu, pass);
            if (bal) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&s.queued, __popc(bal));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
                if (pass) S.queue[at] = (uint16_t)j;
            }
        }
        __syncthreads();
        stamp(kSubBase + 3 * it + 1);
        unsigned long long xnew = 0;
        for (int e = tid; e < s.queued; e += kSmallThreads) {
            const int j = S.queue[e];
            // read ahead of the score: most queued columns are accepted
            const double xj = __ldcg(P.x_hat + c0 + j);
            const uint8_t entered = exact ? (uint8_t)1 : __ldcg(P.in_slots + c0 + j);
            unsigned long long v[DMAX];
#pragma unroll
            for (int t = 0; t < DMAX; ++t)
                v[t] = t < d ? value_bits(S.r[S.rows[t * pitch + j]]) : 0ull;
            unsigned long long bits;
            if (!(spos >= 0
                      ? exact_score_shifted<DMAX>(v, d, spos, a.alpha, a.mode, &bits)
                      : score_pairs<DMAX>(v, d, a.alpha, a.mode, &bits)))
                continue;
            int32_t rows[DMAX];
#pragma unroll
            for (int t = 0; t < DMAX; ++t) rows[t] = t < d ? S.rows[t * pitch + j] : 0;
            const double omega = __longlong_as_double((long long)bits);
            const double xn = __dadd_rn(xj, omega);
            P.x_hat[c0 + j] = xn;
            if (exact) {
                const unsigned long long mag = value_bits(xn) & 0x7fffffffffffffffull;
                xnew = mag > xnew ? mag : xnew;
            } else if (!entered) {
                P.in_slots[c0 + j] = 1;
                enter_slots<DMAX>(P, c0 + j, rows, d);
            }
            // apply here, and let the other CTAs know
            const unsigned k = atomicAdd(&s.acc, 1u);
#pragma unroll
            for (int t = 0; t < DMAX; ++t)
                if (t < d) {
                    if (exact) atomicAdd(delta + rows[t], -omega);
                    touched[rows[t]] = 1;
                }
            if (k < (unsigned)kSmallList) {
                const int at = list + rank * kSmallList + (int)k;
                for (int q = 0; q < C; ++q) {
                    if (q == rank) continue;
                    cluster_set(cluster_addr(S.omega + at, q), omega);
                    const uint32_t where = cluster_addr(S.where + at * d, q);
#pragma unroll
                    for (int t = 0; t < DMAX; ++t)
                        if (t < d) cluster_set(where + 2 * t, (uint16_t)rows[t]);
                }
            }
        }
        xnew = warp_max_bits(xnew);
        if (lane == 0 && xnew) atomicMax(&s.xnew, xnew);
        __syncthreads();
        stamp(kSubBase + 3 * it + 2);
        if (tid < C) {
            cluster_set(cluster_addr(&s.all_acc[par][rank], tid), s.acc);
            cluster_set(cluster_addr(&s.all_xnew[par][rank], tid), s.xnew);
        }
        if (tid == 0) s.rmax = 0;
        cl.sync();
        stamp(1 + 2 * it);

        // ---- the other CTAs' accepted columns into this copy --------------
        const unsigned mine = lane < C ? s.all_acc[par][lane] : 0u;
        const unsigned total = __reduce_add_sync(0xffffffffu, mine);
        const bool listed = __all_sync(0xffffffffu, mine <= (unsigned)kSmallList);
        if (warp == 0) {
            const unsigned long long x =
                warp_max_bits(lane < C ? s.all_xnew[par][lane] : 0ull);
            if (lane == 0) {
                if (x > s.xmax) s.xmax = x;
                s.queued = 0;
                s.acc = 0;
                s.xnew = 0;
            }
        }
        if (listed) {
            const int q = warp % C;  // a share of the warps per source
            if (q != rank) {
                const int len = (int)s.all_acc[par][q] * d, at = list + q * kSmallList;
                for (int e = warp / C * 32 + lane; e < len; e += kSmallThreads / C) {
                    const int row = S.where[at * d + e];
                    if (exact) atomicAdd(delta + row, -S.omega[at + e / d]);
                    touched[row] = 1;
                }
            }
        } else {
            // too many to list: the others' sums, gathered in the arrays of
            // the other parity (which rest, all zero, in this iteration)
            double *const delta_next = S.delta + (par ? 0 : m);
            uint8_t *const touched_next = S.touched + (par ? 0 : m);
            for (int i = tid; i < m; i += kSmallThreads) {
                double sum = 0.0;
                uint8_t hit = 0;
                for (int q = 0; q < C; ++q) {
                    if (q == rank) continue;
                    if (exact) sum = __dadd_rn(sum, *cl.map_shared_rank(delta + i, q));
                    hit |= *cl.map_shared_rank(touched + i, q);
                }
                if (exact) delta_next[i] = sum;
                touched_next[i] = hit;
            }
            cl.sync();
            for (int i = tid; i < m; i += kSmallThreads) {
                // under the ordered residual `delta` belongs from here on to
                // the CTA that sums row i, which may already be storing to it
                if (exact) {
                    delta[i] = __dadd_rn(delta[i], delta_next[i]);
                    delta_next[i] = 0.0;
                }
                touched[i] |= touched_next[i];
                touched_next[i] = 0;
            }
        }
        __syncthreads();

        // ---- residual + ||r||_0 --------------------------------------------
        if (!exact) {
            // ordered sums: the touched rows are shared out over the
            // cluster, and each new r_i goes to every copy (in `delta`)
            for (int i0 = (warp * C + rank) * 32; i0 < m; i0 += kSmallThreads * C) {
                const int i = i0 + lane;
                if (i >= m || !touched[i]) continue;
                int js[kSlotRec];
                load_record(P, i, js);
                if (js[0] > kSlots) {
                    S.over[atomicAdd(&s.n_over, 1)] = (uint16_t)i;
                    continue;
                }
                const double v = __dsub_rn(__ldg(P.y + i), row_sum_from_record(P, i, js));
                for (int q = 0; q < C; ++q) cluster_set(cluster_addr(delta + i, q), v);
            }
            __syncthreads();
            for (int q = warp; q < s.n_over; q += kWarps) {
                const int i = S.over[q];
                const double v =
                    __dsub_rn(__ldg(P.y + i), warp_ordered_row_sum_flagged(P, i, lane));
                if (lane < C) cluster_set(cluster_addr(delta + i, lane), v);
            }
            cl.sync();
        }
        // every CTA brings its own copy up to date
        int change = 0;
        mx = 0;
        for (int i = tid; i < m; i += kSmallThreads) {
            double v = S.r[i];
            if (touched[i]) {
                const unsigned long long o = value_bits(v);
                touched[i] = 0;
                v = exact ? __dadd_rn(v, delta[i]) : delta[i];
                delta[i] = 0.0;
                const unsigned long long b = value_bits(v);
                if (!exact || b != o) {
                    S.r[i] = v;
                    S.fp[i] = fingerprint16_of_bits(b);
                }
                change += (b != 0ull) - (o != 0ull);
            }
            const unsigned long long mag = value_bits(v) & 0x7fffffffffffffffull;
            mx = mag > mx ? mag : mx;
        }
        change = __reduce_add_sync(0xffffffffu, change);
        mx = warp_max_bits(mx);
        if (lane == 0) {
            if (change)
                atomicAdd(reinterpret_cast<unsigned long long *>(&s.r0),
                          (unsigned long long)(long long)change);
            atomicMax(&s.rmax, mx);
        }
        __syncthreads();

        stamp(2 + 2 * it);
        // ---- stop rule, as in the engine --------------------------------
        if (tid == 0) {
            const bool empty = total == 0;
            s.n_over = 0;
            s.empty_run = empty ? s.empty_run + 1 : 0;
            if (empty && s.empty_run >= (a.shifted ? d : 1)) {
                s.status = CCS_STALLED;
            } else {
                s.it = it + 1;
                s.status = s.r0 == 0 ? CCS_CONVERGED
                                     : (it + 1 >= a.max_iter ? CCS_MAX_ITER : kRunning);
                if (rank == 0 && P.r0_hist) P.r0_hist[it + 1] = s.r0;
                if (s.status == kRunning) next_form();
            }
        }
        __syncthreads();
    }

    // ---- what outlives the launch --------------------------------------------
    for (int i = rank * kSmallThreads + tid; i < m; i += C * kSmallThreads)
        P.r[i] = S.r[i];
    if (rank == 0 && tid == 0) {
        ctrl->status = s.status;
        ctrl->iteration = s.it;
        ctrl->r0 = s.r0;
        ctrl->ordered = s.rmode != 0;
    }
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_small(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) char smem[];
    __shared__ ProblemDev P;
    __shared__ SmallState s;
    const cg::cluster_group cl = cg::this_cluster();
    const bool leader = cl.block_rank() == 0 && threadIdx.x == 0;
    // another CTA's shared memory may be written once that CTA runs
    if (a.probs) cl.sync();
    for (bool first = true;; first = false) {
        if (!a.probs) {  // one problem: every CTA knows
            if (threadIdx.x == 0) s.problem = first ? 0 : -1;
        } else if (leader) {  // the cluster's next problem
            const unsigned k = atomicAdd(&a.sync->next, 1u);
            const int p = k < (unsigned)a.P ? (int)k : -1;
            for (int q = 0; q < (int)cl.num_blocks(); ++q) *cl.map_shared_rank(&s.problem, q) = p;
        }
        cl.sync();  // also: every CTA is done with the previous problem
        if (s.problem < 0) break;
        if (threadIdx.x == 0) P = a.probs ? a.probs[s.problem] : a.single;
        __syncthreads();
        if (P.d <= 5) small_decode<5>(a, P, s, smem);
        else if (P.d <= 7) small_decode<7>(a, P, s, smem);
        else if (P.d <= 9) small_decode<9>(a, P, s, smem);
        else if (P.d <= 12) small_decode<12>(a, P, s, smem);
        else small_decode<16>(a, P, s, smem);
        if (leader && a.dev_out) {
            const DecodeCtrl *c = P.ctrl;
            ccs_result res;
            res.status = __ldcg(&c->status);
            res.iterations = __ldcg(&c->iteration);
            res.r0_final = __ldcg(&c->r0);
            res.error = __ldcg(&a.sync->error) ? CCS_ETIMEOUT : CCS_OK;
            res.row_driven = 0;
            res.row_entries = 0;
            res.residual_form =
                __ldcg(&c->ordered) ? CCS_RESIDUAL_ORDERED : CCS_RESIDUAL_EXACT;
            res.reserved = 0;
            a.dev_out[P.out_slot] = res;
        }
    }
}

// ---- host side --------------------------------------------------------------

// CTAs of a cluster that decodes problems of up to `entries` n d.
static int small_cluster(long long entries) {
    int C = 1;
    while (C < kSmallCluster && entries > kSmallPerCta * C) C *= 2;
    return C;
}

bool small_fits(int n, int m, int d) {
    return m <= kSmallMaxM && small_smem(n, m, d, kSmallCluster, nullptr, nullptr) <= kSmallSmem &&
           small_smem(n, m, d, small_cluster((long long)n * d), nullptr, nullptr) <= kSmallSmem;
}

bool small_route(const ProblemDev &pd, const ccs_params &prm, bool alone) {
    if (prm.engine != CCS_ENGINE_AUTO || prm.schedule != 0 || (prm.debug_flags & ~(kFlagOrdered | kFlagSwitch)) != 0 ||
        !small_fits(pd.n, pd.m, pd.d))
        return false;
    return !alone || ((long long)pd.n * pd.d <= kSmallAloneEntries && pd.m <= kSmallAloneM);
}

// Clusters of C CTAs that run at once, cached.
static int small_clusters(int dev, int C) {
    struct Entry {
        int dev, C, clusters;
    };
    static std::mutex mu;
    static Entry cache[256];
    static int used = 0;
    std::lock_guard<std::mutex> lk(mu);
    for (int e = 0; e < used; ++e)
        if (cache[e].dev == dev && cache[e].C == C) return cache[e].clusters;
    if (cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem) !=
        cudaSuccess)
        return 0;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = kSmallSmem;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int k = 0;
    if (cudaOccupancyMaxActiveClusters(&k, k_small, &cfg) != cudaSuccess) return 0;
    if (used < 256) cache[used++] = Entry{dev, C, k};
    return k;
}

// P problems (descriptors `pds` on the host; `dev` the same ones in device
// memory, or null for a single one), enqueued on `s` (`timed`: with the
// profiler's events, which a capture leaves out; `stamps`, or null: the phases
// of the first).  The sync word's `next` starts at zero.
int small_launch(const ProblemDev *pds, const ProblemDev *dev, int P, const ccs_params &prm,
                 EngineSync *sync, ccs_result *dev_out, unsigned long long *stamps,
                 cudaStream_t s, bool timed) {
    long long entries = 0;
    for (int p = 0; p < P; ++p) {
        const long long e = (long long)pds[p].n * pds[p].d;
        entries = e > entries ? e : entries;
    }
    const int C = small_cluster(entries);
    size_t smem = 0;
    for (int p = 0; p < P; ++p) {
        const size_t b = small_smem(pds[p].n, pds[p].m, pds[p].d, C, nullptr, nullptr);
        smem = b > smem ? b : smem;
    }
    int devno = 0;
    CCS_CUDA_TRY(cudaGetDevice(&devno));
    const int most = small_clusters(devno, C);
    if (most < 1) {
        set_last_error("no cluster of the small engine fits the device");
        return CCS_ECUDA;
    }
    SmallArgs a{};
    a.single = pds[0];
    a.probs = dev;
    a.P = P;
    a.alpha = prm.alpha;
    a.mode = prm.score_mode;
    a.max_iter = prm.max_iter;
    a.debug_flags = prm.debug_flags;
    a.shifted = prm.shifted;
    a.sync = sync;
    a.dev_out = dev_out;
    a.stamps = stamps;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    cfg.gridDim = dim3((unsigned)(C * (P < most ? P : most)));
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const int ev = timed ? prof_start(CCS_K_PERSISTENT, s) : -1;
    CCS_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_small, a));
    if (timed) {
        prof_stop(ev, s);
        count_launches(1);
    }
    return CCS_OK;
}

}  // namespace ccs
