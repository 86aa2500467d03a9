// Sparse Ember step (Section 2.2 of "Token Geometry", arXiv 2607.01455) for
// sm_103a.
//
// An embedding table's gradient is nonzero only on the rows of the token ids
// in the batch; a token seen k times receives the sum of its k
// per-occurrence rows (appendix "The Fisher is proportional to inverse
// frequency squared": g_i = (1/B) sum_k h_{i,k}).  The step equals the dense
// step of Algorithm 1 on that V x D gradient:
//   - every row of r decays (r_i <- beta2 r_i + (1-beta2) mean_j g_ij^2 with
//     g_i = 0 for rows not in the batch);
//   - the column statistics divide by V;
//   - only the touched rows of W change.
//
// Kernels, in launch order:
//   dedup     a counting sort by id, in integer atomics, linear in N and V but
//             for runs of more than 128 occurrences (see k_sp_order):
//             k_sp_count counts each id's occurrences in the V-entry map and
//             hands every occurrence an arrival number; k_sp_scan turns the
//             counts into the distinct ids (ascending) and where each id's run
//             starts, and decays r on the rows whose count is zero; k_sp_place
//             puts every occurrence at its run's start plus its arrival
//             number; k_sp_order sorts each run by occurrence, so that
//             arrival order (the only thing that varies from run to run)
//             leaves no trace.  A small batch takes one kernel instead,
//             k_sp_dedup_small.
//   segsum    k_sp_segsum, k_sp_carry: the summed gradient row of every
//             distinct id, adding its occurrences in increasing occurrence
//             order (compensated fp32 sums); per (id, column slice) sums of
//             g^2; per-CTA column sums
//             of g^2.  Each worker owns a contiguous, equal share of the
//             sorted occurrences, so the work is even however skewed the id
//             counts are (a Zipf head id can own thousands of occurrences);
//             a run that crosses worker boundaries leaves one piece per
//             worker, which k_sp_carry adds in worker order.
//   state     the dense step's column/normaliser pass, whose launch also runs
//             the row pass: r for the touched rows, the sums of new r per
//             CTA, and the touched-row map cleared for the next step.
//   apply     k_sp_apply: the update of the touched rows only (once per
//             column panel for tables wider than a CTA holds).
//
// Every kernel is launched with programmatic dependent launch (but see
// small_first_pdl and early_ranges) and waits (griddepcontrol.wait) before it reads anything.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "ember_device.cuh"
#include "ember_internal.h"

namespace ember {
namespace {

using namespace dev;

// Inclusive scan of x over a warp.
__device__ __forceinline__ int warp_scan(int x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    return x;
}

// ---------------------------------------------------------------------------
// Dedup.  The cost is a few trips to L2 per kernel, whatever the number of
// occurrences: sorting 1024-key tiles and ranking every key in every other
// tile took 23.7 us for 32768 ids and 313 us for 262144, most of it the
// ranks, which grow with the square of N.
// ---------------------------------------------------------------------------

// slot[id] <- how often the id occurs; arr[k] <- how many of its occurrences
// arrived before occurrence k (any order: k_sp_order undoes it).  A warp's
// equal ids make one global atomic (one occurrence per thread), or, with
// TABLE, those of the CTA's kCountKeys occurrences, added up in a hash table in
// shared memory first: a frequent id's atomics queue on one address at about
// 3 ns each.  An id that finds its table entry taken goes to the map directly.
// rng[2 q], rng[2 q + 1]: distinct ids and occurrences in the ids
// [q len, (q + 1) len).
template <typename IdT, bool TABLE>
__global__ void __launch_bounds__(kSpThreads)
k_sp_count(const IdT *__restrict__ ids, int64_t N, int64_t V, int32_t *__restrict__ slot,
           int32_t *__restrict__ arr, int32_t *__restrict__ rng, unsigned len, int nrange, DevScalars *sc)
{
    constexpr int kTab = TABLE ? kCountKeys : kSpThreads;  // a power of two
    constexpr int kPer = TABLE ? kCountKeys / kSpThreads : 1;
    __shared__ int tag[kTab], num[kTab];
    __shared__ int cnt[2 * kScanCtas];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t k0 = (int64_t)blockIdx.x * (kPer * kSpThreads) + tid;
    if constexpr (TABLE)
    for (int q = tid; q < kTab; q += kSpThreads) {
        tag[q] = -1;
        num[q] = 0;
    }
    for (int q = tid; q < 2 * nrange; q += kSpThreads)
        cnt[q] = 0;
    grid_dep_wait();  // whatever ran before on the stream
    grid_dep_launch();
    int id[kPer];
    bool bad = false;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const int64_t k = k0 + e * kSpThreads;
        id[e] = -1;
        if (k < N) {
            const int64_t x = (int64_t)ids[k];
            if (x >= 0 && x < V)
                id[e] = (int)x;
            else
                bad = true;  // skipped
        }
    }
    __syncthreads();
    if (__any_sync(0xffffffffu, bad) && lane == 0)
        atomicOr(&sc->flags, kFlagIdRange);
    auto count_in = [&](int x, int n, int before) {  // n occurrences of x reached the map, after `before`
        const unsigned q = (unsigned)x / len;
        atomicAdd(&cnt[2 * q + 1], n);
        if (before == 0)
            atomicAdd(&cnt[2 * q], 1);
    };
    int at[kPer], mine[kPer];  // table entry (-1: none), arrival number so far
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const unsigned peers = __match_any_sync(0xffffffffu, id[e]);
        const int lead = __ffs(peers) - 1;
        const int n = __popc(peers);
        int h = -1, m = 0;
        if (!TABLE && id[e] >= 0 && lane == lead) {
            m = atomicAdd(&slot[id[e]], n);
            count_in(id[e], n, m);
        }
        if (TABLE && id[e] >= 0 && lane == lead) {
            h = (int)(((unsigned)id[e] * 2654435761u) >> 16) & (kTab - 1);  // Fibonacci hashing
            const int old = atomicCAS(&tag[h], -1, id[e]);
            if (old == -1 || old == id[e]) {
                m = atomicAdd(&num[h], n);
            } else {
                h = -1;
                m = atomicAdd(&slot[id[e]], n);
                count_in(id[e], n, m);
            }
        }
        at[e] = __shfl_sync(0xffffffffu, h, lead);
        mine[e] = __shfl_sync(0xffffffffu, m, lead) + __popc(peers & ((1u << lane) - 1u));
    }
    __syncthreads();
    if constexpr (TABLE) {
        // the table's ids to the map, all of a thread's atomics in one trip
        constexpr int kE = kTab / kSpThreads;
        int n[kE], x[kE], before[kE];
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            n[e] = num[tid + e * kSpThreads];
            x[e] = tag[tid + e * kSpThreads];
        }
#pragma unroll
        for (int e = 0; e < kE; ++e)
            before[e] = n[e] ? atomicAdd(&slot[x[e]], n[e]) : 0;
#pragma unroll
        for (int e = 0; e < kE; ++e)
            if (n[e]) {
                num[tid + e * kSpThreads] = before[e];
                count_in(x[e], n[e], before[e]);
            }
        __syncthreads();
    }
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const int64_t k = k0 + e * kSpThreads;
        if (k < N)
            arr[k] = id[e] < 0 ? -1 : mine[e] + (at[e] >= 0 ? num[at[e]] : 0);
    }
    for (int q = tid; q < 2 * nrange; q += kSpThreads)
        if (cnt[q])
            atomicAdd(&rng[q], cnt[q]);
}

// CTA b numbers the distinct ids of [b len, (b + 1) len): uniq, segoff (the
// run's first position among the occurrences in id order), slot <- 1 + the
// number.  Runs longer than kLongRun are listed for k_sp_order (in any
// order).  With r: the rows outside the batch decay, r_i <- beta2 r_i (their
// g is 0), and the CTA's fp32 sum of them goes to rsum_part[b]; the touched
// rows are left to the state pass.
//   A range of one tile (V up to kScanCtas x kScanTile) is one trip to L2.
// The ranges of taller tables are bound by bandwidth: TILES tiles are loaded
// at once, and batches of tiles that no id is in, most of them, are not
// numbered.  With one tile at a time and 4-byte accesses of r, 8192 ids over
// 2^24 x 16 took 126 us and over 2^26 x 8 368; now 87 and 188 (4 tiles 89 and
// 194).
constexpr int kScanPer = 4;                        // ids per thread of a tile
constexpr int kScanTile = kSpThreads * kScanPer;

// r_i .. r_{i+3} below i1 (0 past it), in one access where r allows it.
__device__ __forceinline__ void load_r4(const float *r, bool aligned, int64_t i, int64_t i1,
                                        float (&x)[kScanPer])
{
    if (aligned && i + 3 < i1) {
        const float4 v = *reinterpret_cast<const float4 *>(r + i);
        x[0] = v.x;
        x[1] = v.y;
        x[2] = v.z;
        x[3] = v.w;
    } else {
#pragma unroll
        for (int e = 0; e < kScanPer; ++e)
            x[e] = i + e < i1 ? r[i + e] : 0.f;
    }
}

// The rows of i .. i + 3 that `touched` does not mark decay, r_i <- beta2 r_i
// (their g is 0); their new r is added to rsum in order.
__device__ __forceinline__ void decay_r4(float *r, bool aligned, int64_t i, int64_t i1,
                                         const EmaPair &ema, unsigned touched, float (&x)[kScanPer], float &rsum)
{
#pragma unroll
    for (int e = 0; e < kScanPer; ++e)
        if (i + e < i1 && !(touched >> e & 1u)) {
            x[e] = ema_pair(ema, x[e], 0.f);
            rsum += x[e];
        }
    if (aligned && i + 3 < i1 && (touched & 15u) == 0)
        *reinterpret_cast<float4 *>(r + i) = make_float4(x[0], x[1], x[2], x[3]);
    else
#pragma unroll
        for (int e = 0; e < kScanPer; ++e)
            if (i + e < i1 && !(touched >> e & 1u))
                r[i + e] = x[e];
}

template <int TILES>
__global__ void __launch_bounds__(kSpThreads)
k_sp_scan(int32_t *__restrict__ slot, int64_t V, int64_t len, const int32_t *__restrict__ rng,
          int32_t *__restrict__ uniq, int32_t *__restrict__ segoff, int32_t *__restrict__ longrun,
          int32_t *__restrict__ nlong, DevScalars *sc, float *__restrict__ r, EmaPair ema,
          float *__restrict__ rsum_part)
{
    constexpr int kW = kSpThreads / 32;
    __shared__ int bh[kW], bv[kW];  // of the ranges before this one, per warp of the sum
    __shared__ int wh[TILES][kW], wv[TILES][kW];
    __shared__ float wr[kW];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * len;
    const int64_t i1 = i0 + len < V ? i0 + len : V;
    grid_dep_wait();  // the counts
    grid_dep_launch();
    // distinct ids and occurrences of the ranges before this one
    int h = 0, v = 0;
    for (int q = tid; q < (int)blockIdx.x; q += kSpThreads) {
        h += __ldcg(rng + 2 * q);
        v += __ldcg(rng + 2 * q + 1);
    }
    h = __reduce_add_sync(0xffffffffu, h);
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) {
        bh[w] = h;
        bv[w] = v;
    }
    float rsum = 0.f;
    const bool aligned = (uintptr_t)r % 16 == 0;  // len is a multiple of 4
    int run = 0, pos = 0;  // of the next tile
    for (int64_t tb = i0; tb < i1; tb += TILES * kScanTile) {
        int c[TILES][kScanPer];
        float rr[TILES][kScanPer];
#pragma unroll
        for (int d = 0; d < TILES; ++d) {
            const int64_t i = tb + d * kScanTile + (int64_t)tid * kScanPer;  // a multiple of 4, as len is
            if (i + 3 < i1) {
                const int4 v = __ldcg(reinterpret_cast<const int4 *>(slot + i));
                c[d][0] = v.x;
                c[d][1] = v.y;
                c[d][2] = v.z;
                c[d][3] = v.w;
            } else {
#pragma unroll
                for (int e = 0; e < kScanPer; ++e)
                    c[d][e] = (i + e < i1) ? __ldcg(slot + i + e) : 0;
            }
            if (r)
                load_r4(r, aligned, i, i1, rr[d]);
        }
        // distinct ids and occurrences before this thread's, within its warp
        int xh[TILES], xv[TILES];
        bool any = false;
#pragma unroll
        for (int d = 0; d < TILES; ++d) {
            int nh = 0, nv = 0;
#pragma unroll
            for (int e = 0; e < kScanPer; ++e) {
                nh += c[d][e] > 0;
                nv += c[d][e];
            }
            xh[d] = xv[d] = 0;
            int th = 0, tv = 0;  // of the warp
            if (TILES == 1 || __any_sync(0xffffffffu, nv)) {  // (a tall table has mostly empty stretches)
                th = warp_scan(nh, lane);
                tv = warp_scan(nv, lane);
                xh[d] = th - nh;
                xv[d] = tv - nv;
                any = true;
            }
            if (lane == 31) {
                wh[d][w] = th;
                wv[d][w] = tv;
            }
        }
        any = __syncthreads_or(any);
        if (tb == i0) {
#pragma unroll
            for (int q = 0; q < kW; ++q) {
                run += bh[q];
                pos += bv[q];
            }
        }
#pragma unroll
        for (int d = 0; d < TILES; ++d) {
            const int64_t i = tb + d * kScanTile + (int64_t)tid * kScanPer;
            unsigned touched = 0;
            if (any) {
                int u = run + xh[d], p = pos + xv[d];
#pragma unroll
                for (int q = 0; q < kW; ++q) {
                    u += q < w ? wh[d][q] : 0;
                    p += q < w ? wv[d][q] : 0;
                    run += wh[d][q];
                    pos += wv[d][q];
                }
#pragma unroll
                for (int e = 0; e < kScanPer; ++e)
                    if (c[d][e] > 0) {
                        uniq[u] = (int)(i + e);
                        segoff[u] = p;
                        if (c[d][e] > kLongRun)
                            longrun[atomicAdd(nlong, 1)] = u;
                        ++u;
                        slot[i + e] = u;
                        p += c[d][e];
                        touched |= 1u << e;
                    }
            }
            if (r)
                decay_r4(r, aligned, i, i1, ema, touched, rr[d], rsum);
        }
        if (TILES > 1 && any)
            __syncthreads();  // before the next batch writes wh
    }
    if (blockIdx.x == gridDim.x - 1 && tid == 0) {
        sc->n_unique = run;
        sc->n_valid = pos;
        segoff[run] = pos;
    }
    if (r) {
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1)
            rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
        if (lane == 0)
            wr[w] = rsum;
        __syncthreads();
        if (tid == 0) {
            float t = 0.f;
            for (int q = 0; q < kW; ++q)
                t += wr[q];
            rsum_part[blockIdx.x] = t;
        }
    }
}

// Occurrence k of the id with number u to position segoff[u] + arr[k].
template <typename IdT>
__global__ void __launch_bounds__(kSpThreads)
k_sp_place(const IdT *__restrict__ ids, int64_t N, const int32_t *__restrict__ slot,
           const int32_t *__restrict__ segoff, const int32_t *__restrict__ arr, int32_t *__restrict__ placed,
           int32_t *__restrict__ segidx, int32_t *__restrict__ single)
{
    const int64_t k = (int64_t)blockIdx.x * kSpThreads + threadIdx.x;
    grid_dep_wait();  // runs and arrival numbers
    grid_dep_launch();
    if (k >= N)
        return;
    const int a = arr[k];
    if (a < 0)
        return;
    const int u = slot[ids[k]] - 1;
    const int s = segoff[u];
    const bool once = segoff[u + 1] == s + 1;
    placed[s + a] = (int)k;
    segidx[s + a] = u;
    if (a == 0)  // an id seen once: its summed row is that occurrence's row
        single[u] = once ? (int)k : -1;
}

// Workers split the sorted occurrences into contiguous ranges of equal
// cost, cost(p) = p + segidx[p]: one unit per occurrence row read and one
// per summed row written (runs are numbered in order, so the cost rises by
// one or two per position).  Worker w owns [first(w), first(w + 1)), where
// first(w) is the smallest position whose cost reaches T(w) = w C / nw and
// C = n_valid + U.  T(w) <= c where w C < (c + 1) nw: the tests below multiply
// instead of dividing.

// Workers in use, of the nw1 rg groups of a slice's CTAs (group g of CTA b is
// worker g nw1 + b): nw1 times as many groups as have kMinRows occurrences
// each, or, of a small batch, as many workers as have kFewRows (a batch of
// rows in flight).  More workers would cut frequent ids into more pieces, for
// the carry to add up one after another.  A function of the valid ids, so
// that skipped ones change nothing.
constexpr int kMinRows = 16, kFewRows = 8;
__device__ __forceinline__ int workers_of(int n_valid, int nw1, int rg)
{
    if (n_valid < kFewRows * nw1)
        return n_valid < kFewRows ? 1 : n_valid / kFewRows;
    const int most = n_valid / (kMinRows * nw1);
    return nw1 * (most < 1 ? 1 : most < rg ? most : rg);
}

// The workers that start at position p, of run u, which holds [s, e); `before`
// is the run of position p - 1 (-1 for p = 0): those whose target lies above
// the cost of the position before p and not above that of p, and, at the last
// position, those above every cost, which own nothing.  cuts[q]: the run that
// goes on at the start of worker q and began in worker q - 1's range, and the
// worker it ends in, or (-1, 0).  Both forms of the dedup take the starts from
// here: the sums of a batch do not depend on which one its length chooses.
// Threads `first` of `step` share the workers.
// I: int64_t, or int where 2 kSmallTallN times the number of workers fits it.
template <typename I>
__device__ __forceinline__ void worker_starts(int p, int u, int before, int s, int e, int n_valid, int U, int nw1,
                                              int rg, int32_t *__restrict__ bounds, int2 *__restrict__ cuts,
                                              int first, int step)
{
    const int nw = workers_of(n_valid, nw1, rg);
    const I C = (I)n_valid + U;
    const I c1 = (I)p + u;
    const I c0 = p > 0 ? (I)p - 1 + before : -1;
    for (I q = ((c0 + 1) * nw + C - 1) / C + first; q < nw; q += step) {
        const bool here = q * C < (c1 + 1) * nw;
        if (!here && p + 1 < n_valid)
            break;
        bounds[q] = here ? p : n_valid;
        int2 cut = make_int2(-1, 0);
        if (here && s < p && q > 0 && (q - 1) * C < ((I)s + u + 1) * nw) {
            const I to = (((I)e + u) * nw - 1) / C;  // the last whose target is not above the cost of e - 1
            cut = make_int2(u, (int)(to < nw ? to : nw - 1));
        }
        cuts[q] = cut;
    }
    if (p + 1 == n_valid && first == 0)
        bounds[nw] = n_valid;
}

// Each run's occurrences in increasing order, and the workers' bounds.
// A run of up to kLongRun occurrences: the thread of each position counts the
// smaller ones in its run (a warp's positions mostly share a run, so the
// loads broadcast).  A longer run, by a whole CTA: the occurrences of a
// window of kWinBits are bits of a bitmap in shared memory, read back in
// order; the first `nbig` CTAs take the (long run, window) pairs.  A long
// run is bound by its trips to L2, so a thread has 16 occurrences in flight.
//   Every window reads its whole run, so a long run of L occurrences costs
// L ceil(N / kWinBits) reads and as many bitmaps of kWinWords: linear in N
// while one window holds the batch, then with its square (1M uniform ids over
// 4000 rows, 4000 long runs and 16 windows: 0.70 ms here; the tile sort and
// ranks before took 4.6).
constexpr int kWinWords = 2048;
constexpr int kWinBits = 32 * kWinWords;
// Runs from this length on are looked through for stretches of nothing but one
// id (padding): read back a lane per word, 40000 equal ids take 42 us here,
// and 28 a lane per bit.  Asking costs short runs (262144 Zipf ids have
// hardly a full word) more than it gives.
constexpr int kStretch = 4096;
__global__ void __launch_bounds__(kOrderThreads)
k_sp_order(const int32_t *__restrict__ placed, const int32_t *__restrict__ segidx,
           const int32_t *__restrict__ segoff, const int32_t *__restrict__ longrun,
           const int32_t *__restrict__ nlong, const DevScalars *__restrict__ sc, int64_t N, int nbig,
           int32_t *__restrict__ perm, int32_t *__restrict__ bounds, int2 *__restrict__ cuts, int nw1, int rg)
{
    constexpr int kW = kOrderThreads / 32;
    constexpr int kPer = 16;
    __shared__ unsigned bits[kWinWords];
    __shared__ int wsum[2][kW];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    grid_dep_wait();  // placed occurrences
    grid_dep_launch();
    if ((int)blockIdx.x >= nbig) {
        const int n_valid = sc->n_valid, U = sc->n_unique;
        const int p = ((int)blockIdx.x - nbig) * kOrderThreads + tid;  // N < 2^30
        if (p >= n_valid)
            return;
        const int u = segidx[p];
        const int before = p > 0 ? segidx[p - 1] : -1;
        const int x = placed[p];
        const int s = segoff[u], e = segoff[u + 1];
        if (e - s <= kLongRun) {
            int below = 0;
#pragma unroll 8
            for (int q = s; q < e; ++q)
                below += placed[q] < x;
            perm[s + below] = x;
        }
        worker_starts<int64_t>(p, u, before, s, e, n_valid, U, nw1, rg, bounds, cuts, 0, 1);
        return;
    }
    const int nwin = (int)((N + kWinBits - 1) / kWinBits);
    const int64_t items = (int64_t)*nlong * nwin;
    for (int64_t it = blockIdx.x; it < items; it += nbig) {
        const int u = longrun[it / nwin];
        const int64_t k0 = (it % nwin) * kWinBits;
        const int words = (int)((N - k0 < kWinBits ? N - k0 : kWinBits) + 31) / 32;
        const int s = segoff[u], e = segoff[u + 1];
        for (int q = tid; q < words; q += kOrderThreads)
            bits[q] = 0u;
        __syncthreads();
        int below = 0;  // occurrences before the window
        for (int q0 = s + tid; q0 < e; q0 += kPer * kOrderThreads) {
            int x[kPer];
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int q = q0 + k * kOrderThreads;
                x[k] = q < e ? placed[q] : -1;
            }
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const int64_t b = x[k] - k0;
                if (b >= 0 && b < kWinBits)
                    atomicOr(&bits[b >> 5], 1u << (b & 31));
                below += x[k] >= 0 && b < 0;
            }
        }
        __syncthreads();
        // warp w owns words [w0, w1), 32 of them at a time; the rank of its
        // first bit is the number of bits in the words before them
        const int per = ((words + kW - 1) / kW + 31) / 32 * 32;
        const int w0 = w * per, w1 = w0 + per < words ? w0 + per : words;
        int mine = 0;
        for (int q = w0 + lane; q < w1; q += 32)
            mine += __popc(bits[q]);
        mine = __reduce_add_sync(0xffffffffu, mine);
        below = __reduce_add_sync(0xffffffffu, below);
        if (lane == 0) {
            wsum[0][w] = mine;
            wsum[1][w] = below;
        }
        __syncthreads();
        int at = s;
#pragma unroll
        for (int q = 0; q < kW; ++q)
            at += wsum[1][q] + (q < w ? wsum[0][q] : 0);
        for (int q = w0; q < w1; q += 32) {
            unsigned m = q + lane < w1 ? bits[q + lane] : 0u;
            const int n = __popc(m);
            const int x = warp_scan(n, lane);
            int o = at + x - n;
            if (e - s >= kStretch && __any_sync(0xffffffffu, m == 0xffffffffu)) {
                // a stretch of nothing but this id (a batch of padding): a lane
                // per bit, a word at a time, so that the warp's writes are
                // adjacent
#pragma unroll 4
                for (int k = 0; k < 32; ++k) {
                    const unsigned mk = __shfl_sync(0xffffffffu, m, k);
                    const int ok = __shfl_sync(0xffffffffu, o, k);
                    if (mk >> lane & 1u)
                        perm[ok + __popc(mk & ((1u << lane) - 1u))] = (int)(k0 + (int64_t)(q + k) * 32 + lane);
                }
            } else {
                while (m) {
                    perm[o++] = (int)(k0 + (int64_t)(q + lane) * 32 + __ffs(m) - 1);
                    m &= m - 1;
                }
            }
            at += __shfl_sync(0xffffffffu, x, 31);
        }
        __syncthreads();  // the bitmap is cleared for the next pair
    }
}

// ---------------------------------------------------------------------------
// Dedup of a small batch (N <= kSmallN) in one launch.  Every CTA takes the
// batch into shared memory, where a hash table picks one occurrence of every
// id to stand for it; a warp per occurrence then counts the smaller
// occurrences, those among them that stand for their id, and the earlier ones
// of its own id, which gives its sorted position and the number of its run.
// Nothing has to be scanned, and numbers, worker starts and the order in
// which r is summed are those of the four kernels above, so that a batch gives
// the same bits however many skipped ids it is padded with.
//   Bound by the N^2 integer compares and adds, over the CTAs, and by the tries
// that a CTA's last lane needs for its entry of the table.  50257 x 768, Zipf
// ids, us per step with it and with the four kernels: 1024 ids 25.3 and 30.2,
// 1536 25.8 and 29.4, 2048 29.1 and 30.9, 3000 29.5 and 31.7 (262144 x 2048:
// 38.3 and 38.0).
// 2^24 x 8, where the four kernels scan a map of 64 MB: 3500 ids 51.7 and
// 78.5, 4096 57.9 and 80.3; 10^7 x 8 43.8 and 56.9, 49.5 and 57.8.
// Without the table, runs numbered by their first position, 1024 Zipf ids took
// 24.6 to 24.9 and as many uniform ones 24.2 (27.1 with it), but the workers' shares and the sums of r depended on the padding.
//   The CTAs from `nkey` on decay r on the rows outside the batch, the ranges
// and tiles of k_sp_scan, from a bitmap of the ids, kDecayTiles tiles at once
// (1024 ids over 2^23 x 8 31.1 us per step, one at a time 37; eight 33.1).
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 512;
constexpr int kBitmapWords = 2048;
constexpr int kDecayTiles = 4;  // in flight per CTA
constexpr int small_pad(int N) { return (N + 127) / 128 * 128; }
// 1 << log_slots entries of the hash table: at least three quarters stay empty,
// so that the last lane of a warp takes its entry at the second try, not the
// fourth (2048 uniform ids over 50257 x 768: 30.2 us per step, 32.7 with half as
// many entries).
constexpr int small_log_slots(int N)
{
    int log_slots = 7;
    while (1 << log_slots < 4 * N)
        ++log_slots;
    return log_slots;
}
// The ids, their weights, the table (or the bitmap).  Never less than kSmallSmem: what a kernel asks for
// decides how its SMs split shared memory and L1, and with the 12 KB that
// 1024 occurrences needed at first the step took 26.5 us (50257 x 768), with
// twice as much or more 25.4.
constexpr size_t kSmallSmem = 46 << 10;
constexpr size_t small_smem(int N)
{
    const size_t slots = (size_t)1 << small_log_slots(N);
    const size_t b = sizeof(int) * (2 * (size_t)small_pad(N) + (slots > kBitmapWords ? slots : kBitmapWords));
    return b > kSmallSmem ? b : kSmallSmem;
}
template <typename IdT>
__global__ void __launch_bounds__(kSmallThreads)
k_sp_dedup_small(const IdT *__restrict__ ids, int N, int64_t V, int32_t *__restrict__ perm,
                 int32_t *__restrict__ segidx, int32_t *__restrict__ uniq, int32_t *__restrict__ single,
                 int32_t *__restrict__ bounds, int2 *__restrict__ cuts, int nw1, int rg, DevScalars *sc, int nkey,
                 int npad, int log_slots, int64_t len, float *__restrict__ r, EmaPair ema,
                 float *__restrict__ rsum_part)
{
    constexpr int kW = kSmallThreads / 32;
    constexpr int kNone = 0x7fffffff;  // a skipped id: V < 2^31, so every valid one is below
    constexpr int kFree = -1;
    __shared__ int total[2];  // distinct ids, valid ones
    __shared__ float wr[kSpThreads / 32];
    extern __shared__ __align__(16) int sid[];  // the ids, npad of them
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // 1, plus 1 << 16 where the occurrence stands for its id
    unsigned *const weight = reinterpret_cast<unsigned *>(sid + npad);
    int *const words = sid + 2 * npad;  // hash table of the ids, or a bitmap of a range's ids
    const bool keys = (int)blockIdx.x < nkey;
    grid_dep_wait();  // whatever ran before on the stream
    grid_dep_launch();
    constexpr int kAtOnce = 4;
    int64_t id[kAtOnce];
    auto load = [&](int q0) {
#pragma unroll
        for (int e = 0; e < kAtOnce; ++e)
            id[e] = q0 + e * kSmallThreads < N ? (int64_t)ids[q0 + e * kSmallThreads] : 0;
    };
    load(tid);  // in flight while the table is cleared
    if (keys) {
        for (int q = tid; q < 1 << (log_slots - 2); q += kSmallThreads)
            reinterpret_cast<int4 *>(words)[q] = make_int4(kFree, kFree, kFree, kFree);
        if (tid < 2)
            total[tid] = 0;
        __syncthreads();
    }
    bool bad = false;
    int U = 0, valid = 0;
    for (int q0 = tid; q0 < npad; q0 += kAtOnce * kSmallThreads) {
        if (q0 != tid)
            load(q0);
#pragma unroll
        for (int e = 0; e < kAtOnce; ++e) {
            const int q = q0 + e * kSmallThreads;
            if (q >= npad)
                break;  // whole warps: npad is a multiple of 32
            const bool ok = q < N && id[e] >= 0 && id[e] < V;
            bad |= q < N && !ok;
            const int x = ok ? (int)id[e] : kNone;
            sid[q] = x;
            if (!keys)
                continue;
            // an entry holds the id that took it; whoever took it stands for the id
            int was = x;
            if (ok)
                for (unsigned h = (unsigned)x * 2654435761u >> (32 - log_slots);;  // Fibonacci hashing
                     h = (h + 1) & ((1u << log_slots) - 1)) {
                    was = atomicCAS(words + h, kFree, x);
                    if (was == kFree || was == x)
                        break;
                }
            weight[q] = was == kFree ? 1u + (1u << 16) : 1u;
            U += __popc(__ballot_sync(0xffffffffu, was == kFree));
            valid += __popc(__ballot_sync(0xffffffffu, ok));
        }
    }
    if (bad && blockIdx.x == 0)
        atomicOr(&sc->flags, kFlagIdRange);
    if (keys && lane == 0) {
        atomicAdd(&total[0], U);
        atomicAdd(&total[1], valid);
    }
    __syncthreads();
    if (keys) {
        U = total[0];
        valid = total[1];
        if (blockIdx.x == 0 && tid == 0) {
            sc->n_unique = U;
            sc->n_valid = valid;
        }
        const int k = (int)blockIdx.x * kW + w;
        if (k >= N)
            return;
        const int x = sid[k];
        if (x == kNone)
            return;
        // smaller occurrences and, in the upper half, smaller distinct ids;
        // occurrences of x before k and from k on
        unsigned below = 0;
        int before = 0, after = 0;
        auto smaller = [&](const int4 &y, int q) {
            const uint4 o = *reinterpret_cast<const uint4 *>(weight + q);
            below += (y.x < x ? o.x : 0u) + (y.y < x ? o.y : 0u) + (y.z < x ? o.z : 0u) + (y.w < x ? o.w : 0u);
        };
        int q = lane * 4;
        for (; q + 3 < k; q += 128) {
            const int4 y = *reinterpret_cast<const int4 *>(sid + q);
            smaller(y, q);
            before += (y.x == x) + (y.y == x) + (y.z == x) + (y.w == x);
        }
        for (; q < npad; q += 128) {
            const int4 y = *reinterpret_cast<const int4 *>(sid + q);
            smaller(y, q);
            after += (y.x == x) + (y.y == x) + (y.z == x) + (y.w == x);
            if (q < k) {  // the four that hold k - 1 and k
                const int some = (y.x == x) + (q + 1 < k && y.y == x) + (q + 2 < k && y.z == x);
                before += some;
                after -= some;
            }
        }
        below = __reduce_add_sync(0xffffffffu, below);
        before = __reduce_add_sync(0xffffffffu, before);
        const int same = before + __reduce_add_sync(0xffffffffu, after);
        const int less = below & 0xffffu, u = below >> 16;
        const int p = less + before;
        if (lane == 0) {
            perm[p] = k;
            segidx[p] = u;
            if (before == 0) {
                uniq[u] = x;
                single[u] = same == 1 ? k : -1;
            }
        }
        worker_starts<int>(p, u, before > 0 ? u : u - 1, less, less + same, valid, U, nw1, rg, bounds, cuts, lane, 32);
        return;
    }
    constexpr int kBitmapIds = 32 * kBitmapWords;  // a multiple of kScanTile
    const bool aligned = (uintptr_t)r % 16 == 0;
    const int64_t b = (int)blockIdx.x - nkey;
    const int64_t i1 = (b + 1) * len < V ? (b + 1) * len : V;
    float rsum = 0.f;
    for (int64_t c0 = b * len; c0 < i1; c0 += kBitmapIds) {
        const int n = (int)(i1 - c0 < kBitmapIds ? i1 - c0 : kBitmapIds);
        for (int q = tid; q < (n + 31) / 32; q += kSmallThreads)
            words[q] = 0;
        __syncthreads();
        for (int q = tid; q < N; q += kSmallThreads) {
            const int64_t o = sid[q] - c0;
            // (a frequent id's bit is mostly there already)
            if (o >= 0 && o < n && !((unsigned)*(volatile int *)(words + (o >> 5)) >> (o & 31) & 1u))
                atomicOr(&words[o >> 5], (int)(1u << (o & 31)));
        }
        __syncthreads();
        // by the threads and in the order of k_sp_scan
        for (int q0 = tid * kScanPer; tid < kSpThreads && q0 < n; q0 += kDecayTiles * kScanTile) {
            float rr[kDecayTiles][kScanPer];
#pragma unroll
            for (int d = 0; d < kDecayTiles; ++d)
                if (q0 + d * kScanTile < n)
                    load_r4(r, aligned, c0 + q0 + d * kScanTile, c0 + n, rr[d]);
#pragma unroll
            for (int d = 0; d < kDecayTiles; ++d) {
                const int q = q0 + d * kScanTile;
                if (q < n)
                    decay_r4(r, aligned, c0 + q, c0 + n, ema, (unsigned)words[q >> 5] >> (q & 31), rr[d], rsum);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
        rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
    if (lane == 0 && w < kSpThreads / 32)
        wr[w] = rsum;
    __syncthreads();
    if (tid == 0) {
        float t = 0.f;
        for (int q = 0; q < kSpThreads / 32; ++q)
            t += wr[q];
        rsum_part[b] = t;
    }
}

// How the segment sums cover D columns: NS slices of tpb threads (one access
// each, equal slices so that few threads are idle), and rg groups of tpb
// threads per CTA (a narrow row leaves room for several), each group a worker
// of its own.
struct SumMap {
    int NS, tpb, rg;
};
SumMap sum_map(int DV)
{
    SumMap m;
    m.NS = (DV + kThreads - 1) / kThreads;
    m.tpb = ((DV + m.NS - 1) / m.NS + 31) / 32 * 32;
    m.rg = kThreads / m.tpb;
    return m;
}

// Barrier over the tpb threads of one group (named barriers 1 .. 8), or over
// the CTA when it is one group.
__device__ __forceinline__ void group_bar(int g, int rg, int tpb)
{
    if (rg == 1)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(tpb) : "memory");
}

// Column sums of the CTA's groups, added in group order, to (or onto) its
// partial row.
template <int VEC, bool ADD>
__device__ __forceinline__ void combine_groups(const float (&colacc)[VEC], float *comb, float *out, int g, int l,
                                               int tpb, int rg, int col0, int width)
{
#pragma unroll
    for (int e = 0; e < VEC; ++e)
        comb[(g * tpb + l) * VEC + e] = colacc[e];
    __syncthreads();
    for (int j = threadIdx.x; j < width; j += blockDim.x) {
        float t = comb[j];
        for (int q = 1; q < rg; ++q)
            t += comb[q * tpb * VEC + j];
        if (ADD)
            t += out[col0 + j];
        out[col0 + j] = t;
    }
}

// Sum the occurrences of each run.  A group of tpb threads works on column
// slice sigma of the sorted positions of its worker, adding each run's rows
// in increasing occurrence order with a running sum that crosses the worker's
// whole range.  A run that starts before the range or ends after it leaves
// its piece in the carry buffer (slot 0: the range's first run, slot 1: its
// last run); k_sp_carry adds the pieces in worker order.  Completed runs are
// written to S with their sum of g^2 per slice.
//   Bound by HBM (the occurrence rows are read once).  Each thread copies its
// own column slice of the rows to come into a ring of kRing rows in shared
// memory with cp.async, kBatch rows per commit group, so that the copies in
// flight take no registers and no row waits for the adds of another; a thread
// reads back only what it copied itself, so the ring needs no barrier.  A
// ring is 48 KiB (two CTAs: 96 KiB in flight per SM) whatever the width:
// 32768 rows of 2048 columns (4 KiB slices) take 105.8 us per step with 12
// rows, 115 with 18 of them per CTA's worth in flight (three CTAs); 262144 rows
// of 768 columns 219.7 us with 16 rows, 222.0 with 12, 226.7 with 20.
//   4-byte accesses are loaded into registers, kRows rows ahead, and put into
// the same slots from there: 4-byte copies into shared memory take the step
// for 40000 Zipf ids of 2049 columns 534 us against 269, 1119 columns 193
// against 168, 203 columns 68 against 60 (16 to 40 rows make no difference).
constexpr int kBatch = 4;
constexpr int kRingBytes = 48 << 10;
template <int VEC, int NT>
constexpr int ring_rows() { return kRingBytes / (4 * VEC * NT) / kBatch * kBatch; }
template <int VEC, int NT>  // NT: at least the CTA's threads
__global__ void __launch_bounds__(kThreads, kSparseCtasPerSm)
k_sp_segsum(const float *__restrict__ rows, const int32_t *__restrict__ perm,
            const int32_t *__restrict__ segidx, const DevScalars *__restrict__ sc,
            float *__restrict__ S, float *__restrict__ rowpart, float *__restrict__ carry,
            float *__restrict__ colpart, const int32_t *__restrict__ bounds, int D, SumMap map,
            int32_t *__restrict__ counters, int ncounters)
{
    using F = typename Vec<VEC>::F;
    constexpr int kRing = ring_rows<VEC, NT>();
    constexpr int kRows = 24;             // rows of 4-byte accesses in flight per thread
    static_assert(VEC == 4 || kRows <= kRing, "they pass through the ring");
    constexpr int kFin = 8;               // completed runs buffered before their g^2 sums are written
    constexpr int kWarps = kThreads / 32;
    constexpr int kIdxWindow = 1024;      // occurrences whose indices the CTA holds
    __shared__ float rp[kFin][kThreads];
    __shared__ int fin[kWarps][kFin];
    __shared__ int edge[kWarps][4];
    __shared__ int sperm[kIdxWindow];
    __shared__ int sseg[kIdxWindow];
    __shared__ float comb[kThreads * VEC];
    const int DV = D / VEC;
    const int NS = map.NS, tpb = map.tpb, rg = map.rg;
    const int g = threadIdx.x / tpb;
    const int l = threadIdx.x - g * tpb;
    const int sigma = blockIdx.x % NS;
    const int nw1 = (int)(gridDim.x / NS);
    const int b1 = (int)(blockIdx.x / NS);  // nw1 or more: a CTA left over by the division
    const int w = g * nw1 + b1;
    const int col = sigma * tpb + l;
    const bool active = col < DV;
    // threads past the row's end load its last vector (and discard the sums)
    const float *src = rows + (int64_t)(active ? col : DV - 1) * VEC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wpg = tpb >> 5;
    const int window = kIdxWindow / rg;
    int *const wperm = sperm + g * window, *const wseg = sseg + g * window;
    extern __shared__ __align__(16) unsigned char sp_ring[];
    F *const ring = reinterpret_cast<F *>(sp_ring) + threadIdx.x;  // slot q at ring[q * NT]
    grid_dep_wait();  // runs and occurrence order from the dedup kernels
    grid_dep_launch();
    // (the bounds are loaded with n_valid, before it says whether they count)
    const int q0 = bounds[w], q1 = bounds[w + 1];
    const int n_valid = sc->n_valid;
    float colacc[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e)
        colacc[e] = 0.f;
    // the occurrence rows stream through once: evict them first, so that
    // the summed rows written here stay in L2 for the update that reads them
    const uint64_t pol_rows = policy_evict_first();
    const uint64_t pol_sums = policy_evict_last();

    int p0 = 0, p1 = 0;
    if (b1 < nw1 && n_valid > 0 && w < workers_of(n_valid, nw1, rg)) {
        p0 = q0;
        p1 = q1;
        if (p0 == p1 && active) {
            // an empty range holds no piece of the run that spans it
            const F z = zero_vec<VEC>();
            *reinterpret_cast<F *>(carry + ((int64_t)2 * w) * D + (int64_t)col * VEC) = z;
            *reinterpret_cast<F *>(carry + ((int64_t)2 * w + 1) * D + (int64_t)col * VEC) = z;
        }
    }
    int nfin = 0;
    // the buffered runs' sums of g^2 over the group's threads, a warp per run
    auto drain = [&]() {  // uniform over the group
        group_bar(g, rg, tpb);
        for (int q = warp - g * wpg; q < nfin; q += wpg) {
            float t = 0.f;
            for (int k = lane; k < tpb; k += 32)
                t += rp[q][g * tpb + k];
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1)
                t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0)
                rowpart[(int64_t)fin[g][q] * NS + sigma] = t;
        }
        group_bar(g, rg, tpb);
        nfin = 0;
    };
    if (p0 < p1) {
        // Only the range's first run can have started before it and only
        // its last run can continue after it; both are decided once, from the
        // run indices at the range's edges, loaded with the first window's.
        if (l < 4) {
            const int at = l == 0 ? p0 - 1 : l == 1 ? p0 : l == 2 ? p1 - 1 : p1;
            edge[g][l] = at >= 0 && at < n_valid ? segidx[at] : -1;
        }
        int u_first = -1, u_last = -1;
        bool first_cut = false, last_cut = false;
        int cur = -1;
        int len = 0;  // occurrences of `cur` seen in this range
        // Per-id sums in occurrence order, compensated (Kahan): `acc` is the
        // running sum, `cmp` the part of it that rounding added, so the sum
        // stays within about an ulp even over thousands of duplicates.
        F acc = zero_vec<VEC>();
        F cmp = zero_vec<VEC>();
        auto flush = [&](int u) {
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                set_comp(acc, e, comp(acc, e) - comp(cmp, e));
            const bool before = first_cut && u == u_first;
            const bool after = last_cut && u == u_last;
            if (!before && !after) {
                float ps = 0.f;
                if (active) {
                    // an id seen once needs no summed row: the apply reads its occurrence row
                    if (len > 1)
                        store_g_hint<VEC>(S + (int64_t)u * D + (int64_t)col * VEC, acc, pol_sums);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const float a = comp(acc, e);
                        colacc[e] += a * a;
                        ps += a * a;
                    }
                }
                rp[nfin][threadIdx.x] = ps;
                if (l == 0)
                    fin[g][nfin] = u;
                ++nfin;
                if (nfin == kFin)
                    drain();
            } else if (active) {
                const int which = before ? 0 : 1;
                *reinterpret_cast<F *>(carry + ((int64_t)2 * w + which) * D + (int64_t)col * VEC) = acc;
            }
        };
        // The range's occurrence and run indices go to shared memory a
        // window at a time, so that a row costs one trip to HBM.
        for (int wb = p0; wb < p1; wb += window) {
            const int n = (wb + window < p1 ? wb + window : p1) - wb;
            group_bar(g, rg, tpb);  // the previous window's indices are no longer read
            for (int q = l; q < n; q += tpb) {
                wperm[q] = perm[wb + q];
                wseg[q] = segidx[wb + q];
            }
            group_bar(g, rg, tpb);
            if (wb == p0) {
                u_first = cur = edge[g][1];
                u_last = edge[g][2];
                first_cut = edge[g][0] == u_first;
                last_cut = edge[g][3] == u_last;
            }
            // rows b .. b + kBatch - 1 of the window into the kBatch slots
            // from `slot` on, one commit group
            auto fetch = [&](int b, F *slot) {
                if (b + kBatch <= n) {
#pragma unroll
                    for (int k = 0; k < kBatch; ++k)
                        cp_async_hint<VEC>(slot + k * NT, src + (int64_t)wperm[b + k] * D, pol_rows);
                } else {
                    for (int k = 0; b + k < n; ++k)
                        cp_async_hint<VEC>(slot + k * NT, src + (int64_t)wperm[b + k] * D, pol_rows);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            auto add = [&](const F &x, int u) {
                if (u != cur) {
                    flush(cur);
                    acc = zero_vec<VEC>();
                    cmp = zero_vec<VEC>();
                    cur = u;
                    len = 0;
                }
                ++len;
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float y = comp(x, e) - comp(cmp, e);
                    const float t = comp(acc, e) + y;
                    set_comp(cmp, e, (t - comp(acc, e)) - y);
                    set_comp(acc, e, t);
                }
            };
            if constexpr (VEC == 1) {
                F next[kRows];
                auto load = [&](int b) {  // rows b .. b + kRows - 1, the last one again past the end
                    if (b < n)
#pragma unroll
                        for (int k = 0; k < kRows; ++k)
                            next[k] = load_g_hint<VEC>(src + (int64_t)wperm[b + k < n ? b + k : n - 1] * D, pol_rows);
                };
                load(0);
#pragma unroll 1
                for (int b = 0; b < n; b += kRows) {
#pragma unroll
                    for (int k = 0; k < kRows; ++k)
                        ring[k * NT] = next[k];
                    load(b + kRows);
                    const int m = n - b < kRows ? n - b : kRows;
                    int k = 0;
#pragma unroll 1
                    for (; k + kBatch <= m; k += kBatch) {
                        F v[kBatch];
                        int u[kBatch];
#pragma unroll
                        for (int e = 0; e < kBatch; ++e) {
                            v[e] = ring[(k + e) * NT];
                            u[e] = wseg[b + k + e];
                        }
#pragma unroll
                        for (int e = 0; e < kBatch; ++e)
                            add(v[e], u[e]);
                    }
                    for (; k < m; ++k)
                        add(ring[k * NT], wseg[b + k]);
                }
                continue;
            }
            F *slot = ring;
#pragma unroll 1
            for (int b = 0; b < kRing; b += kBatch)
                fetch(b, ring + b * NT);
            int b = 0;
#pragma unroll 1
            for (; b + kBatch <= n; b += kBatch) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kRing / kBatch - 1) : "memory");
                F v[kBatch];
                int u[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    v[k] = slot[k * NT];
                    u[k] = wseg[b + k];
                }
#pragma unroll
                for (int k = 0; k < kBatch; ++k)
                    add(v[k], u[k]);
                fetch(b + kRing, slot);
                slot = (slot == ring + (kRing - kBatch) * NT) ? ring : slot + kBatch * NT;
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            for (int k = 0; b + k < n; ++k)
                add(slot[k * NT], wseg[b + k]);
        }
        flush(cur);
    }
    if (nfin > 0)
        drain();
    // this CTA's partial row: its own slice's column sums (the column pass
    // reads no other columns of it)
    const int col0 = sigma * tpb * VEC;
    combine_groups<VEC, false>(colacc, comb, colpart + (int64_t)blockIdx.x * D, g, l, tpb, rg, col0,
                               col0 + tpb * VEC < D ? tpb * VEC : D - col0);

    // the dedup's range counts and list length start the next step at zero
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q < ncounters; q += blockDim.x)
            counters[q] = 0;
}

// Runs cut by worker boundaries.  Group g of CTA b handles the boundary
// before worker bd = g nw1 + b / NS + 1 on slice b % NS: if a run that
// started inside the previous worker's range goes on there, this group adds
// the run's pieces -- the previous worker's last piece, then the first pieces
// of the following workers up to the one holding the run's end -- in worker
// order.
template <int VEC>
__global__ void __launch_bounds__(kThreads, kSparseCtasPerSm)
k_sp_carry(const int2 *__restrict__ cuts, const DevScalars *__restrict__ sc, const float *__restrict__ carry, float *__restrict__ S, float *__restrict__ rowpart,
           float *__restrict__ colpart, int D, SumMap map)
{
    using F = typename Vec<VEC>::F;
    constexpr int kWarps = kThreads / 32;
    constexpr int kManyPieces = 24;
    __shared__ float red[kWarps];
    __shared__ float comb[kThreads * VEC];
    __shared__ int3 shared_cut[kWarps];
    const int DV = D / VEC;
    const int NS = map.NS, tpb = map.tpb, rg = map.rg;
    const int g = threadIdx.x / tpb;
    const int l = threadIdx.x - g * tpb;
    const int sigma = blockIdx.x % NS;
    const int nw1 = (int)(gridDim.x / NS);
    const int bd = g * nw1 + (int)(blockIdx.x / NS) + 1;
    const int col = sigma * tpb + l;
    const bool active = col < DV;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wpg = tpb >> 5;
    grid_dep_wait();  // carry pieces from k_sp_segsum
    grid_dep_launch();
    const int n_valid = sc->n_valid;
    float colacc[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e)
        colacc[e] = 0.f;
    const bool in_use = (int)(blockIdx.x / NS) < nw1 && n_valid > 0 && bd < workers_of(n_valid, nw1, rg);
    const int2 cut = in_use ? cuts[bd] : make_int2(-1, 0);
    const bool mine = cut.x >= 0;
    // pieces q0 .. q1 of the run that began in worker w (piece 0: its last
    // piece; piece q: the first piece of worker w + q, zero where that range is
    // empty), compensated as in k_sp_segsum
    const int64_t off = (int64_t)(active ? col : DV - 1) * VEC;
    auto sum_pieces = [&](int w, int q0, int q1) {
        F acc = zero_vec<VEC>();
        F cmp = zero_vec<VEC>();
        constexpr int kB = 12;
        for (int qb = q0; qb <= q1; qb += kB) {
            F v[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                const int q = qb + k;
                v[k] = (q <= q1) ? load_g<VEC>(carry + ((int64_t)2 * (w + q) + (q == 0)) * D + off) : zero_vec<VEC>();
            }
#pragma unroll
            for (int k = 0; k < kB; ++k)
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float y = comp(v[k], e) - comp(cmp, e);
                    const float t = comp(acc, e) + y;
                    set_comp(cmp, e, (t - comp(acc, e)) - y);
                    set_comp(acc, e, t);
                }
        }
#pragma unroll
        for (int e = 0; e < VEC; ++e)
            set_comp(acc, e, comp(acc, e) - comp(cmp, e));
        return acc;
    };
    auto finish = [&](const F &acc, int u) {  // by a whole group
        float ps = 0.f;
        if (active) {
            *reinterpret_cast<F *>(S + (int64_t)u * D + off) = acc;
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const float a = comp(acc, e);
                colacc[e] += a * a;
                ps += a * a;
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1)
            ps += __shfl_xor_sync(0xffffffffu, ps, o);
        if (lane == 0)
            red[warp] = ps;
        group_bar(g, rg, tpb);
        if (l == 0) {
            float t = 0.f;
            for (int k = 0; k < wpg; ++k)
                t += red[g * wpg + k];
            rowpart[(int64_t)u * NS + sigma] = t;
        }
        group_bar(g, rg, tpb);
    };
    // a run of many pieces is added by all the CTA's groups, a stretch each
    const bool many = rg > 1 && mine && cut.y - (bd - 1) >= kManyPieces;
    if (l == 0)
        shared_cut[g] = many ? make_int3(cut.x, bd - 1, cut.y) : make_int3(-1, 0, 0);
    if (mine && !many)  // uniform over the group
        finish(sum_pieces(bd - 1, 0, cut.y - (bd - 1)), cut.x);
    if (__syncthreads_or(many))
        for (int q = 0; q < rg; ++q) {
            const int3 run = shared_cut[q];
            if (run.x < 0)
                continue;
            const int n = run.z - run.y + 1, per = (n + rg - 1) / rg;
            const F part = sum_pieces(run.y, g * per, (g + 1) * per < n ? (g + 1) * per - 1 : n - 1);
#pragma unroll
            for (int e = 0; e < VEC; ++e)
                comb[(g * tpb + l) * VEC + e] = comp(part, e);
            __syncthreads();
            if (g == q) {
                F acc = zero_vec<VEC>(), cmp = zero_vec<VEC>();
                for (int k = 0; k < rg; ++k)
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const float y = comb[(k * tpb + l) * VEC + e] - comp(cmp, e);
                        const float t = comp(acc, e) + y;
                        set_comp(cmp, e, (t - comp(acc, e)) - y);
                        set_comp(acc, e, t);
                    }
#pragma unroll
                for (int e = 0; e < VEC; ++e)
                    set_comp(acc, e, comp(acc, e) - comp(cmp, e));
                finish(acc, run.x);
            }
            __syncthreads();
        }
    // CTA b of this kernel and CTA b of k_sp_segsum share the workers bd - 1
    // and slice sigma: add these runs' column sums to that CTA's partial row
    if (__syncthreads_or(mine)) {
        const int col0 = sigma * tpb * VEC;
        combine_groups<VEC, true>(colacc, comb, colpart + (int64_t)blockIdx.x * D, g, l, tpb, rg, col0,
                                  col0 + tpb * VEC < D ? tpb * VEC : D - col0);
    }
}

// The update of the touched rows: W[uniq[u]] from the summed row S[u].
// Three CTAs per SM (two for the widest rows): each CTA has only a few rows,
// so more of them are kept in flight at once.  D columns from row stride ld
// (a column panel of a wider table: W, S, rows and c point at its first
// column).
constexpr int apply_ctas_per_sm(int cpt) { return cpt >= 8 ? 2 : cpt >= 4 ? 4 : 3; }
template <int VEC, int CPT, int R, bool BF16>
__global__ void __launch_bounds__(kThreads, apply_ctas_per_sm(CPT))
k_sp_apply(void *__restrict__ W, const float *__restrict__ S, const float *__restrict__ rows,
           const int32_t *__restrict__ uniq, const int32_t *__restrict__ single,
           const float *__restrict__ r, const float *__restrict__ c,
           const DevScalars *__restrict__ sc, NormSource norm, int D, int ld, int tpr, StepConsts kc,
           float eps, float lr_signed, int variant)
{
    using F = typename Vec<VEC>::F;
    using WT = typename WRaw<BF16, VEC>::T;
    extern __shared__ float cs[];
    const int DV = D / VEC;
    const int tid = threadIdx.x;
    const int rg = kThreads / tpr;
    const int g = tid / tpr;
    const int l = tid - g * tpr;
    grid_dep_wait();  // c, r, their sums and the summed rows
    grid_dep_launch();
    const int U = sc->n_unique;
    const float inv_bc = kc.inv_bc;
    const float inv_s = (variant == EMBER_VARIANT_FULL) ? step_inv_s<kThreads>(norm, kc) : 1.f;
    for (int j = tid; j < D; j += kThreads)
        cs[j] = (variant == EMBER_VARIANT_ROW) ? 1.f : sqrtf(c[j] * inv_bc * inv_s);
    __syncthreads();

    // the summed rows, the W rows and the written W are touched for the last
    // time in the step
    const uint64_t pol = policy_evict_first();
    const int64_t stride = (int64_t)gridDim.x * rg * R;
    const int64_t ub0 = ((int64_t)blockIdx.x * rg + g) * R;
    // row ids (and, for ids seen once, the occurrence row) of the next
    // iteration are loaded while this one's rows are in flight
    int64_t next[R];
    int nsingle[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        next[k] = (ub0 + k < U) ? (int64_t)uniq[ub0 + k] : -1;
        nsingle[k] = (ub0 + k < U) ? single[ub0 + k] : -1;
    }
    for (int64_t ub = ub0; ub < U; ub += stride) {
        F gv[R][CPT];
        WT wr[R][CPT];
        int64_t row[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int64_t u = ub + k;
            row[k] = next[k];
            const float *src = (nsingle[k] >= 0) ? rows + (int64_t)nsingle[k] * ld : S + u * ld;
#pragma unroll
            for (int cc = 0; cc < CPT; ++cc) {
                const int col = l + cc * tpr;
                if (row[k] >= 0 && col < DV) {
                    gv[k][cc] = load_g_hint<VEC>(src + (int64_t)col * VEC, pol);
                    wr[k][cc] = load_w_hint<BF16, VEC>(W, row[k] * ld + (int64_t)col * VEC, pol);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int64_t un = ub + stride + k;
            next[k] = (un < U) ? (int64_t)uniq[un] : -1;
            nsingle[k] = (un < U) ? single[un] : -1;
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (row[k] < 0)
                continue;
            const float rs = (variant == EMBER_VARIANT_COL) ? 1.f : sqrtf(__ldg(r + row[k]) * inv_bc);
#pragma unroll
            for (int cc = 0; cc < CPT; ++cc) {
                const int col = l + cc * tpr;
                if (col >= DV)
                    continue;
                float wv[VEC];
                unpack_w(wr[k][cc], wv);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const float den = fmaf(rs, cs[col * VEC + e], eps);
                    const float u = update_ratio(comp(gv[k][cc], e), den);
                    wv[e] = fmaf(lr_signed, u, wv[e]);
                }
                store_w_hint<BF16, VEC>(W, row[k] * ld + (int64_t)col * VEC, wv, pol);
            }
        }
    }
}

// The launches of one step or dedup on its stream, in order, with the trace
// events between them.  After a launch that fails nothing more is launched:
// the kernels after it would read what it has not written (k_sp_place, for
// one, would take the counts left in the map for run numbers).
struct Launches {
    const cudaEvent_t *ev;
    int n, next;
    cudaStream_t s;
    cudaError_t err = cudaSuccess;  // of the first launch that failed
    template <typename K, typename... Args>
    void launch(K kernel, dim3 grid, dim3 block, size_t smem, bool early, Args &&...args)
    {
        if (err == cudaSuccess)
            err = launch_k(kernel, grid, block, smem, s, early, static_cast<Args &&>(args)...);
    }
    void mark()
    {
        if (err == cudaSuccess && ev && next < n)
            cudaEventRecord(ev[next], s);
        ++next;
    }
    // programmatic dependent launch, unless events are recorded between the kernels
    bool pdl() const { return ev == nullptr; }
};

// The map and the counters back to zero, as every step expects them.
cudaError_t clear_dedup(const SparseArgs &a)
{
    const cudaError_t e = cudaMemsetAsync(a.ws + a.lay.sp_slot, 0, sizeof(int32_t) * (size_t)a.V, a.stream);
    return e != cudaSuccess ? e
                            : cudaMemsetAsync(a.ws + a.lay.sp_rng, 0, sizeof(int32_t) * kScanCounters, a.stream);
}

// Before the first launch: what an earlier call could not clear.  A clear that
// is only captured leaves the next call to clear again.
cudaError_t begin(const SparseArgs &a)
{
    if (!*a.unclean)
        return cudaSuccess;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(a.stream, &capture);
    if (e == cudaSuccess)
        e = clear_dedup(a);
    if (e == cudaSuccess && capture == cudaStreamCaptureStatusNone)
        *a.unclean = false;
    return e;
}

// After the last launch.  A failed one leaves counts, run numbers or range
// counters behind, which the kernels launched next would add to and take
// positions from: they are cleared behind the kernels that did run, or, where
// that fails too, before the next step.
cudaError_t finish(const SparseArgs &a, const Launches &la)
{
    if (la.err == cudaSuccess)
        return cudaGetLastError();
    cudaGetLastError();  // reported here, not by the next call
    if (clear_dedup(a) != cudaSuccess)
        *a.unclean = true;
    cudaGetLastError();
    return la.err;
}

// Fewest occurrences that are counted through the hash table: below, at most
// 3.3 ns of atomics queue on one address per 32 occurrences of one id, and
// the direct form's one trip to L2 ends sooner.  Zipf ids over 50257 x 256, us
// per step through the table and directly: 32768 48.5 and 45.0, 49152 53.0
// and 52.9, 65536 59.1 and 59.6, 131072 74.1 and 79.8, 262144 113.3 and 130.1
// (uniform ids, where no address queues: 53.9 and 51.7, 58.5 and 56.1, 76.1 and
// 74.6, 105.3 and 107.8 from 49152 on).
constexpr int64_t kTableMinN = 65536;

// Ids per range of k_sp_count and k_sp_scan, and the number of ranges: a
// function of V alone.
int64_t scan_len(int64_t V)
{
    int64_t len = (V + kScanCtas - 1) / kScanCtas;
    if (len < kScanMin)
        len = kScanMin;
    return (len + 3) / 4 * 4;
}
int scan_ranges(int64_t V) { return (int)((V + scan_len(V) - 1) / scan_len(V)); }

// Tiles in flight in a CTA of the scan of a tall table.
constexpr int kTallTiles = 8;

// Whether the kernels that read a range of the table per CTA are launched
// early.  Of a tall table that loses more than the launch latency it gains:
// 8 ids over 2^24 x 16 49 us early and 37 not, 8192 ids over 2^22 x 64 52.7
// and 50.9; over 2^20 x 64 22.2 and 23.9, 45.3 and 46.4.  (CTAs launched onto
// SMs that are still busy are spread unevenly, likely, and a long range is
// bound by bandwidth.)
bool early_ranges(int64_t V) { return V <= int64_t(1) << 22; }

// Count the ids and number the distinct ones; with r also decay the rows
// outside the batch (their sums to rsum_part[0 .. scan_ranges)).
template <typename IdT>
void launch_count_scan(const SparseArgs &a, Launches &la, float *r, const EmaPair &ema, float *rsum_part)
{
    unsigned char *ws = a.ws;
    const Layout &L = a.lay;
    DevScalars *sc = reinterpret_cast<DevScalars *>(ws + L.scalars);
    auto *slot = reinterpret_cast<int32_t *>(ws + L.sp_slot);
    auto *rng = reinterpret_cast<int32_t *>(ws + L.sp_rng);
    const int64_t len = scan_len(a.V);
    const int nr = scan_ranges(a.V);
    if (a.N > 0) {
        const bool table = a.N >= kTableMinN;
        const int keys = table ? kCountKeys : kSpThreads;
        la.launch(table ? k_sp_count<IdT, true> : k_sp_count<IdT, false>, dim3((int)((a.N + keys - 1) / keys)),
                  dim3(kSpThreads), 0, la.pdl(),
                 static_cast<const IdT *>(a.ids), a.N, a.V, slot, reinterpret_cast<int32_t *>(ws + L.sp_arr), rng,
                 (unsigned)len, nr, sc);
        la.mark();
    }
    la.launch(len > kScanTile ? k_sp_scan<kTallTiles> : k_sp_scan<1>, dim3(nr), dim3(kSpThreads), 0,
              la.pdl() && early_ranges(a.V), slot, a.V, len, rng,
             reinterpret_cast<int32_t *>(ws + L.sp_uniq), reinterpret_cast<int32_t *>(ws + L.sp_segoff),
             reinterpret_cast<int32_t *>(ws + L.sp_long), rng + kScanCounters - 1, sc, r, ema, rsum_part);
    la.mark();
}

// Every occurrence to its place in (id, occurrence) order; bounds of the
// workers of the segment sums (rg groups in each of nw1 CTAs per slice).
template <typename IdT>
void launch_place_order(const SparseArgs &a, Launches &la, int nw1, int rg)
{
    unsigned char *ws = a.ws;
    const Layout &L = a.lay;
    DevScalars *sc = reinterpret_cast<DevScalars *>(ws + L.scalars);
    auto *segidx = reinterpret_cast<int32_t *>(ws + L.sp_segidx);
    auto *segoff = reinterpret_cast<int32_t *>(ws + L.sp_segoff);
    auto *placed = reinterpret_cast<int32_t *>(ws + L.sp_placed);
    const int nb = (int)((a.N + kSpThreads - 1) / kSpThreads);
    if (nb == 0)
        return;  // no occurrence: the segment sums and the carry see n_valid = 0
    la.launch(k_sp_place<IdT>, dim3(nb), dim3(kSpThreads), 0, la.pdl(), static_cast<const IdT *>(a.ids), a.N,
             reinterpret_cast<int32_t *>(ws + L.sp_slot), segoff, reinterpret_cast<int32_t *>(ws + L.sp_arr), placed,
             segidx, reinterpret_cast<int32_t *>(ws + L.sp_single));
    la.mark();
    const int64_t nbig64 = a.N / (kLongRun + 1) * ((a.N + kWinBits - 1) / kWinBits);
    const int nbig = (int)(nbig64 < kGridCtas ? nbig64 : kGridCtas);
    la.launch(k_sp_order, dim3(nbig + (int)((a.N + kOrderThreads - 1) / kOrderThreads)), dim3(kOrderThreads), 0,
              la.pdl(), placed, segidx, segoff,
             reinterpret_cast<int32_t *>(ws + L.sp_long),
             reinterpret_cast<int32_t *>(ws + L.sp_rng) + kScanCounters - 1, sc, a.N, nbig,
             reinterpret_cast<int32_t *>(ws + L.sp_perm), reinterpret_cast<int32_t *>(ws + L.sp_bounds),
             reinterpret_cast<int2 *>(ws + L.sp_cuts), nw1, rg);
    la.mark();
}

// Distinct ids, their counts and U to caller buffers; the map and the counters
// cleared for the next call.
__global__ void k_sp_export(const int32_t *__restrict__ uniq, const int32_t *__restrict__ segoff,
                            const DevScalars *__restrict__ sc, int64_t N, int32_t *__restrict__ uniq_out,
                            int32_t *__restrict__ counts_out, int32_t *__restrict__ n_unique_out,
                            int32_t *__restrict__ slot, int32_t *__restrict__ counters, int ncounters)
{
    grid_dep_wait();
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q < ncounters; q += blockDim.x)
            counters[q] = 0;
    const int U = sc->n_unique;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < N;
         u += (int64_t)gridDim.x * blockDim.x) {
        if (u < U) {
            const int id = uniq[u];
            uniq_out[u] = id;
            slot[id] = 0;  // the map is all zero again for the next call
            counts_out[u] = segoff[u + 1] - segoff[u];
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *n_unique_out = U;
}

// Whether the one dedup kernel of a small batch may be launched while the
// kernel before it on the stream is still running.  Early, it gains a launch
// latency; the CTAs that then wait hold SMs which the kernel before, the update
// of the step before in a run of steps, still wants, and their number grows
// with N.  us per step early and not: 50257 x 768, 64 Zipf ids 18.9 and 20.8,
// 128 21.0 and 22.8, 256 22.9 and 23.1, 384 24.2 and 24.8, 512 26.1 and 24.8,
// 1024 27.9 and 25.5.  The line does not move with V: 128 ids of 256 columns
// 20.5 and 21.0 over 2000 rows, 19.2 and 20.7 over 16384, 21.5 and 22.8 over
// 262144, 22.3 and 23.1 over 1000000; 1024 ids 25.7 and 23.0, 25.2 and 23.0,
// 25.5 and 23.9, 26.5 and 24.8.
bool small_first_pdl(int64_t N) { return N <= 256; }

// Whether a batch takes the one-launch dedup: up to kSmallN occurrences, and,
// of a table so tall that the counting form's scan of the map shows, up to
// kSmallTallN (see k_sp_dedup_small for both sides of the lines).
bool one_launch_dedup(int64_t N, int64_t V)
{
    return N > 0 && (N <= kSmallN || (N <= kSmallTallN && V >= int64_t(1) << 23));
}

template <int VEC, int CPT>
cudaError_t launch_sparse_t(const SparseArgs &a)
{
    constexpr int R = (4 / CPT) < 1 ? 1 : (4 / CPT);
    unsigned char *ws = a.ws;
    const Layout &L = a.lay;
    DevScalars *sc = reinterpret_cast<DevScalars *>(ws + L.scalars);
    auto *perm = reinterpret_cast<int32_t *>(ws + L.sp_perm);
    auto *segidx = reinterpret_cast<int32_t *>(ws + L.sp_segidx);
    auto *uniq = reinterpret_cast<int32_t *>(ws + L.sp_uniq);
    auto *slot = reinterpret_cast<int32_t *>(ws + L.sp_slot);
    auto *single = reinterpret_cast<int32_t *>(ws + L.sp_single);
    auto *rowpart = reinterpret_cast<float *>(ws + L.sp_rowpart);
    auto *carry = reinterpret_cast<float *>(ws + L.sp_carry);
    auto *bounds = reinterpret_cast<int32_t *>(ws + L.sp_bounds);
    auto *cuts = reinterpret_cast<int2 *>(ws + L.sp_cuts);
    auto *S = reinterpret_cast<float *>(ws + L.sp_rows);
    auto *colpart = reinterpret_cast<float *>(ws + L.colpart);
    auto *rsum_part = reinterpret_cast<float *>(ws + L.rsum_part);
    auto *csum_part = reinterpret_cast<float *>(ws + L.csum_part);
    const int D = (int)a.D;
    const int DV = D / VEC;
    const SumMap map = sum_map(DV);
    const int NS = map.NS;
    const dim3 sum_threads(map.rg * map.tpb);
    Launches la{a.trace, a.n_trace, 0, a.stream};

    // (a CTA has 160, 192, 224 or 256 threads: see sum_map)
    auto *segsum = sum_threads.x > 192 ? k_sp_segsum<VEC, 256> : k_sp_segsum<VEC, 192>;
    // the ring and the static arrays together pass 48 KiB
    cudaError_t e = cudaFuncSetAttribute(segsum, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
    if (e == cudaSuccess)
        e = begin(a);
    if (e != cudaSuccess)
        return e;

    la.mark();
    const int G = kSparseCtas;
    const StepConsts kc = make_consts(a.beta2, a.one_minus_beta2, a.V, a.D, a.inv_bc);
    if (one_launch_dedup(a.N, a.V)) {
        const int nkey = (int)((a.N + kSmallThreads / 32 - 1) / (kSmallThreads / 32));
        const size_t sm = small_smem((int)a.N);
        auto go = [&](auto *ids) {
            using IdT = std::remove_const_t<std::remove_pointer_t<decltype(ids)>>;
            if (sm > (size_t)47 << 10)  // with the static arrays up to 48 KiB need no leave
                la.err = cudaFuncSetAttribute(k_sp_dedup_small<IdT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)sm);
            la.launch(k_sp_dedup_small<IdT>, dim3(nkey + scan_ranges(a.V)), dim3(kSmallThreads), sm,
                      la.pdl() && small_first_pdl(a.N) && early_ranges(a.V), ids, (int)a.N, a.V, perm, segidx, uniq, single, bounds, cuts,
                      G / NS, map.rg, sc, nkey, small_pad((int)a.N), small_log_slots((int)a.N), scan_len(a.V), a.r,
                      kc.ema, rsum_part);
        };
        if (a.ids64)
            go(static_cast<const int64_t *>(a.ids));
        else
            go(static_cast<const int32_t *>(a.ids));
        la.mark();
    } else if (a.ids64) {
        launch_count_scan<int64_t>(a, la, a.r, kc.ema, rsum_part);
        launch_place_order<int64_t>(a, la, G / NS, map.rg);
    } else {
        launch_count_scan<int32_t>(a, la, a.r, kc.ema, rsum_part);
        launch_place_order<int32_t>(a, la, G / NS, map.rg);
    }
    la.launch(segsum, dim3(G), sum_threads, kRingBytes, la.pdl(), a.rows, perm, segidx, sc, S, rowpart, carry,
             colpart, bounds, D, map, reinterpret_cast<int32_t *>(ws + L.sp_rng), kScanCounters);
    la.mark();
    la.launch(k_sp_carry<VEC>, dim3(G), sum_threads, 0, la.pdl(), cuts, sc, carry, S, rowpart,
             colpart, D, map);
    la.mark();
    // the touched rows' r and the column pass in one launch (a row per thread
    // for up to one CTA per SM: more would only wait for a place); the per-CTA
    // sums of r follow the scan CTAs' sums of the decayed rows
    const int nr = scan_ranges(a.V);
    const int64_t ub = (a.N + kStateThreads - 1) / kStateThreads;
    const int GU = (int)(ub < kSms ? ub : kSms);
    const NormSource norm{rsum_part, nr + GU, csum_part, (D + kStateCols - 1) / kStateCols, nullptr, nullptr, D};
    // (segment-sum CTA b writes only the columns of its slice b % NS)
    if (la.err == cudaSuccess)
        la.err = launch_state(colpart, G, rsum_part, a.c, csum_part, sc, a.V, D, kc, a.stream, la.pdl(), a.r, slot,
                              rowpart, NS, GU, uniq, nr, NS, map.tpb * VEC);
    la.mark();
    // one launch per column panel (one unless D is wider than a CTA's row)
    const int np = a.map.npanels, pw = a.map.pw;
    const size_t cs_bytes = (size_t)pw * sizeof(float);
    const int GA = kSms * apply_ctas_per_sm(CPT);
    for (int q = 0; q < np; ++q) {
        const int64_t c0 = (int64_t)q * pw;
        const int dq = (q + 1 < np) ? pw : (int)(a.D - c0);
        void *Wq = static_cast<unsigned char *>(a.W) + c0 * (a.wbf16 ? 2 : 4);
        const float *rq = a.rows ? a.rows + c0 : nullptr;
        if (a.wbf16)
            la.launch(k_sp_apply<VEC, CPT, R, true>, dim3(GA), dim3(kThreads), cs_bytes, la.pdl(), Wq,
                     S + c0, rq, uniq, single, a.r, a.c + c0, sc, norm, dq, (int)a.D, a.map.tpr, kc, a.eps,
                     a.lr_signed, a.variant);
        else
            la.launch(k_sp_apply<VEC, CPT, R, false>, dim3(GA), dim3(kThreads), cs_bytes, la.pdl(), Wq,
                     S + c0, rq, uniq, single, a.r, a.c + c0, sc, norm, dq, (int)a.D, a.map.tpr, kc, a.eps,
                     a.lr_signed, a.variant);
    }
    la.mark();
    return finish(a, la);
}

}  // namespace

cudaError_t launch_sparse_step(const SparseArgs &a)
{
    if (a.map.vec == 4) {
        switch (a.map.cpt) {
        case 1: return launch_sparse_t<4, 1>(a);
        case 2: return launch_sparse_t<4, 2>(a);
        case 4: return launch_sparse_t<4, 4>(a);
        case 8: return launch_sparse_t<4, 8>(a);
        }
    } else {
        switch (a.map.cpt) {
        case 1: return launch_sparse_t<1, 1>(a);
        case 2: return launch_sparse_t<1, 2>(a);
        case 4: return launch_sparse_t<1, 4>(a);
        case 8: return launch_sparse_t<1, 8>(a);
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_sparse_unique(const SparseArgs &a, int32_t *uniq_out, int32_t *counts_out,
                                 int32_t *n_unique_out)
{
    cudaError_t e = begin(a);
    if (e != cudaSuccess)
        return e;
    Launches la{nullptr, 0, 0, a.stream};
    if (a.ids64)
        launch_count_scan<int64_t>(a, la, nullptr, EmaPair{}, nullptr);
    else
        launch_count_scan<int32_t>(a, la, nullptr, EmaPair{}, nullptr);
    const DevScalars *sc = reinterpret_cast<const DevScalars *>(a.ws + a.lay.scalars);
    const int32_t *uniq = reinterpret_cast<const int32_t *>(a.ws + a.lay.sp_uniq);
    const int32_t *segoff = reinterpret_cast<const int32_t *>(a.ws + a.lay.sp_segoff);
    int64_t nb = (a.N + kThreads - 1) / kThreads;
    if (nb < 1)
        nb = 1;
    if (nb > 4 * kGridCtas)
        nb = 4 * kGridCtas;
    la.launch(k_sp_export, dim3((int)nb), dim3(kThreads), 0, la.pdl(), uniq, segoff, sc, a.N,
             uniq_out, counts_out, n_unique_out, reinterpret_cast<int32_t *>(a.ws + a.lay.sp_slot),
             reinterpret_cast<int32_t *>(a.ws + a.lay.sp_rng), kScanCounters);
    return finish(a, la);
}

}  // namespace ember
