// k_direct.cu -- the whole barcode path for clouds of up to kDirectMaxN points
// without sorting the edges (Rawson, Sec. 2; Sec. 4 steps 1-5).
//
// The reduction of Sec. 2 keeps n-1 of the n(n-1)/2 columns, the edges of the
// minimum spanning tree in the order (distance, u, v); of all other edges a
// bar only reads counts: its position `order` (edges before it) and its index
// a (distinct distances up to it).  At these sizes the keys fit the L2 cache
// (67 MB for both triangles at 2896 points), so the path finds the tree
// straight from the distance matrix and counts, in four launches instead of
// the sorted path's about forty:
//   memset           header and counters to zero,
//   k_direct_dist    step 1: the keys of both triangles; per row and block of
//                    columns the smallest key, where the tree search starts;
//                    every key once more in a bucket chosen by a hash,
//   k_direct_mst     steps 4-5 on one thread-block cluster: the tree by
//                    Boruvka's rounds (every component takes its first edge),
//                    its edges ordered, and their columns reduced by the claim
//                    rounds of k_reduce.cu, which give the pivot rows.  The
//                    other clusters find the repeated distances meanwhile
//                    (step 3), a bucket per CTA in a shared-memory hash table,
//   k_direct_count   every edge up to the last killing edge is counted at its
//                    place among the n-1 killing edges (a binary search); the
//                    last CTA to finish adds the counts up and writes the bars.
// Ties are ordered by (u, v) throughout, so the results equal the sorted
// path's bit for bit on any input (lattices, duplicate points, crowded
// distances): nothing depends on how the distances are spread.  Measured
// (device time of a call, uniform clouds): 256 points in 3 dimensions 65 us
// (dist 15, tree 36, count 14; the short sort's path 480 us), 700 in 2 104 us
// (470), 2048 in 3 195 us (62, 105, 29; 520), 2896 in 3 273 us (655).  The
// steps are bound by latency: the tree by its rounds' exchanges and dependent
// L2 reads.  kDirectMaxN ends at 2^22 edges: above, the matrix outgrows the L2
// cache and one cluster the tree's rounds, and k_large.cu takes over.
#include <cooperative_groups.h>

#include "emu64.cuh"
#include "ph0_common.cuh"

namespace cg = cooperative_groups;

namespace ph0 {

constexpr int kDirThreads = 1024;
constexpr int kDirCountThreads = 512;
constexpr int kDirMaxBuckets = 512;        // of kDirBucketLarge keys up to kDirectMaxN points
constexpr int kDirBucketSmall = 4096, kDirBucketLarge = 8192;
constexpr int kDirStrip = 32;              // rows of a tile staged at a time
#ifndef PH0_DIR_PROBES
#define PH0_DIR_PROBES 512
#endif
constexpr int kDirProbes = PH0_DIR_PROBES; // of a bucket's table, at most half full but for repeated distances
constexpr double kDirCrowd = 6.0;          // standard deviations over the mean that crowd a bucket
constexpr int kDirMaxRounds = 13;          // 2^12 > kDirectMaxN components halve each round
constexpr int kDirMstThreads = 1024;
constexpr int kDirOwn = 3;                 // columns per thread of the claim rounds
constexpr int kDirClaimRounds = 64;        // then one thread finishes in order
static_assert(kDirOwn * kDirMstThreads >= kDirectMaxN, "every column has a thread");
constexpr uint64_t kNoKey = kKeyBits;      // above every squared distance
constexpr size_t kDirDistSmem = 221 * 1024;
constexpr size_t kDirMstSmem = 224 * 1024;  // beside the static words, below the 227 KB of a CTA

struct DirectArgs {
    const float *pts;
    int64_t ld;
    int n, d, bt, nch, ldm;    // points, dimension, tile edge, tiles per side, row length of mat
    int buckets, bcap, table;  // hash buckets of keys, room of each, slots of its table
    uint64_t *bkeys;           // [buckets][bcap]
    uint32_t *bcount;          // [buckets] keys appended (beyond bcap: not stored)
    uint64_t *repk;            // [3 m / 4 + 1] repeated distances: key and how many occurrences
    uint32_t *repx;            //     it stands for beyond the one left (a key may have several records)
    uint32_t crowd;            // keys of a strip in one bucket that only repeated distances explain
    uint64_t *mat;             // [n][ldm] keys
    uint64_t *candk;           // [n][kDirectChunks] smallest key of each row and block of columns
    uint16_t *candv;           // ... and its column
    uint64_t *pkey;            // [n] the tree's edges in order: key,
    uint32_t *puv;             //     (u << 16) | v,
    uint32_t *plow;            //     pivot row
    int32_t *cnt, *corr, *dup; // [n] counts per place among the tree's edges
    Header *h;
    uint64_t *trace;
    ph0_bar *bars;
    ph0_inf_bar *inf;
};

// Least value of a 64-bit key over the warp and the lowest lane that holds it.
__device__ __forceinline__ int warp_argmin(uint64_t k, uint64_t &mn) {
    const uint32_t hi = uint32_t(k >> 32);
    const uint32_t mh = __reduce_min_sync(0xffffffffu, hi);
    const uint32_t lo = hi == mh ? uint32_t(k) : 0xffffffffu;
    const uint32_t ml = __reduce_min_sync(0xffffffffu, lo);
    const unsigned who = __ballot_sync(0xffffffffu, hi == mh && lo == ml);
    mn = (uint64_t(mh) << 32) | ml;
    return __ffs(who) - 1;
}

// key_hash: the bucket from the high bits, the slot in its table from the low ones.
__device__ __forceinline__ uint32_t hash_bucket(uint64_t x, int buckets) {
    return __umulhi(uint32_t(x >> 32), uint32_t(buckets));
}
__device__ __forceinline__ uint32_t hash_slot(uint64_t x, int table) {
    return uint32_t(x >> 8) & uint32_t(table - 1);
}

// ------------------------------------------------------------- distances ---
// One CTA per tile of the upper triangle, as k_dist (same staging and
// arithmetic), in strips of 32 rows: the strip's keys go to shared memory,
// from where both triangles of the matrix are written in whole rows and the
// row and column minima of the tile are taken.  1024 threads with one to four
// keys each: at these sizes there are few tiles per SM and the time is the
// latency of the steps.  The keys of the upper triangle are also appended to
// the hash buckets, one counter addition per strip and bucket (a global hash
// table with one compare-and-swap per key took 14 us of 28 at 256 points: an
// SM gets about one such atomic back per ten clocks).  A strip that crowds a
// bucket (kDirCrowd standard deviations over the mean, which distinct keys
// reach in one strip of hundreds) holds repeated distances: it appends one
// key of each and records the others as repeats at once, so that lattices
// and the like do not overflow the buckets (14^3 lattice points: 2744 points,
// 299 distances; without this step 4.6 ms a call, the sorted path 0.63).
template <int D, int BT>
__global__ void __launch_bounds__(kDirThreads) k_direct_dist(const DirectArgs A) {
    const int n = A.n, d = D > 0 ? D : A.d;
    constexpr int bt = BT;
    extern __shared__ double s_coord[];
    __shared__ uint64_t s_min[kDirThreads / 32], s_max[kDirThreads / 32];
    __shared__ int s_fixed;
    __shared__ uint32_t s_bcnt[kDirMaxBuckets], s_bbase[kDirMaxBuckets];
    __shared__ uint32_t s_nrep, s_rbase, s_extra;
    double *su = s_coord, *sv = s_coord + size_t(d) * bt;
    int64_t *xu = reinterpret_cast<int64_t *>(su), *xv = reinterpret_cast<int64_t *>(sv);
    uint64_t *s_strip = reinterpret_cast<uint64_t *>(s_coord + size_t(2) * d * bt);  // [32][bt + 1]
    uint64_t *s_colk = s_strip + kDirStrip * (bt + 1);                               // [bt]
    int32_t *s_g = reinterpret_cast<int32_t *>(s_colk + bt);
    int32_t *s_lo = s_g + d, *s_hi = s_lo + d;
    uint32_t *s_first = reinterpret_cast<uint32_t *>(s_hi + d), *s_last = s_first + d;
    uint32_t *s_narrow = s_last + d;  // [(d+31)/32]
    uint16_t *s_colv = reinterpret_cast<uint16_t *>(s_narrow + (d + 31) / 32);  // [bt]
    // a crowded strip's hash table of the places of its distinct keys, and
    // their occurrences (two 16-bit counts per word; bt is even)
    uint16_t *s_tab = s_colv + bt;                                                // [2 * 32 * bt]
    uint32_t *s_occ = reinterpret_cast<uint32_t *>(s_tab + 2 * kDirStrip * bt);   // [32 * bt / 2]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kDirThreads / 32;
    static_assert(kWarps == 32, "one warp reduces the others' values");

    // tile (bi, bj), bi <= bj, row-major over the upper triangle
    int bi = 0, rest = blockIdx.x;
    while (rest >= A.nch - bi) {
        rest -= A.nch - bi;
        ++bi;
    }
    const int bj = bi + rest;
    const int u0 = bi * bt, v0 = bj * bt;

    for (int k = tid; k < d; k += kDirThreads) {
        s_lo[k] = 1 << 30;
        s_hi[k] = -(1 << 30);
        s_first[k] = ~0u;
        s_last[k] = 0;
    }
    for (int j = tid; j < bt; j += kDirThreads) s_colk[j] = kNoKey;
    // the trace of an earlier call's reduction (this form keeps one record)
    for (int i = blockIdx.x * kDirThreads + tid; i < kTraceWindows * kTraceWords; i += gridDim.x * kDirThreads)
        A.trace[i] = 0;
    __syncthreads();
    // coordinates, finiteness and the span of set bits per dimension
    bool bad = false;
    for (int idx = tid; idx < 2 * bt * d; idx += kDirThreads) {
        const int side = idx >= bt * d, r = idx - side * bt * d;
        const int p = r / d, k = r - p * d;
        const int row = (side ? v0 : u0) + p;
        const float x = row < n ? A.pts[int64_t(row) * A.ld + k] : 0.0f;
        const uint32_t b = __float_as_uint(x);
        if ((b & 0x7f800000u) == 0x7f800000u) {
            bad = true;
        } else {
            if (row < n) {
                const uint32_t o = emu::order_f32(b);
                if (o < *(volatile uint32_t *)(s_first + k)) atomicMin(s_first + k, o);
                if (o > *(volatile uint32_t *)(s_last + k)) atomicMax(s_last + k, o);
            }
            if (b & 0x7fffffffu) {
                int32_t lo, hi;
                emu::bit_range_f32(b, lo, hi);
                if (lo < *(volatile int32_t *)(s_lo + k)) atomicMin(s_lo + k, lo);
                if (hi > *(volatile int32_t *)(s_hi + k)) atomicMax(s_hi + k, hi);
            }
        }
        (side ? xv : xu)[k * bt + p] = int64_t(b);
    }
    if (bad) set_status(A.h, PH0_ENONFINITE);
    __syncthreads();
    if (warp == 0) {
        bool wide = false;
        for (int w = 0; w < (d + 31) / 32; ++w) {
            const int k = w * 32 + lane;
            bool nar = false;
            if (k < d) {
                const bool zero = s_lo[k] == (1 << 30);
                s_g[k] = zero ? 0 : s_lo[k];
                const int span = zero ? 0 : s_hi[k] + 1 - s_lo[k];
                if (span > 52) wide = true;
                nar = span <= 52 && emu::within_32_bits(s_first[k], s_last[k], s_g[k]);
            }
            const unsigned bits = __ballot_sync(0xffffffffu, nar);
            if (lane == 0) s_narrow[w] = bits;
        }
        wide = __any_sync(0xffffffffu, wide);
        if (lane == 0) {
            s_fixed = !wide;
            atomicAdd(&A.h->dist_tiles, 1ull);
            if (!wide) atomicAdd(&A.h->dist_tiles_exact_int, 1ull);
        }
    }
    __syncthreads();
    const bool fixed = s_fixed != 0;
    for (int idx = tid; idx < 2 * bt * d; idx += kDirThreads) {
        int64_t *x = xu + idx;  // xv follows xu
        const uint32_t b = uint32_t(*x);
        if (fixed) *x = emu::to_fixed(b, s_g[(idx / bt) % d]);
        else su[idx] = double(__uint_as_float(b));
    }
    __syncthreads();

    const int j = tid % bt, v = v0 + j, rpp = kDirThreads / bt;
    const bool diag = bi == bj;
    const uint32_t nw = s_narrow[0];
    uint64_t kmin = ~0ull, kmax = 0;
    constexpr int kPer = kDirStrip * 128 / kDirThreads;  // keys per thread and strip, at most
    for (int s0 = 0; s0 < bt; s0 += kDirStrip) {
        for (int b = tid; b < A.buckets; b += kDirThreads) s_bcnt[b] = 0;
        // the strip's keys (a thread's rows of its column)
#pragma unroll 1
        for (int i = s0 + tid / bt; i < s0 + kDirStrip; i += rpp) {
            const int u = u0 + i;
            uint64_t kb = kNoKey;
            if (u < n && v < n && u != v) {
                if (fixed) {
                    if constexpr (D > 0) kb = emu::sq_dist_mixed_ct<D, BT>(xu + i, xv + j, s_g, nw);
                    else kb = emu::sq_dist_mixed_st<BT>(xu + i, xv + j, s_g, d, s_narrow);
                } else {
                    double s = 0.0;
                    for (int k = 0; k < d; ++k) {
                        const double t = __dsub_rn(sv[k * bt + j], su[k * bt + i]);
                        s = __dadd_rn(s, __dmul_rn(t, t));
                    }
                    kb = uint64_t(__double_as_longlong(s));
                }
                kb &= kKeyBits;
                if (u < v) {
                    kmin = kb < kmin ? kb : kmin;
                    kmax = kb > kmax ? kb : kmax;
                }
            }
            s_strip[(i - s0) * (bt + 1) + j] = kb;
        }
        __syncthreads();
        // the place of each key of the upper triangle among the strip's keys of its bucket
        uint32_t place[kPer];
        bool crowded = false;
#pragma unroll
        for (int w = 0; w < kPer; ++w) {
            const int i = tid / bt + w * rpp;
            if (i < kDirStrip && u0 + s0 + i < v && v < n) {
                place[w] = atomicAdd(s_bcnt + hash_bucket(key_hash(s_strip[i * (bt + 1) + j]), A.buckets), 1u);
                crowded |= place[w] >= A.crowd;
            }
        }
        if (__syncthreads_or(crowded)) {
            const uint32_t slots = uint32_t(2 * kDirStrip * bt);
            uint32_t *tab32 = reinterpret_cast<uint32_t *>(s_tab);
            for (uint32_t i = tid; i < slots / 2; i += kDirThreads) tab32[i] = 0xffffffffu;
            for (int i = tid; i < kDirStrip * bt / 2; i += kDirThreads) s_occ[i] = 0;
            for (int b = tid; b < A.buckets; b += kDirThreads) s_bcnt[b] = 0;
            if (tid == 0) s_nrep = s_extra = 0;
            __syncthreads();
            // one key of each distance keeps its place, the others count for it
            uint32_t mine = 0;
#pragma unroll
            for (int w = 0; w < kPer; ++w) {
                const int i = tid / bt + w * rpp;
                if (i >= kDirStrip || u0 + s0 + i >= v || v >= n) continue;
                const uint64_t k = s_strip[i * (bt + 1) + j];
                uint32_t slot = hash_slot(key_hash(k), int(slots));
                for (uint32_t pr = 0; pr < slots; ++pr) {  // at most half the slots fill
                    uint32_t old = *(volatile uint16_t *)(s_tab + slot);
                    if (old == 0xffffu)
                        old = atomicCAS(s_tab + slot, (unsigned short)0xffffu, (unsigned short)(i * bt + j));
                    const uint32_t at = old == 0xffffu ? uint32_t(i * bt + j) : old;
                    if (old == 0xffffu) mine |= 1u << w;
                    if (old == 0xffffu || s_strip[(at / bt) * (bt + 1) + at % bt] == k) {
                        atomicAdd(s_occ + at / 2, 1u << (16 * (at & 1)));
                        break;
                    }
                    slot = (slot + 1) & (slots - 1);
                }
                place[w] = 0xffffffffu;
            }
            __syncthreads();
            uint32_t at[kPer];
#pragma unroll
            for (int w = 0; w < kPer; ++w) {
                if (!((mine >> w) & 1u)) continue;
                const int i = tid / bt + w * rpp, x = i * bt + j;
                const uint32_t extra = ((s_occ[x / 2] >> (16 * (x & 1))) & 0xffffu) - 1;
                place[w] = atomicAdd(s_bcnt + hash_bucket(key_hash(s_strip[i * (bt + 1) + j]), A.buckets), 1u);
                if (extra) {
                    at[w] = atomicAdd(&s_nrep, 1u);
                    atomicAdd(&s_extra, extra);
                } else {
                    mine &= ~(1u << w);
                }
            }
            __syncthreads();
            if (tid == 0 && s_nrep) {
                s_rbase = atomicAdd(&A.h->direct_strips, s_nrep);
                atomicAdd(&A.h->direct_dups, s_extra);
            }
            __syncthreads();
#pragma unroll
            for (int w = 0; w < kPer; ++w) {
                if (!((mine >> w) & 1u)) continue;
                const int i = tid / bt + w * rpp, x = i * bt + j;
                A.repk[s_rbase + at[w]] = s_strip[i * (bt + 1) + j];
                A.repx[s_rbase + at[w]] = ((s_occ[x / 2] >> (16 * (x & 1))) & 0xffffu) - 1;
            }
        }
        uint32_t base = 0;
        if (tid < A.buckets && s_bcnt[tid]) base = atomicAdd(A.bcount + tid, s_bcnt[tid]);
        // rows: the upper triangle (a diagonal tile: all of the tile)
        for (int i = warp; i < kDirStrip; i += kWarps) {
            const int u = u0 + s0 + i;
            if (u >= n) break;
            uint64_t best = kNoKey;
            int bv = 0;
            for (int c = lane; c < bt && v0 + c < n; c += 32) {
                const uint64_t k = s_strip[i * (bt + 1) + c];
                A.mat[size_t(u) * A.ldm + v0 + c] = k;
                if (k < best) {
                    best = k;
                    bv = v0 + c;
                }
            }
            uint64_t mn;
            warp_argmin(best, mn);
            const uint32_t mv = __reduce_min_sync(0xffffffffu, best == mn ? uint32_t(bv) : 0xffffu);
            if (lane == 0) {
                A.candk[size_t(u) * kDirectChunks + bj] = mn;
                A.candv[size_t(u) * kDirectChunks + bj] = uint16_t(mv);
            }
        }
        // columns: the lower triangle
        if (!diag) {
            for (int c = warp; c < bt && v0 + c < n; c += kWarps) {
                const int u = u0 + s0 + lane;  // below n: bi < bj
                const uint64_t k = s_strip[lane * (bt + 1) + c];
                A.mat[size_t(v0 + c) * A.ldm + u] = k;
                uint64_t mn;
                const int src = warp_argmin(k, mn);
                if (lane == 0 && mn < s_colk[c]) {  // equal keys: the earlier strip's row stays
                    s_colk[c] = mn;
                    s_colv[c] = uint16_t(u0 + s0 + src);
                }
            }
        }
        if (tid < A.buckets) s_bbase[tid] = base;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kPer; ++w) {
            const int i = tid / bt + w * rpp;
            if (i < kDirStrip && u0 + s0 + i < v && v < n && place[w] != 0xffffffffu) {
                const uint64_t k = s_strip[i * (bt + 1) + j];
                const uint32_t b = hash_bucket(key_hash(k), A.buckets), at = s_bbase[b] + place[w];
                if (at < uint32_t(A.bcap)) A.bkeys[size_t(b) * A.bcap + at] = k;
            }
        }
        __syncthreads();
    }
    if (!diag) {
        for (int c = tid; c < bt && v0 + c < n; c += kDirThreads) {
            A.candk[size_t(v0 + c) * kDirectChunks + bi] = s_colk[c];
            A.candv[size_t(v0 + c) * kDirectChunks + bi] = s_colv[c];
        }
    }
    // key range
    uint64_t t;
    warp_argmin(kmin, t);
    if (lane == 0) s_min[warp] = t;
    warp_argmin(~kmax, t);
    if (lane == 0) s_max[warp] = ~t;
    __syncthreads();
    if (warp == 0) {
        warp_argmin(s_min[lane], kmin);
        warp_argmin(~s_max[lane], kmax);
        kmax = ~kmax;
        if (lane == 0 && kmin != ~0ull) {
            // the header starts at zero: the minimum is kept as its complement
            atomicMax((unsigned long long *)&A.h->direct_nkmin, (unsigned long long)~kmin);
            atomicMax((unsigned long long *)&A.h->kmax, (unsigned long long)kmax);
        }
    }
}

// ------------------------------------------------------------------ tree ---
__device__ __forceinline__ bool before(uint64_t ka, uint32_t ua, uint64_t kb, uint32_t ub) {
    return ka < kb || (ka == kb && ua < ub);
}

__device__ __forceinline__ uint32_t dir_find(uint16_t *par, uint32_t x) {
    volatile uint16_t *p = par;
    for (;;) {
        const uint32_t a = p[x];
        if (a == x) return x;
        const uint32_t b = p[a];
        p[x] = uint16_t(b);  // path halving (benign race: only moves toward the root)
        x = b;
    }
}

// Shared memory of the tree kernel for n points on clusters of cl CTAs.
struct DirMst {
    int npad, R;
    size_t rbk, ck, bk, ub, mk, buv, muv, rbv, cv, comp, par, sel, total;
    __host__ __device__ DirMst(int n, int cl) {
        npad = n + 16;
        R = (n + cl - 1) / cl;
        size_t off = 0;
        auto take = [&](size_t b) {
            const size_t o = off;
            off = align_up(off + b, 16);
            return o;
        };
        rbk = take(16 * size_t(npad));
        ck = take(8 * size_t(R) * kDirectChunks);
        bk = take(8 * size_t(npad));
        ub = take(8 * size_t(npad));
        mk = take(8 * size_t(npad));
        buv = take(4 * size_t(npad));
        muv = take(4 * size_t(npad));
        rbv = take(4 * size_t(npad));
        cv = take(2 * size_t(R) * kDirectChunks);
        comp = take(2 * size_t(npad));
        par = take(2 * size_t(npad));
        sel = take(2 * size_t(npad));
        total = off;
    }
};

// The repeated distances of the buckets first, first + step, ...: a hash table
// of (key + 1, occurrences) in shared memory per bucket.  A bucket whose keys
// did not fit its room (distances that occur many times, but seldom within a
// strip) takes the upper triangle's keys from the matrix instead, with the
// repeats that crowded strips recorded taken off.  The hash spreads distinct
// keys evenly, the mean is at most half the table, and a bucket whose distinct
// keys do not fit all the same (a key finds no slot in kDirProbes) is taken in
// two halves by bits of the hash, and so on: a one-to-one hash ends that
// at one key.
__device__ void direct_repeats(const DirectArgs &A, unsigned char *s_dyn, int first, int step) {
    unsigned long long *s_key = reinterpret_cast<unsigned long long *>(s_dyn);
    uint32_t *s_occ = reinterpret_cast<uint32_t *>(s_key + A.table);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    int bits = 0;  // of the hash, those of the part looked at
    uint64_t part = 0;
    bool full = false;
    // (the bucket comes from the hash's high word, the slot from bits 8 to 21)
    auto within = [&](uint64_t x) { return bits == 0 || (x << 32 | x >> 32) >> (64 - bits) == part; };
    auto insert = [&](uint64_t key, uint64_t x) {
        const unsigned long long tag = key + 1;
        uint32_t slot = hash_slot(x, A.table);
        for (int pr = 0; pr < kDirProbes; ++pr) {
            unsigned long long old = *(volatile unsigned long long *)(s_key + slot);
            if (old == 0) old = atomicCAS(s_key + slot, 0ull, tag);
            if (old == 0 || old == tag) {
                atomicAdd(s_occ + slot, 1u);
                return;
            }
            slot = (slot + 1) & uint32_t(A.table - 1);
        }
        full = true;
    };
    for (int b = first; b < A.buckets;) {
        for (int i = tid; i < A.table; i += T) {
            s_key[i] = 0;
            s_occ[i] = 0;
        }
        __syncthreads();
        const uint32_t cnt = A.bcount[b];
        const bool stored = cnt <= uint32_t(A.bcap);
        if (stored) {
            const uint64_t *keys = A.bkeys + size_t(b) * A.bcap;
            if (bits == 0) {  // nearly always
                for (uint32_t i = tid; i < cnt; i += T) {
                    const uint64_t k = keys[i];
                    insert(k, key_hash(k));
                }
            } else {
                for (uint32_t i = tid; i < cnt; i += T) {
                    const uint64_t k = keys[i], x = key_hash(k);
                    if (within(x)) insert(k, x);
                }
            }
        } else {
            const uint32_t n = uint32_t(A.n), items = n * n;
            for (uint32_t i0 = tid; i0 < items; i0 += 8 * T) {
                uint64_t key[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint32_t i = i0 + q * T, u = i / n, v = i - u * n;
                    key[q] = i < items && u < v ? __ldcg(A.mat + size_t(u) * A.ldm + v) : kNoKey;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint64_t x = key_hash(key[q]);
                    if (key[q] != kNoKey && hash_bucket(x, A.buckets) == uint32_t(b) && within(x)) insert(key[q], x);
                }
            }
        }
        full = __syncthreads_or(full);
        if (full) {
            full = false;
            ++bits;
            part <<= 1;
            continue;
        }
        if (!stored) {
            const uint32_t strips = A.h->direct_strips;
            for (uint32_t r = tid; r < strips; r += T) {
                const uint64_t k = A.repk[r], x = key_hash(k);
                if (hash_bucket(x, A.buckets) != uint32_t(b) || !within(x)) continue;
                uint32_t slot = hash_slot(x, A.table);
                for (int pr = 0; pr < A.table && s_key[slot] != k + 1; ++pr) slot = (slot + 1) & uint32_t(A.table - 1);
                if (s_key[slot] == k + 1) atomicSub(s_occ + slot, A.repx[r]);
            }
            __syncthreads();
        }
        uint32_t extra = 0;
        for (int i = tid; i < A.table; i += T) {
            const uint32_t o = s_occ[i];
            if (o > 1) {
                const uint32_t q = A.h->direct_strips + atomicAdd(&A.h->direct_repeats, 1u);
                A.repk[q] = s_key[i] - 1;
                A.repx[q] = o - 1;
                extra += o - 1;
            }
        }
        extra = __reduce_add_sync(0xffffffffu, extra);
        if (lane == 0 && extra) atomicAdd(&A.h->direct_dups, extra);
        __syncthreads();
        // the next half, or bucket
        while (bits > 0 && (part & 1)) {
            part >>= 1;
            --bits;
        }
        if (bits > 0) part |= 1;
        else b += step;
    }
}

// Cluster 0 finds the tree.  CTA r owns rows u = r (mod CTAs); every CTA keeps
// the components of all vertices, so a round needs one exchange: each row's
// first edge that leaves its component, written into every CTA's shared
// memory.  A row keeps the smallest key of each block of BT columns.  When
// that entry's column has joined the row's component the block's next key is
// at least as large, so the entry is still a bound: a block is read again only
// when its bound is not above the row's and the component's best entry that is
// still valid (a few blocks per row over the whole search instead of the row
// in every round), and up to eight 32-column reads are in flight at a time.
template <int BT>
__global__ void __launch_bounds__(kDirMstThreads, 1) k_direct_mst(const DirectArgs A) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    cg::cluster_group cluster = cg::this_cluster();
    const int cl = int(cluster.num_blocks()), rank = int(cluster.block_rank());
    if (int(blockIdx.x) >= cl) {
        direct_repeats(A, s_dyn, int(blockIdx.x) - cl, int(gridDim.x) - cl);
        return;
    }
    constexpr int kReads = BT / 32, kBlocks = 8 / kReads;  // reads per block, blocks at a time
    const int n = A.n, nch = A.nch;
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const DirMst S(n, cl);
    uint64_t *s_rbk = reinterpret_cast<uint64_t *>(s_dyn + S.rbk);  // [2][npad] rows' first edges: key,
    uint16_t *s_rbv = reinterpret_cast<uint16_t *>(s_dyn + S.rbv);  // [2][npad] other end
    uint64_t *s_ck = reinterpret_cast<uint64_t *>(s_dyn + S.ck);    // [R][chunks] own rows' block minima
    uint16_t *s_cv = reinterpret_cast<uint16_t *>(s_dyn + S.cv);
    unsigned long long *s_ub = reinterpret_cast<unsigned long long *>(s_dyn + S.ub);  // [n] best valid entry (own rows)
    unsigned long long *s_bk = reinterpret_cast<unsigned long long *>(s_dyn + S.bk);  // [n] per component: key,
    uint32_t *s_buv = reinterpret_cast<uint32_t *>(s_dyn + S.buv);                    // (u << 16) | v
    uint64_t *s_mk = reinterpret_cast<uint64_t *>(s_dyn + S.mk);    // [n] tree edge of each absorbed component
    uint32_t *s_muv = reinterpret_cast<uint32_t *>(s_dyn + S.muv);
    uint16_t *s_comp = reinterpret_cast<uint16_t *>(s_dyn + S.comp);
    uint16_t *s_par = reinterpret_cast<uint16_t *>(s_dyn + S.par);
    uint16_t *s_sel = reinterpret_cast<uint16_t *>(s_dyn + S.sel);  // [n] component at the other end
    const int own = n > rank ? (n - rank + cl - 1) / cl : 0;  // rows of this CTA
    // no CTA writes to another's shared memory before all have started
    cluster.barrier_arrive();

    for (int u = tid; u < n; u += T) {
        s_comp[u] = uint16_t(u);
        s_par[u] = uint16_t(u);
        s_mk[u] = kNoKey;
        s_muv[u] = 0xffffffffu;
        s_ub[u] = kNoKey;
    }
    for (int k = warp; k < own; k += nw) {
        const size_t g = size_t(k * cl + rank) * kDirectChunks + lane;
        s_ck[k * kDirectChunks + lane] = lane < nch ? A.candk[g] : kNoKey;
        s_cv[k * kDirectChunks + lane] = lane < nch ? A.candv[g] : uint16_t(0);
    }
    int buf = 0;
    bool more = n > 1;
    cluster.barrier_wait();
    for (int round = 0; round < kDirMaxRounds && more; ++round) {
        buf = round & 1;
        for (int c = tid; c < n; c += T) {
            s_bk[c] = kNoKey;
            s_buv[c] = 0xffffffffu;
        }
        __syncthreads();
        // the best valid entry of each component over this CTA's rows
        if (round > 0) {
            for (int k = warp; k < own; k += nw) {
                const uint32_t cu = s_comp[k * cl + rank];
                uint64_t key = s_ck[k * kDirectChunks + lane], mn;
                if (key != kNoKey && s_comp[s_cv[k * kDirectChunks + lane]] == cu) key = kNoKey;
                warp_argmin(key, mn);
                if (lane == 0 && mn < *(volatile unsigned long long *)&s_ub[cu])
                    atomicMin(&s_ub[cu], (unsigned long long)mn);
            }
            __syncthreads();
        }
        for (int k = warp; k < own; k += nw) {
            const int u = k * cl + rank;
            const uint32_t cu = s_comp[u];
            const uint64_t *row = A.mat + size_t(u) * A.ldm;
            uint64_t key = s_ck[k * kDirectChunks + lane], mn;
            uint32_t v = s_cv[k * kDirectChunks + lane];
            const uint64_t ub = *(volatile unsigned long long *)&s_ub[cu];
            bool changed = false;
            int src;
            for (;;) {
                const bool inside = key != kNoKey && s_comp[v] == cu;
                src = warp_argmin(inside ? kNoKey : key, mn);  // equal keys: the earlier block
                const uint64_t lim = mn < ub ? mn : ub;
                unsigned need = __ballot_sync(0xffffffffu, inside && key <= lim);
                if (!need) break;
                // read these blocks again: the first key outside the component
                changed = true;
                int blk[kBlocks];
                uint64_t raw[8];
#pragma unroll
                for (int s = 0; s < kBlocks; ++s) {
                    blk[s] = need ? __ffs(need) - 1 : -1;
                    need &= need - 1;
#pragma unroll
                    for (int q = 0; q < kReads; ++q) {
                        const int c = blk[s] * BT + q * 32 + lane;
                        raw[s * kReads + q] = blk[s] >= 0 && c < n ? __ldcg(row + c) : kNoKey;
                    }
                }
#pragma unroll
                for (int s = 0; s < kBlocks; ++s) {
                    if (blk[s] < 0) continue;
                    uint64_t best = kNoKey, bm;
                    uint32_t bv = 0xffffu;
#pragma unroll
                    for (int q = 0; q < kReads; ++q) {
                        const int c = blk[s] * BT + q * 32 + lane;
                        if (c < n && raw[s * kReads + q] < best && s_comp[c] != cu) {
                            best = raw[s * kReads + q];
                            bv = uint32_t(c);
                        }
                    }
                    warp_argmin(best, bm);
                    const uint32_t mv = __reduce_min_sync(0xffffffffu, best == bm ? bv : 0xffffu);
                    if (lane == blk[s]) {
                        key = bm;
                        v = bm == kNoKey ? 0u : mv;
                    }
                }
            }
            if (changed) {
                s_ck[k * kDirectChunks + lane] = key;
                s_cv[k * kDirectChunks + lane] = uint16_t(v);
            }
            const uint32_t vm = __shfl_sync(0xffffffffu, v, src);
            if (lane == 0 && mn < ub) atomicMin(&s_ub[cu], (unsigned long long)mn);
            if (lane < cl) {
                *cluster.map_shared_rank(s_rbk + buf * S.npad + u, lane) = mn > ub ? kNoKey : mn;
                *cluster.map_shared_rank(s_rbv + buf * S.npad + u, lane) = uint16_t(vm);
            }
        }
        cluster.sync();
        // every CTA merges the components alike
        const uint64_t *rk = s_rbk + buf * S.npad;
        const uint16_t *rv = s_rbv + buf * S.npad;
        for (int u = tid; u < n; u += T) {
            const uint64_t k = rk[u];
            const uint32_t c = s_comp[u];
            s_ub[u] = kNoKey;
            if (k < *(volatile unsigned long long *)&s_bk[c]) atomicMin(&s_bk[c], (unsigned long long)k);
        }
        __syncthreads();
        for (int u = tid; u < n; u += T) {
            const uint64_t k = rk[u];
            const uint32_t c = s_comp[u], v = rv[u];
            if (k != kNoKey && k == s_bk[c])
                atomicMin(&s_buv[c], uint32_t(u) < v ? (uint32_t(u) << 16) | v : (v << 16) | uint32_t(u));
        }
        __syncthreads();
        for (int c = tid; c < n; c += T) {
            uint32_t o = uint32_t(c);
            if (s_comp[c] == c && s_bk[c] != kNoKey) {
                const uint32_t uv = s_buv[c], a = s_comp[uv >> 16], b = s_comp[uv & 0xffffu];
                o = a == uint32_t(c) ? b : a;
            }
            s_sel[c] = uint16_t(o);
        }
        __syncthreads();
        for (int c = tid; c < n; c += T) {
            const uint32_t o = s_sel[c];
            // of two components that chose the same edge the smaller stays a root
            if (s_comp[c] != c || o == uint32_t(c) || (s_sel[o] == c && uint32_t(c) < o)) continue;
            s_par[c] = uint16_t(o);  // absorbed: once in the whole search
            s_mk[c] = s_bk[c];
            s_muv[c] = s_buv[c];
        }
        __syncthreads();
        uint32_t r0 = 0;
        for (uint32_t p; (p = s_par[r0]) != r0;) r0 = p;
        bool apart = false;
        for (int u = tid; u < n; u += T) {
            uint32_t r = s_comp[u];
            for (uint32_t p; (p = s_par[r]) != r;) r = p;
            s_comp[u] = uint16_t(r);
            apart |= r != r0;
        }
        more = __syncthreads_or(apart);  // the same in every CTA
    }
    if (more && rank == 0 && tid == 0) set_status(A.h, PH0_EINTERNAL);  // keys that are not numbers

    // ---- the tree's edges in order: each CTA sorts its share, then finds its
    // edges' places in the others' runs (the one root left comes last) ----
    const int alt = buf ^ 1;
    uint64_t *run_k = s_rbk + alt * S.npad;                       // [cl][R]
    uint32_t *run_uv = reinterpret_cast<uint32_t *>(s_ck);        // [cl][R]
    static_assert(2 * kDirectChunks >= 16, "the runs' edges fit the block minima");
    uint64_t *own_k = reinterpret_cast<uint64_t *>(s_bk);         // [own]
    uint32_t *own_uv = s_buv, *s_rank = reinterpret_cast<uint32_t *>(s_ub);
    for (int i = tid; i < own; i += T) {
        own_k[i] = s_mk[i * cl + rank];
        own_uv[i] = s_muv[i * cl + rank];
        s_rank[i] = 0;
    }
    __syncthreads();
    for (int i = warp; i < own; i += nw) {
        const uint64_t k = own_k[i];
        const uint32_t uv = own_uv[i];
        uint32_t less = 0;
        for (int q = lane; q < own; q += 32) less += before(own_k[q], own_uv[q], k, uv);
        less = __reduce_add_sync(0xffffffffu, less);
        if (lane < cl) {
            *cluster.map_shared_rank(run_k + rank * S.R + less, lane) = k;
            *cluster.map_shared_rank(run_uv + rank * S.R + less, lane) = uv;
        }
    }
    cluster.sync();
    const int lcl = __ffs(cl) - 1;  // clusters of 8 or 16
    for (int x = tid; x < own * cl; x += T) {
        const int i = x >> lcl, r = x & (cl - 1);
        const uint64_t k = run_k[rank * S.R + i];
        const uint32_t uv = run_uv[rank * S.R + i];
        int lo = 0, hi = n > r ? (n - r + cl - 1) / cl : 0;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (before(run_k[r * S.R + mid], run_uv[r * S.R + mid], k, uv)) lo = mid + 1;
            else hi = mid;
        }
        if (lo) atomicAdd(&s_rank[i], uint32_t(lo));
    }
    __syncthreads();
    for (int i = tid; i < own; i += T) {  // to CTA 0, whose tree-edge slots are free now
        const uint32_t p = s_rank[i];
        *cluster.map_shared_rank(s_mk + p, 0) = run_k[rank * S.R + i];
        *cluster.map_shared_rank(s_muv + p, 0) = run_uv[rank * S.R + i];
    }
    cluster.sync();
    if (rank != 0) return;

    // ---- the columns' pivot rows: claim rounds as in k_reduce.cu, on the
    // n-1 nonzero columns alone, priority to the lower position ----
    uint32_t *s_res = s_buv;
    uint16_t *s_low = s_comp;
    for (int c = tid; c < n; c += T) {
        s_par[c] = uint16_t(c);
        s_res[c] = 0xffffffffu;
        s_low[c] = 0xffffu;
    }
    __syncthreads();
    uint32_t act = 0, eu[kDirOwn], ev[kDirOwn], claims = 0;
#pragma unroll
    for (int q = 0; q < kDirOwn; ++q) {
        const int p = tid + q * T;
        const uint32_t uv = p < n - 1 ? s_muv[p] : 0u;
        eu[q] = uv >> 16;
        ev[q] = uv & 0xffffu;
        if (p < n - 1 && eu[q] < ev[q] && ev[q] < uint32_t(n)) act |= 1u << q;
    }
    int rounds = 0;
    while (__syncthreads_or(act != 0) && rounds < kDirClaimRounds) {
        ++rounds;
        uint32_t a[kDirOwn], b[kDirOwn];
#pragma unroll
        for (int q = 0; q < kDirOwn; ++q) {
            if (!((act >> q) & 1u)) continue;
            a[q] = dir_find(s_par, eu[q]);
            b[q] = dir_find(s_par, ev[q]);
            atomicMin(s_res + a[q], uint32_t(tid + q * T));
            atomicMin(s_res + b[q], uint32_t(tid + q * T));
            claims += 2;
        }
        __syncthreads();
        const uint32_t was = act;
#pragma unroll
        for (int q = 0; q < kDirOwn; ++q) {
            if (!((act >> q) & 1u)) continue;
            const uint32_t hi = a[q] > b[q] ? a[q] : b[q], lo = a[q] > b[q] ? b[q] : a[q];
            if (s_res[hi] == uint32_t(tid + q * T)) {
                s_par[hi] = uint16_t(lo);
                s_low[tid + q * T] = uint16_t(hi);
                act &= ~(1u << q);
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kDirOwn; ++q) {
            if (!((was >> q) & 1u)) continue;
            s_res[a[q]] = 0xffffffffu;
            s_res[b[q]] = 0xffffffffu;
        }
    }
    __syncthreads();
    if (tid == 0 && rounds == kDirClaimRounds) {  // long chains of waiting columns: in order
        for (int p = 0; p < n - 1; ++p) {
            if (s_low[p] != 0xffffu) continue;
            const uint32_t uv = s_muv[p];
            if ((uv >> 16) >= (uv & 0xffffu) || (uv & 0xffffu) >= uint32_t(n)) continue;
            const uint32_t a = dir_find(s_par, uv >> 16), b = dir_find(s_par, uv & 0xffffu);
            s_par[a > b ? a : b] = uint16_t(a > b ? b : a);
            s_low[p] = uint16_t(a > b ? a : b);
        }
    }
    __syncthreads();
    for (int p = tid; p < n - 1; p += T) {
        A.pkey[p] = s_mk[p];
        A.puv[p] = s_muv[p];
        A.plow[p] = s_low[p];
    }
    claims = __reduce_add_sync(0xffffffffu, claims);
    if (lane == 0 && claims) atomicAdd(&A.h->claim_attempts, (unsigned long long)claims);
    if (tid == 0) {
        const int64_t m = n_edges(n);
        A.h->windows = 1;
        A.h->edges_scanned = m;
        A.h->sorted_edges = m;
        A.h->candidates = n - 1;
        A.h->rounds = rounds;
        A.h->claim_rounds_max = uint32_t(rounds);
        A.h->n_bars = n - 1;
        A.trace[1] = uint64_t(m);
        A.trace[2] = uint64_t(n - 1);
        A.trace[4] = uint64_t(rounds);
        A.trace[5] = uint64_t(n - 1);
    }
}

// ---------------------------------------------------------- counts, bars ---
// With the tree's edges p in order, s(e) of an edge e = tree edges before it,
// t(e) = tree edges of a smaller key: order(p) counts the edges other than p
// with s(e) <= p, and a(p) the edges with t(e) <= p less the repeated ones
// (dup).  s and t differ only for edges as long as a tree edge (corr moves
// those).  Edges beyond the
// last killing edge, most of a cloud's, are read and dropped.
__global__ void __launch_bounds__(kDirCountThreads, 2) k_direct_count(const DirectArgs A) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int n = A.n, np = n - 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t *s_key = reinterpret_cast<uint64_t *>(s_dyn);       // [np]
    int32_t *s_cnt = reinterpret_cast<int32_t *>(s_key + np);    // [np] each
    int32_t *s_corr = s_cnt + np, *s_dup = s_corr + np;
    __shared__ int s_last;
    for (int p = tid; p < np; p += kDirCountThreads) {
        s_key[p] = A.pkey[p];
        s_cnt[p] = s_corr[p] = s_dup[p] = 0;
    }
    __syncthreads();
    const uint64_t top = s_key[np - 1];
    auto place = [&](uint64_t key) {  // tree edges of a smaller key
        int lo = 0, hi = np - 1;      // s_key[np - 1] >= key
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (s_key[mid] < key) lo = mid + 1;
            else hi = mid;
        }
        return lo;
    };
    auto take = [&](uint64_t key, uint32_t u, uint32_t v) {
        if (key > top) return;
        const int t = place(key);
        int s = t;
        if (s_key[t] == key) {  // among the tree's edges of this length
            const uint32_t uv = (u << 16) | v;
            int lo = t, hi = np;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (before(s_key[mid], A.puv[mid], key, uv)) lo = mid + 1;
                else hi = mid;
            }
            s = lo;
        }
        if (s < np) atomicAdd(s_cnt + s, 1);
        if (s != t) {
            atomicAdd(s_corr + t, 1);
            if (s < np) atomicSub(s_corr + s, 1);
        }
    };
    const uint32_t reps = A.h->direct_strips + A.h->direct_repeats;
    for (uint32_t q = blockIdx.x * kDirCountThreads + tid; q < reps; q += gridDim.x * kDirCountThreads) {
        const uint64_t k = A.repk[q];
        if (k <= top) atomicAdd(s_dup + place(k), int32_t(A.repx[q]));
    }
    // rows a and n-2-a together hold n edges (n - 1 - a and a + 1; the middle
    // row of an even n stands alone): item i is edge i % n of pair i / n
    const uint32_t items = uint32_t(n / 2) * uint32_t(n), span = 2 * kDirCountThreads;
    for (uint32_t i0 = blockIdx.x * span + tid; i0 < items; i0 += gridDim.x * span) {
        uint64_t key[2];
        uint32_t u[2], v[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint32_t i = i0 + q * kDirCountThreads, a = i / uint32_t(n), x = i - a * uint32_t(n);
            const uint32_t la = uint32_t(n) - 1 - a, b = uint32_t(n) - 2 - a;
            u[q] = x < la ? a : b;
            v[q] = x < la ? a + 1 + x : b + 1 + (x - la);
            const bool in = i < items && (x < la || b > a);
            key[q] = in ? __ldcg(A.mat + size_t(u[q]) * A.ldm + v[q]) : ~0ull;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) take(key[q], u[q], v[q]);
    }
    __syncthreads();
    for (int p = tid; p < np; p += kDirCountThreads) {
        if (s_cnt[p]) atomicAdd(A.cnt + p, s_cnt[p]);
        if (s_corr[p]) atomicAdd(A.corr + p, s_corr[p]);
        if (s_dup[p]) atomicAdd(A.dup + p, s_dup[p]);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&A.h->direct_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();

    // the last CTA: running sums over the tree's edges, then the bars
    constexpr int kWarps = kDirCountThreads / 32;
    __shared__ int32_t s_wo[kWarps], s_wa[kWarps];
    const int per = (np + kDirCountThreads - 1) / kDirCountThreads, p0 = tid * per;
    int32_t so = 0, sa = 0;
    for (int p = p0; p < p0 + per && p < np; ++p) {
        const int32_t c = __ldcg(A.cnt + p);
        so += c;
        sa += c + __ldcg(A.corr + p) - __ldcg(A.dup + p);
        s_cnt[p] = so;
        s_corr[p] = sa;
    }
    int32_t io = so, ia = sa;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t yo = __shfl_up_sync(0xffffffffu, io, o), ya = __shfl_up_sync(0xffffffffu, ia, o);
        if (lane >= o) {
            io += yo;
            ia += ya;
        }
    }
    if (lane == 31) {
        s_wo[warp] = io;
        s_wa[warp] = ia;
    }
    __syncthreads();
    int32_t bo = io - so, ba = ia - sa;
    for (int w = 0; w < warp; ++w) {
        bo += s_wo[w];
        ba += s_wa[w];
    }
    for (int p = p0; p < p0 + per && p < np; ++p) {
        s_cnt[p] += bo;
        s_corr[p] += ba;
    }
    __syncthreads();
    uint32_t x = 0;
    for (int p = tid; p < np; p += kDirCountThreads) {
        const uint32_t uv = A.puv[p], low = A.plow[p];
        x ^= low;
        ph0_bar b;
        b.u = int32_t(uv >> 16);
        b.v = int32_t(uv & 0xffffu);
        b.a = uint32_t(s_corr[p]);
        b.low = int32_t(low);
        b.order = int64_t(s_cnt[p] - 1);
        b.death_sq = __longlong_as_double((long long)s_key[p]);
        b.death = __dsqrt_rn(b.death_sq);
        A.bars[p] = b;
    }
    for (int q = tid; q < n; q += kDirCountThreads) x ^= uint32_t(q);
    x = __reduce_xor_sync(0xffffffffu, x);
    __syncthreads();
    if (lane == 0) s_wo[warp] = int32_t(x);
    __syncthreads();
    if (tid == 0) {
        // the vertex that is no pivot row: the bar that never dies
        x = 0;
        for (int w = 0; w < kWarps; ++w) x ^= uint32_t(s_wo[w]);
        if (x >= uint32_t(n)) {  // only after a reported error
            set_status(A.h, PH0_EINTERNAL);
            x = 0;
        }
        Header *h = A.h;
        h->inf_vertex = int32_t(x);
        h->kmin = ~h->direct_nkmin;
        h->n_distinct = n_edges(n) - int64_t(h->direct_dups);
        h->sort_passes = 0;
        h->key_bits = make_plan(h->kmin, h->kmax).bits;
        h->direct = 1;
        if (A.inf) {
            ph0_inf_bar b;
            b.vertex = int32_t(x);
            b._pad = 0;
            b.birth = 0.0;
            b.death = __longlong_as_double(0x7ff0000000000000ll);  // +inf
            *A.inf = b;
        }
    }
}

// ------------------------------------------------------------------ host ---
int sm_count();

namespace {

// Tile edge: blocks of 32, 64 or 128 columns, so that a row has at most
// kDirectChunks of them; the smallest that does, for the most tiles.
int direct_tile(int64_t n) { return n <= 32 * kDirectChunks ? 32 : n <= 64 * kDirectChunks ? 64 : 128; }

size_t direct_dist_smem(int bt, int d) {
    return size_t(2) * bt * d * 8 + size_t(kDirStrip) * (bt + 1) * 8 + size_t(bt) * 8 + size_t(5) * d * 4 +
           size_t((d + 31) / 32) * 4 + size_t(bt) * 2 + size_t(6) * kDirStrip * bt;
}

// The regions of this form within a workspace (from L.key[0] on, up to the
// gradient accumulator; the header and the trace keep their places).
struct DirectRegions {
    int64_t ldm;
    int buckets, bcap, table;
    size_t bcount, cnt, corr, dup, zero_end, bkeys, repk, repx, mat, candk, candv, pkey, puv, plow, total;
    explicit DirectRegions(const Layout &L) {
        const size_t n = size_t(L.n);
        size_t off = L.key[0];
        auto take = [&](size_t b) {
            const size_t o = off;
            off = align_up(off + b, 256);
            return o;
        };
        ldm = (L.n + 3) & ~int64_t(3);
        // buckets of at most 4096 or 8192 keys on average: enough of them for
        // the idle SMs, few counters per strip.  Twice the room (small clouds:
        // what the workspace has): distances
        // repeated hundreds of times each, but seldom within a strip (random
        // integers in one dimension), spread the buckets' counts that far
        const int per = L.m <= int64_t(1) << 19 ? kDirBucketSmall : kDirBucketLarge;
        buckets = int((L.m + per - 1) / per);
        bcap = int((L.m + buckets - 1) / buckets) * (per == kDirBucketSmall ? 7 : 8) / 4 + 64;
        table = 2 * per;
        bcount = take(4 * size_t(buckets));
        cnt = take(4 * n);
        corr = take(4 * n);
        dup = take(4 * n);
        zero_end = off;
        bkeys = take(8 * size_t(buckets) * size_t(bcap));
        // a strip's record takes at least one key away, a bucket's at least
        // one of those left, and there are no more of the first than keys left
        repk = take(8 * size_t(L.m * 3 / 4 + 1));
        repx = take(4 * size_t(L.m * 3 / 4 + 1));
        mat = take(8 * n * size_t(ldm));
        candk = take(8 * n * kDirectChunks);
        candv = take(2 * n * kDirectChunks);
        pkey = take(8 * n);
        puv = take(4 * n);
        plow = take(4 * n);
        total = off;
    }
};

static_assert((kDirectMaxN * (kDirectMaxN - 1) / 2 + kDirBucketLarge - 1) / kDirBucketLarge <= kDirMaxBuckets,
              "a counter per bucket in shared memory");

}  // namespace

// Whether the whole path of n points in dimension d takes this form: up to
// kDirectMaxN points, while the tile's coordinates fit shared memory (d up
// to about 300 to 1024 points, 150 to 2048, 60 above) and the regions fit
// the workspace.
bool direct_applies(const Layout &L, int32_t d) {
    if (L.n < 2 || L.n > kDirectMaxN) return false;
    return direct_dist_smem(direct_tile(L.n), d) <= kDirDistSmem && DirectRegions(L).total <= L.grad;
}

// after_dist, after_tree: events recorded between the stages, or null.
cudaError_t launch_direct(void *ws, const Layout &L, const float *pts, int64_t n, int32_t d, int64_t ld,
                          ph0_bar *bars, ph0_inf_bar *inf, cudaStream_t s, cudaEvent_t after_dist,
                          cudaEvent_t after_tree) {
    const DirectRegions G(L);
    DirectArgs A;
    A.pts = pts;
    A.ld = ld;
    A.n = int(n);
    A.d = d;
    A.bt = direct_tile(n);
    A.nch = int((n + A.bt - 1) / A.bt);
    A.ldm = int(G.ldm);
    A.buckets = G.buckets;
    A.bcap = G.bcap;
    A.table = G.table;
    const double mean = double(kDirStrip * A.bt) / double(A.buckets);
    A.crowd = uint32_t(mean + kDirCrowd * sqrt(mean)) + 1;
    A.bkeys = at<uint64_t>(ws, G.bkeys);
    A.bcount = at<uint32_t>(ws, G.bcount);
    A.repk = at<uint64_t>(ws, G.repk);
    A.repx = at<uint32_t>(ws, G.repx);
    A.mat = at<uint64_t>(ws, G.mat);
    A.candk = at<uint64_t>(ws, G.candk);
    A.candv = at<uint16_t>(ws, G.candv);
    A.pkey = at<uint64_t>(ws, G.pkey);
    A.puv = at<uint32_t>(ws, G.puv);
    A.plow = at<uint32_t>(ws, G.plow);
    A.cnt = at<int32_t>(ws, G.cnt);
    A.corr = at<int32_t>(ws, G.corr);
    A.dup = at<int32_t>(ws, G.dup);
    A.h = at<Header>(ws, L.hdr);
    A.trace = at<uint64_t>(ws, L.trace);
    A.bars = bars;
    A.inf = inf;
    cudaError_t e = cudaMemsetAsync(at<char>(ws, L.hdr), 0, G.zero_end - L.hdr, s);
    if (e != cudaSuccess) return e;

    const unsigned tiles = unsigned(A.nch) * unsigned(A.nch + 1) / 2;
    const size_t dsm = direct_dist_smem(A.bt, d);
    auto go = [&](auto kernel) {
        cudaError_t r = smem_limit<kDirDistSmem>(kernel);
        if (r != cudaSuccess) return r;
        kernel<<<tiles, kDirThreads, dsm, s>>>(A);
        return cudaGetLastError();
    };
    auto pick = [&]() {
#define PH0_DIRECT_CASE(DD)                                     \
    case DD:                                                    \
        if (A.bt == 32) return go(k_direct_dist<DD, 32>);       \
        if (A.bt == 64) return go(k_direct_dist<DD, 64>);       \
        return go(k_direct_dist<DD, 128>);
        switch (d) {
            PH0_DIRECT_CASE(2)
            PH0_DIRECT_CASE(3)
            PH0_DIRECT_CASE(8)
            PH0_DIRECT_CASE(16)
            PH0_DIRECT_CASE(32)
            default:
                if (A.bt == 32) return go(k_direct_dist<0, 32>);
                if (A.bt == 64) return go(k_direct_dist<0, 64>);
                return go(k_direct_dist<0, 128>);
        }
#undef PH0_DIRECT_CASE
    };
    e = pick();
    if (e == cudaSuccess && after_dist) e = cudaEventRecord(after_dist, s);
    if (e != cudaSuccess) return e;

    // the tree on one cluster of 8 CTAs (16 above 1024 points: half the rows
    // per CTA), the buckets on up to seven others
    const int cl = n > 1024 ? 16 : 8;
    const size_t tsm = size_t(12) * size_t(A.table), msm = DirMst(int(n), cl).total;
    int more = (A.buckets + cl - 1) / cl;
    if (more > 112 / cl) more = 112 / cl;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(cl * (1 + more)));
    cfg.blockDim = dim3(n <= 512 ? 512 : kDirMstThreads);
    cfg.dynamicSmemBytes = tsm > msm ? tsm : msm;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(cl);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto tree = [&](auto kernel) {
        cudaError_t r = smem_limit<kDirMstSmem>(kernel);
        if (r == cudaSuccess && cl > 8) r = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (r == cudaSuccess) r = cudaLaunchKernelEx(&cfg, kernel, (const DirectArgs)A);
        return r;
    };
    e = A.bt == 32 ? tree(k_direct_mst<32>) : A.bt == 64 ? tree(k_direct_mst<64>) : tree(k_direct_mst<128>);
    if (e == cudaSuccess && after_tree) e = cudaEventRecord(after_tree, s);
    if (e != cudaSuccess) return e;

    // a kernel has 48 KB less its static shared memory without it (2,451
    // points need more); asked for with a margin, but not by the smallest
    // calls, which the host's share bounds
    constexpr size_t kPerPoint = 20;
    const size_t csm = kPerPoint * size_t(n);
    if (csm > 40 * 1024) {
        e = smem_limit<kPerPoint * kDirectMaxN>(k_direct_count);
        if (e != cudaSuccess) return e;
    }
    // two CTAs per SM, or fewer with at least 2048 edges each
    int grid = int((L.m + 2047) / 2048);
    if (grid > 2 * sm_count()) grid = 2 * sm_count();
    k_direct_count<<<unsigned(grid), kDirCountThreads, csm, s>>>(A);
    return cudaGetLastError();
}

}  // namespace ph0
