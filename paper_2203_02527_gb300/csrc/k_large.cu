// k_large.cu -- the whole barcode path without a sort for clouds above the
// size of k_direct.cu (Rawson, Sec. 2; Sec. 4 steps 1-5).
//
// As there, the reduction keeps n-1 of the n(n-1)/2 columns, the minimum
// spanning tree in the order (distance, u, v), and of the other edges a bar
// only reads counts.  Sorting every edge to get them moved 77 to 130 bytes per
// edge in four or five passes bound by integer work; here every edge's key is
// written once, read a few times as a stream, and moved twice:
//   k_dist              step 1: the key of edge e at e; a histogram of a hash
//   k_large_sample,     places of the 512 hash partitions; from a sample of
//   k_large_prep        the keys a threshold that about 64 n edges lie below
//   k_large_move<0>     the keys by partition; the edges below the threshold
//                       as a list; a tile of few distances keeps one key of
//                       each and records how many more it stands for
//   k_large_tree        the tree by Boruvka's rounds (cooperative): equal
//                       points first where there are many, then on the list
//                       while it joins components, then on all keys
//   k_large_runs, merge the tree's edges in order
//   k_reduce            their columns' pivot rows (k_reduce.cu)
//   k_large_count       every edge up to the last killing edge counted at its
//                       place among the killing edges
//   k_large_sub,        the partitions' keys by bucket of about ten thousand
//   k_large_move<1>
//   k_large_repeats     step 3: repeated distances, a bucket at a time in a
//                       bit table in shared memory, buckets beyond their room
//                       in tables of their distinct keys
//   k_large_emit        running sums, the bars
// Every step is exact for any input: partitions and buckets are counted before
// they are filled, a list that overflows is not used, and ties are ordered by
// (u, v) throughout, so the results equal the sorted path's bit for bit.
//
// Measured (device time, 1.25G edges of 50,021 points in the plane; the short
// sort's path 67.4 ms): k_dist 5.8 ms, k_large_move<0> 6.6, the tree and its
// pivots 1.3, the count 1.9, k_large_sub 1.4, k_large_move<1> 5.8,
// k_large_repeats 5.2: 28.1 ms.  32,768 points of four circles in 16
// dimensions (537M edges): 26.4 ms (packed sort 34.4), of which the distances,
// bound by the binary64 adder, 15.6.  The count, k_large_sub and the tree's
// passes run near the copy bandwidth; the moves are bound by shared-memory
// wavefronts (60 to 66% of the peak) and their barriers, with spills to local
// memory on the same pipe: at the 32 registers that 2,048 threads per SM leave,
// k_large_move<0> has a frame of 152 bytes and k_large_move<1> of 64, and a
// warp issues 38 and 27 spill instructions for its 256 keys of a tile;
// k_large_tree (64 registers) has a frame of 80 bytes.
#include "ph0_common.cuh"

namespace ph0 {

int sm_count();

namespace {

#ifndef PH0_LG_TILE
#define PH0_LG_TILE 8192
#endif
constexpr int kLgTile = PH0_LG_TILE;           // keys a CTA moves at a time
constexpr int kLgThreads = kLgTile / 8;
constexpr int kLgPer = kLgTile / kLgThreads;
constexpr int kLgParts = 512;
constexpr int kLgMaxSub = 512;                 // buckets per partition
constexpr int kLgBucket = 10240;               // keys per bucket on average, at most
constexpr int kLgPass = 14336;                 // keys of a bucket looked at at once (14 bits)
constexpr int kLgWords = 20480;                // of a bucket's bit table, slots of its hash table
constexpr int kLgSuspects = 512, kLgSusSlots = 2048, kLgSusKeys = 1024;
#ifndef PH0_LG_PROBES
#define PH0_LG_PROBES 64
#endif
constexpr int kLgSlots = 6784, kLgProbes = PH0_LG_PROBES; // larger buckets: keys with their occurrences
static_assert(3 * kLgSlots <= kLgWords, "in the same room");
constexpr int kLgRepThreads = 512;
constexpr int kLgListPerPoint = 64;            // edges per point the list aims at
constexpr int kLgListRoom = 512;               // ... and has room for
constexpr int kLgSample = 1 << 17;
constexpr int kLgTreeThreads = 512;
constexpr int kLgRun = 2048;                   // tree edges sorted by a CTA
constexpr int kLgHot = 8192;                   // longest tree edges whose counts stay in shared memory
constexpr int kLgCountThreads = 512;
constexpr int kLgRuns = 512;                   // runs of equal tree edges remembered by a CTA
constexpr int kLgLutBits = 11, kLgLut = 1 << kLgLutBits;
constexpr int kLgSubCtas = 4;                  // CTAs per partition
// keys of a tile in one partition that only repeated distances explain: the
// mean and seven standard deviations
constexpr uint32_t kLgCrowd = kLgTile == 8192 ? 44 : 28;
static_assert(kLgTile == 8192 || kLgTile == 4096, "kLgCrowd");
constexpr uint64_t kNone = ~uint64_t(0);       // above every key

struct LgRepeat {
    uint64_t key;
    uint32_t extra, pad;
};

struct LgArgs {
    int64_t m;
    int n, nsub;
    const float *pts;          // [n][ld] coordinates, d of each row (the tree alone)
    int64_t ld;
    int d;
    const uint64_t *mat;       // [m] key of edge e
    uint64_t *part, *bkt;      // [m] keys by partition, by bucket
    LgRepeat *rep;             // [m / 2] records of crowded tiles (in bkt's place, read before it is filled)
    uint64_t *lkey;            // [lcap] the edges below the threshold: key,
    uint32_t *luv;             //     (u << 16) | v
    uint32_t lcap;
    uint32_t *cand;            // [ccap] edges that bettered a component's best
    uint32_t ccap;
    uint32_t *comp, *parent;   // [n]
    unsigned long long *best;  // [n] per component: smallest key leaving it,
    uint32_t *buv;             //     its edge
    uint64_t *tkey, *skey;     // [n] the tree's edges as found, in order
    uint32_t *tuv, *suv;
    const unsigned long long *kill_key;  // [n] k_reduce's pivots: position,
    const uint32_t *kill_val;            //     row
    uint32_t *low;             // [n] pivot row by position
    uint32_t *cnt, *late, *dup;  // [n] counts per place among the tree's edges
    uint32_t *poff, *pcur;     // [512 + 1], [512] places of the partitions, their ends
    uint32_t *bcnt, *bcur;     // [512][nsub] keys per bucket, filled
    uint32_t *boff;            // [512][nsub]
    bool prefix;               // the early path: step 3 on the keys up to the last killing edge only,
    uint64_t *keep;            //     [m] which the count puts here
    Header *h;
    ph0_bar *bars;
    ph0_inf_bar *inf;
    uint32_t spin_limit;
};

// All distances zero, the points all equal: the tree is vertex 0's edges and
// every count is known, so the kernels that read the keys leave them alone
// (20,000 points: 1.07 ms a call; 3.8 with the keys moved and counted, 2.0
// by the sorted form, whose passes see that no digit varies).
__device__ __forceinline__ bool lg_all_equal(const LgArgs &A) { return __ldcg(&A.h->kmax) == 0; }

__device__ __forceinline__ uint32_t hash_sub(uint32_t x, int nsub) { return __umulhi(x << 9, uint32_t(nsub)); }

// Exclusive prefix sum over the CTA (T threads); s_w: T / 32 + 1 words.
template <int T>
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t *s_w, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < T / 32 ? s_w[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < T / 32) s_w[lane] = wi - w;
        if (lane == T / 32 - 1) s_w[T / 32] = wi;
    }
    __syncthreads();
    const uint32_t r = inc - x + s_w[warp];
    total = s_w[T / 32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ bool lg_before(uint64_t ka, uint32_t ua, uint64_t kb, uint32_t ub) {
    return ka < kb || (ka == kb && ua < ub);
}

// Tree edges of a smaller key (the last tree edge's is at least as large).
__device__ __forceinline__ int lg_place(const uint64_t *skey, int lo, int hi, uint64_t key) {
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (skey[mid] < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// ------------------------------------------------------------------ prep ---
// One CTA: the partitions' places from the distance kernel's histogram; the
// list's threshold from a sample of the keys (evenly spread, jittered):
// a bin of key >> 48 (sixteen to the octave) and within it one of the next 15
// bits, so that about kLgListPerPoint n edges lie below; and the bin below
// which at most a sixteenth of those do (for the rounds on the list).  More
// zeros than an eighth of that (copies of points): the list leaves them out,
// and the tree joins the points that are equal by their coordinates.
__host__ __device__ __forceinline__ int lg_samples(int n) {
    // four keys per point, so that a few hundred lie below the threshold
    const int S = 4 * n;
    return S < kLgSample / 8 ? kLgSample / 8 : S > kLgSample ? kLgSample : S;
}
__global__ void __launch_bounds__(256) k_large_sample(const LgArgs A) {
    const uint32_t S = uint32_t(lg_samples(A.n)), step = uint32_t(A.m / S);  // m > 2^22
    for (uint32_t i = blockIdx.x * 256 + threadIdx.x; i < S; i += gridDim.x * 256)
        A.lkey[i] = A.mat[size_t(i) * step + __umulhi(i * 2654435761u, step)];
}
// The partitions' places from their histogram (1024 threads; s_w: 33 words).
__device__ __forceinline__ void lg_places(const LgArgs &A, uint32_t *s_w) {
    const int tid = threadIdx.x;
    const uint32_t c = tid < kLgParts ? A.h->phist[0][tid] : 0u;
    uint32_t total;
    const uint32_t off = block_scan<1024>(c, s_w, total);
    if (tid < kLgParts) {
        A.poff[tid] = off;
        A.pcur[tid] = off;
    }
    if (tid == 0) A.poff[kLgParts] = total;
}
__global__ void __launch_bounds__(1024) k_large_places(const LgArgs A) {
    __shared__ uint32_t s_w[33];
    lg_places(A, s_w);
}
__global__ void __launch_bounds__(1024) k_large_prep(const LgArgs A) {
    extern __shared__ uint32_t s_bin[];  // [32768]
    __shared__ uint32_t s_w[33];
    __shared__ uint32_t s_at, s_below, s_zeros;
    const int tid = threadIdx.x;
    if (tid == 0) s_zeros = 0;
    lg_places(A, s_w);
    const int S = lg_samples(A.n);
    const double want = double(kLgListPerPoint) * double(A.n) * double(S) / double(A.m);
    uint64_t limit = 0, lo = 0;
    uint32_t target = uint32_t(want);
    uint64_t prefix = 0;
    for (int level = 0; level < 2; ++level) {
        for (int i = tid; i < 32768; i += 1024) s_bin[i] = 0;
        __syncthreads();
#pragma unroll 16
        for (uint32_t i = tid; i < uint32_t(S); i += 1024) {
            const uint64_t k = A.lkey[i];
            if (level == 0) atomicAdd(s_bin + ((k >> 48) & 32767), 1u);
            else if ((k >> 48) == prefix) atomicAdd(s_bin + ((k >> 33) & 32767), 1u);
        }
        __syncthreads();
        if (prefix == 0 && s_bin[0] > uint32_t(want) / 8) {  // (few clouds; the same for all threads)
            if (level == 0) {
                for (uint32_t i = tid; i < uint32_t(S); i += 1024)
                    if (A.lkey[i] == 0) atomicAdd(&s_zeros, 1u);
            }
            __syncthreads();
            lo = s_zeros > uint32_t(want) / 8;
            if (tid == 0 && lo) s_bin[0] -= s_zeros;
            __syncthreads();
        }
        // the bin in which the running count passes the target
        uint32_t sum = 0;
        for (int i = 0; i < 32; ++i) sum += s_bin[tid * 32 + ((i + tid) & 31)];
        uint32_t total;
        uint32_t run = block_scan<1024>(sum, s_w, total);
        if (tid == 0) s_at = 32768;
        __syncthreads();
        if (level == 0 && run <= target / 16 && run + sum > target / 16) {
            uint32_t sixteenth = run;
            for (int i = 0; i < 32; ++i) {
                sixteenth += s_bin[tid * 32 + i];
                if (sixteenth > target / 16) {
                    A.h->lg_first = uint64_t(tid * 32 + i) << 48;
                    break;
                }
            }
        }
        if (run <= target && run + sum > target) {
            for (int i = 0; i < 32; ++i) {
                const uint32_t c = s_bin[tid * 32 + i];
                if (run + c > target) {
                    s_at = uint32_t(tid * 32 + i);
                    s_below = run;
                    break;
                }
                run += c;
            }
        }
        __syncthreads();
        const uint32_t at = s_at;
        if (level == 0) {
            if (at == 32768) {
                limit = kNone;  // fewer edges than wanted in all
                break;
            }
            prefix = at;
            target -= s_below;
            limit = uint64_t(at) << 48;
        } else if (at < 32768) {
            limit |= uint64_t(at) << 33;
        } else {
            limit = (prefix + 1) << 48;
        }
        __syncthreads();
    }
    if (tid == 0) {
        A.h->lg_limit = limit > lo ? limit : lo;
        A.h->lg_lo = uint32_t(lo);
    }
}

// A thread's place for the `mine` entries it appends, by one addition per
// warp to the counter.  For the list the counter is the CTA's, in shared
// memory; after a barrier one thread takes the CTA's room in the list with one
// addition to the global counter (an addition per warp there: all the GPU's
// warps on one word, about one a nanosecond, 0.93 ms to list 1.3M of 200M keys
// instead of 0.52, and 0.7 of the 7.7 ms of k_large_move<0> on 1.25G).
__device__ __forceinline__ uint32_t lg_rank(uint32_t mine, uint32_t *s_n) {
    const int lane = threadIdx.x & 31;
    if (!__any_sync(0xffffffffu, mine != 0)) return 0;
    uint32_t at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    uint32_t base = 0;
    if (lane == 31) base = atomicAdd(s_n, at);
    return __shfl_sync(0xffffffffu, base, 31) + at - mine;
}
__device__ __forceinline__ void lg_room(uint32_t *counter, uint32_t *s_n, uint32_t *s_base) {
    if (threadIdx.x == 0) {
        if (*s_n) *s_base = atomicAdd(counter, *s_n);
        *s_n = 0;
    }
}
// The keys of a thread from lo on and below the limit, with their edges, to
// the list from place `at` on.  (kNone, past the end, is below no limit.)
template <int N>
__device__ __forceinline__ void lg_list_put(const LgArgs &A, const uint64_t (&key)[N], int64_t e0, int64_t step,
                                            uint64_t lo, uint64_t limit, uint32_t at) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
        if (key[q] >= limit || key[q] < lo) continue;
        if (at < A.lcap) {
            uint32_t u, v;
            edge_uv(e0 + q * step, A.n, u, v);
            A.lkey[at] = key[q];
            A.luv[at] = (u << 16) | v;
        }
        ++at;
    }
}

// The list alone (the early path, whose keys are not all moved).  ZEROS: they
// are listed too.
template <bool ZEROS>
__device__ __forceinline__ void lg_list_all(const LgArgs &A, uint32_t *s_n, uint32_t *s_base) {
    constexpr int kU = 8;
    const uint64_t lo = ZEROS ? 0 : 1, limit = A.h->lg_limit;
    const int64_t stride = int64_t(gridDim.x) * 1024;
    for (int64_t b = int64_t(blockIdx.x) * 1024; b < A.m; b += kU * stride) {  // the same for a whole CTA
        const int64_t e0 = b + threadIdx.x;
        uint64_t key[kU];
        uint32_t mine = 0;
#pragma unroll
        for (int q = 0; q < kU; ++q) key[q] = e0 + q * stride < A.m ? A.mat[e0 + q * stride] : kNone;
#pragma unroll
        for (int q = 0; q < kU; ++q) mine += key[q] < limit && key[q] >= lo;
        const uint32_t at = lg_rank(mine, s_n);
        __syncthreads();
        lg_room(&A.h->lg_list, s_n, s_base);
        __syncthreads();
        if (mine) lg_list_put<kU>(A, key, e0, stride, lo, limit, *s_base + at);
    }
}
__global__ void __launch_bounds__(1024, 2) k_large_list(const LgArgs A) {
    __shared__ uint32_t s_n, s_base;
    if (lg_all_equal(A)) return;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    if (A.h->lg_lo == 0) lg_list_all<true>(A, &s_n, &s_base);
    else lg_list_all<false>(A, &s_n, &s_base);
}

// ----------------------------------------------------- moving keys by hash ---
// Tiles of eight keys per thread: a key's place among the tile's keys of
// its partition by a shared-memory counter, the tile reordered there and
// written out in runs.  The order within a partition is free.  LEVEL 0: all
// keys to the partitions (with the list, and crowded tiles deduplicated); 1: a
// partition's keys to its buckets.
template <int LEVEL>
__global__ void __launch_bounds__(kLgThreads, 2048 / kLgThreads) k_large_move(const LgArgs A) {
    constexpr int kDig = LEVEL == 0 ? kLgParts : kLgMaxSub;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    uint64_t *s_key = reinterpret_cast<uint64_t *>(s_dyn);          // [kLgTile]
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_key + kLgTile);  // [kDig]
    uint32_t *s_off = s_cnt + kDig, *s_to = s_off + kDig, *s_base = s_to + kDig;  // s_base: LEVEL 1
    __shared__ uint32_t s_w[kLgThreads / 32 + 1], s_nrep, s_rbase, s_extra, s_nlist, s_list;
    const int tid = threadIdx.x;
    if (LEVEL == 0 && lg_all_equal(A)) return;  // the partitions stay empty
    int64_t begin = 0, end = A.prefix ? int64_t(A.h->lg_keep) : A.m, first = blockIdx.x, step = gridDim.x;
    const uint64_t *src = A.prefix ? A.keep : A.mat;
    uint64_t *dst = A.part;
    uint32_t *cursor = A.pcur;
    int ndig = kLgParts;
    const int p = blockIdx.x / kLgSubCtas;
    if constexpr (LEVEL == 1) {
        begin = A.poff[p];
        end = A.pcur[p];
        first = blockIdx.x % kLgSubCtas;
        step = kLgSubCtas;
        src = A.part;
        dst = A.bkt;
        ndig = A.nsub;
        cursor = A.bcur + size_t(p) * ndig;
        // the buckets' places
        uint32_t total;
        const uint32_t c = tid < ndig ? A.bcnt[size_t(p) * ndig + tid] : 0u;
        const uint32_t run = uint32_t(begin) + block_scan<kLgThreads>(c, s_w, total);
        if (tid < kDig) s_base[tid] = run;
        if (tid < ndig && first == 0) A.boff[size_t(p) * ndig + tid] = run;
    }
    const bool listing = LEVEL == 0 && !A.prefix;
    const uint64_t lo = listing ? A.h->lg_lo : 0, limit = listing ? A.h->lg_limit : 0;
    if (tid == 0) s_nlist = 0;
    auto digit = [&](uint64_t k) { return LEVEL == 0 ? hash_part(part_hash(k)) : hash_sub(part_hash(k), ndig); };
    for (int64_t t0 = begin + first * kLgTile; t0 < end; t0 += step * kLgTile) {
        for (int i = tid; i < kDig; i += kLgThreads) s_cnt[i] = 0;
        __syncthreads();
        uint64_t key[kLgPer];
        uint32_t place[kLgPer];  // (digit << 16) | place among the tile's keys of the digit
#pragma unroll
        for (int q = 0; q < kLgPer; ++q) {
            const int64_t i = t0 + q * kLgThreads + tid;
            key[q] = i < end ? __ldcs(src + i) : kNone;
        }
        bool crowded = false;
#pragma unroll
        for (int q = 0; q < kLgPer; ++q) {
            place[q] = 0xffffffffu;
            if (t0 + q * kLgThreads + tid >= end) continue;
            const uint32_t dg = digit(key[q]), at = atomicAdd(s_cnt + dg, 1u);
            place[q] = (dg << 16) | at;
            crowded |= at >= kLgCrowd;
        }
        uint32_t mine = 0, at = 0;  // for the list
        if constexpr (LEVEL == 0) {
#pragma unroll
            for (int q = 0; q < kLgPer; ++q) mine += key[q] - lo < limit - lo;
            at = lg_rank(mine, &s_nlist);
        }
        const bool dedupe = __syncthreads_or(crowded);
        if (LEVEL == 0) lg_room(&A.h->lg_list, &s_nlist, &s_list);
        if (LEVEL == 0 && dedupe) {
            // one key of each distance stays; a table of half the tile's keys,
            // at most eight probes (a key that finds no slot stays as it is)
            constexpr int kSlots = kLgTile / 2;
            unsigned long long *tab = reinterpret_cast<unsigned long long *>(s_key);
            uint32_t *occ = reinterpret_cast<uint32_t *>(tab + kSlots);
            for (int i = tid; i < kSlots; i += kLgThreads) {
                tab[i] = 0;
                occ[i] = 0;
            }
            for (int i = tid; i < kDig; i += kLgThreads) s_cnt[i] = 0;
            if (tid == 0) s_nrep = s_extra = 0;
            __syncthreads();
            uint32_t stays = 0;
            uint16_t slot_of[kLgPer];
#pragma unroll
            for (int q = 0; q < kLgPer; ++q) {
                slot_of[q] = 0xffffu;
                if (place[q] == 0xffffffffu) continue;
                const unsigned long long tag = key[q] + 1;
                uint32_t slot = uint32_t(key_hash(key[q])) & (kSlots - 1);
                stays |= 1u << q;
                for (int pr = 0; pr < 8; ++pr) {
                    unsigned long long old = *(volatile unsigned long long *)(tab + slot);
                    if (old == 0) old = atomicCAS(tab + slot, 0ull, tag);
                    if (old == 0 || old == tag) {
                        atomicAdd(occ + slot, 1u);
                        if (old == 0) slot_of[q] = uint16_t(slot);
                        else stays &= ~(1u << q);
                        break;
                    }
                    slot = (slot + 1) & (kSlots - 1);
                }
            }
            __syncthreads();
            uint32_t to[kLgPer], extra[kLgPer];
#pragma unroll
            for (int q = 0; q < kLgPer; ++q) {
                extra[q] = 0;
                if (!((stays >> q) & 1u)) {
                    place[q] = 0xffffffffu;
                    continue;
                }
                const uint32_t dg = digit(key[q]);
                place[q] = (dg << 16) | atomicAdd(s_cnt + dg, 1u);
                if (slot_of[q] != 0xffffu) extra[q] = occ[slot_of[q]] - 1;
                if (extra[q]) {
                    to[q] = atomicAdd(&s_nrep, 1u);
                    atomicAdd(&s_extra, extra[q]);
                }
            }
            __syncthreads();
            if (tid == 0 && s_nrep) {
                s_rbase = atomicAdd(&A.h->lg_reps, s_nrep);
                atomicAdd(&A.h->direct_dups, s_extra);
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kLgPer; ++q)
                if (extra[q]) A.rep[s_rbase + to[q]] = LgRepeat{key[q], extra[q], 0u};
        }
        // room for each digit's keys, their place within the tile
        uint32_t total;
        {
            static_assert(kDig <= kLgThreads, "a thread per digit");
            const uint32_t c = tid < kDig ? s_cnt[tid] : 0u;
            uint32_t to = c ? atomicAdd(cursor + tid, c) : 0u;
            if (LEVEL == 1 && tid < kDig) to += s_base[tid];
            const uint32_t run = block_scan<kLgThreads>(c, s_w, total);
            if (tid < kDig) {
                s_off[tid] = run;
                s_to[tid] = to - run;
            }
        }
        __syncthreads();
        if (LEVEL == 0 && mine) lg_list_put<kLgPer>(A, key, t0 + tid, kLgThreads, lo, limit, s_list + at);
#pragma unroll
        for (int q = 0; q < kLgPer; ++q) {
            if (place[q] == 0xffffffffu) continue;
            s_key[s_off[place[q] >> 16] + (place[q] & 0xffffu)] = key[q];
        }
        __syncthreads();
        for (uint32_t i = tid; i < total; i += kLgThreads) {
            const uint64_t k = s_key[i];
            dst[s_to[digit(k)] + i] = k;
        }
        __syncthreads();
    }
}

constexpr size_t move_smem(int level) {
    return size_t(kLgTile) * 8 + size_t(level == 0 ? kLgParts : kLgMaxSub) * 16;
}

// Keys per bucket of each partition.
__global__ void __launch_bounds__(kLgThreads) k_large_sub(const LgArgs A) {
    __shared__ uint32_t s_cnt[kLgMaxSub];
    const int p = blockIdx.x / kLgSubCtas, tid = threadIdx.x;
    for (int i = tid; i < A.nsub; i += kLgThreads) s_cnt[i] = 0;
    __syncthreads();
    const int64_t begin = A.poff[p], end = A.pcur[p];
    constexpr int kU = 8;
    for (int64_t i0 = begin + int64_t(blockIdx.x % kLgSubCtas) * kU * kLgThreads + tid; i0 < end;
         i0 += int64_t(kLgSubCtas) * kU * kLgThreads) {
        uint64_t key[kU];
#pragma unroll
        for (int q = 0; q < kU; ++q) key[q] = i0 + q * kLgThreads < end ? A.part[i0 + q * kLgThreads] : kNone;
#pragma unroll
        for (int q = 0; q < kU; ++q)
            if (i0 + q * kLgThreads < end) atomicAdd(s_cnt + hash_sub(part_hash(key[q]), A.nsub), 1u);
    }
    __syncthreads();
    for (int i = tid; i < A.nsub; i += kLgThreads)
        if (s_cnt[i]) atomicAdd(A.bcnt + size_t(p) * A.nsub + i, s_cnt[i]);
}

// The records of crowded tiles, at their places among the tree's edges.
__device__ __forceinline__ void lg_reps(const LgArgs &A, uint32_t first, uint32_t step) {
    const int np = A.n - 1;
    const uint64_t top = A.skey[np - 1];
    const uint32_t reps = A.h->lg_reps;
    for (uint32_t q = first; q < reps; q += step) {
        const LgRepeat r = A.rep[q];
        if (r.key <= top) atomicAdd(A.dup + lg_place(A.skey, 0, np - 1, r.key), r.extra);
    }
}

// The slot of a tag that is there already, -2 when it was put there, -1 when
// kLgProbes slots from the first were others'.  (Not inlined: the loop that
// looks at a table of few distances holds eight copies of what is.)
__device__ __noinline__ int lg_insert(unsigned long long *tab, uint32_t slot, unsigned long long tag) {
    for (int pr = 0; pr < kLgProbes; ++pr) {
        unsigned long long old = *(volatile unsigned long long *)(tab + slot);
        if (old == 0) old = atomicCAS(tab + slot, 0ull, tag);
        if (old == 0) return -2;
        if (old == tag) return int(slot);
        slot = slot + 1 == kLgSlots ? 0 : slot + 1;
    }
    return -1;
}

// Repeated distances, a bucket at a time.  Few repeats: a bit table in shared
// memory, one bit per key (10,240 keys set 1.6% of 655,360 bits); a key that
// finds its bit set is a suspect, and a second look over the bucket's keys
// picks out those that share a suspect's bit (about 160), which a small hash
// table compares.  Where more than kLgSuspects are, a hash table of all keys
// (32-bit slots: the key's place in the bucket and 18 bits of its hash, so an
// occupied slot needs the key itself only when those agree); a bucket of more
// than kLgPass keys by one of the distinct keys and their occurrences, in as
// many parts as those need.  (The hash tables alone took 8.3 ps per key: a warp waits
// for its lane with the most probes.)
__global__ void __launch_bounds__(kLgRepThreads, 2) k_large_repeats(const LgArgs A) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    uint32_t *s_tab = reinterpret_cast<uint32_t *>(s_dyn);  // [kLgWords] bits, slots, or keys + 1 and occurrences
    __shared__ uint64_t s_key[kLgSusKeys];
    __shared__ uint32_t s_sus[kLgSusSlots], s_ns, s_nk;
    const int tid = threadIdx.x, np = A.n - 1;
    const uint64_t top = A.skey[np - 1];
    const bool two = A.nsub > 1;
    const uint64_t *all = two ? A.bkt : A.part;
    const int64_t buckets = int64_t(kLgParts) * A.nsub;
    uint32_t dups = 0;
    bool crowded = false;  // the last bucket was: likely the next one is too
    constexpr int kU = 8;
    // (an occurrence beyond the first; those of one key after the other are
    // placed together: on the early path, where every key is placed, 78 points
    // in 256 copies each took 0.43 ms for all buckets instead of 0.21)
    uint64_t again_key = kNone;
    uint32_t again_n = 0;
    auto settle = [&]() {
        if (again_n) atomicAdd(A.dup + lg_place(A.skey, 0, np - 1, again_key), again_n);
        again_n = 0;
    };
    auto again = [&](uint64_t key) {
        ++dups;
        if (key > top) return;
        if (key != again_key) settle();
        again_key = key;
        ++again_n;
    };
    auto clear = [&]() {
        for (int i = tid; i < kLgWords / 4; i += kLgRepThreads) reinterpret_cast<uint4 *>(s_tab)[i] = make_uint4(0, 0, 0, 0);
    };
    if (A.prefix) lg_reps(A, blockIdx.x * kLgRepThreads + tid, gridDim.x * kLgRepThreads);
    // the repeats among the first nk of s_key (ends with a barrier)
    auto compare = [&](uint32_t nk) {
        for (int i = tid; i < kLgSusSlots; i += kLgRepThreads) s_sus[i] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < nk; i += kLgRepThreads) {
            const uint64_t key = s_key[i];
            uint32_t slot = uint32_t(key_hash(key)) & (kLgSusSlots - 1);
            for (;;) {  // at most kLgSusKeys of the slots fill
                const uint32_t old = atomicCAS(s_sus + slot, 0u, i + 1);
                if (old == 0) break;
                if (s_key[old - 1] == key) {
                    again(key);
                    break;
                }
                slot = (slot + 1) & (kLgSusSlots - 1);
            }
        }
        __syncthreads();
    };
    auto bit_of = [](uint64_t x) { return __umulhi(uint32_t(x >> 24), uint32_t(kLgWords * 32)); };
    for (int64_t b = blockIdx.x; b < buckets; b += gridDim.x) {
        const uint32_t begin = two ? A.boff[b] : A.poff[b];
        const uint32_t size = two ? A.bcur[b] : A.pcur[b] - begin;
        const uint64_t *keys = all + begin;
        if (size < 2) continue;
        if (size <= uint32_t(kLgSusKeys)) {  // few keys: compared at once
            for (uint32_t i = tid; i < size; i += kLgRepThreads) s_key[i] = keys[i];
            compare(size);
            continue;
        }
        if (size <= uint32_t(kLgPass) && !crowded) {
            clear();
            for (int i = tid; i < kLgSusSlots; i += kLgRepThreads) s_sus[i] = 0;
            if (tid == 0) s_ns = s_nk = 0;
            __syncthreads();
            for (uint32_t i0 = tid; i0 < size; i0 += kU * kLgRepThreads) {
                uint64_t key[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) key[q] = i0 + q * kLgRepThreads < size ? keys[i0 + q * kLgRepThreads] : kNone;
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    if (key[q] == kNone) continue;
                    const uint32_t bit = bit_of(key_hash(key[q])), mask = 1u << (bit & 31);
                    if (!(atomicOr(s_tab + (bit >> 5), mask) & mask)) continue;
                    if (atomicAdd(&s_ns, 1u) >= kLgSuspects) continue;
                    uint32_t slot = bit * 2654435761u >> 21;
                    for (;;) {  // at most kLgSuspects of the slots fill
                        const uint32_t old = atomicCAS(s_sus + slot, 0u, bit + 1);
                        if (old == 0 || old == bit + 1) break;
                        slot = (slot + 1) & (kLgSusSlots - 1);
                    }
                }
            }
            __syncthreads();
            const uint32_t ns = s_ns;
            __syncthreads();  // before s_ns is reset
            if (ns == 0) continue;
            crowded = ns > kLgSuspects;
            if (!crowded) {
                for (uint32_t i0 = tid; i0 < size; i0 += kU * kLgRepThreads) {
                    uint64_t key[kU];
#pragma unroll
                    for (int q = 0; q < kU; ++q) key[q] = i0 + q * kLgRepThreads < size ? keys[i0 + q * kLgRepThreads] : kNone;
#pragma unroll
                    for (int q = 0; q < kU; ++q) {
                        if (key[q] == kNone) continue;
                        const uint32_t bit = bit_of(key_hash(key[q]));
                        uint32_t slot = bit * 2654435761u >> 21, w;
                        while ((w = s_sus[slot]) != 0 && w != bit + 1) slot = (slot + 1) & (kLgSusSlots - 1);
                        if (w == 0) continue;
                        const uint32_t at = atomicAdd(&s_nk, 1u);
                        if (at < kLgSusKeys) s_key[at] = key[q];
                    }
                }
                __syncthreads();
                const uint32_t nk = s_nk;
                crowded = nk > kLgSusKeys;
                if (!crowded) {
                    compare(nk);
                    continue;
                }
            }
            __syncthreads();  // before the table is cleared again
        }
        if (size <= uint32_t(kLgPass)) {
            clear();
            __syncthreads();
            uint32_t found = dups;
            for (uint32_t i0 = tid; i0 < size; i0 += kU * kLgRepThreads) {
                uint64_t key[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) key[q] = i0 + q * kLgRepThreads < size ? keys[i0 + q * kLgRepThreads] : kNone;
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    if (key[q] == kNone) continue;
                    const uint64_t x = key_hash(key[q]);
                    const uint32_t print = uint32_t(x) << 14, word = print | (i0 + q * kLgRepThreads + 1);
                    uint32_t slot = __umulhi(uint32_t(x) * 0x9E3779B9u, uint32_t(kLgWords));
                    for (;;) {  // at most kLgPass of kLgWords fill: a free slot comes
                        uint32_t old = *(volatile uint32_t *)(s_tab + slot);
                        if (old == 0) old = atomicCAS(s_tab + slot, 0u, word);
                        if (old == 0) break;
                        if (((old ^ print) >> 14) == 0 && keys[(old & 16383u) - 1] == key[q]) {
                            again(key[q]);
                            break;
                        }
                        slot = slot + 1 == kLgWords ? 0 : slot + 1;
                    }
                }
            }
            // few after all: back to the bits
            crowded = __syncthreads_count(dups != found) > kLgRepThreads / 4;
            continue;
        }
        // a bucket this size holds distances repeated often beside about as
        // many others as any bucket: a table of the distinct keys and (up to
        // the last tree edge) how often each comes again, of one part of the
        // hash's values at a time (all at first; a part whose keys do not fit
        // is taken in two halves, which a one-to-one hash ends at one key).
        // 50,000 points, a fifth of them equal: 11.1 ms for all buckets, 59.8
        // when the number of parts followed a bucket's size; half of them on a
        // line, at 300 places: 4.8 and 9.8.  (Of 6,784 slots 64 probes fail
        // from about 5,500 keys on; 128 took a third longer.)
        unsigned long long *tab = reinterpret_cast<unsigned long long *>(s_tab);
        uint32_t *occ = reinterpret_cast<uint32_t *>(tab + kLgSlots);
        int bits = 0;
        uint64_t part = 0;
        for (;;) {
            clear();
            if (tid == 0) s_ns = 0;
            uint32_t more = 0;  // beyond the first of each distance
            bool placed = false;
            __syncthreads();
            for (uint32_t i0 = tid; i0 < size; i0 += kU * kLgRepThreads) {
                uint64_t key[kU];
#pragma unroll
                for (int q = 0; q < kU; ++q) key[q] = i0 + q * kLgRepThreads < size ? keys[i0 + q * kLgRepThreads] : kNone;
                if (*(volatile uint32_t *)&s_ns) break;  // a key found no slot
#pragma unroll
                for (int q = 0; q < kU; ++q) {
                    if (key[q] == kNone) continue;
                    const uint64_t x = key_hash(key[q]);
                    if (bits && x >> (64 - bits) != part) continue;
                    uint32_t slot = __umulhi(uint32_t(x) * 0x9E3779B9u, uint32_t(kLgSlots));
                    const unsigned long long tag = key[q] + 1;
                    if (*(volatile unsigned long long *)(tab + slot) != tag) {
                        const int to = lg_insert(tab, slot, tag);
                        if (to == -1) *(volatile uint32_t *)&s_ns = 1;
                        if (to < 0) continue;
                        slot = uint32_t(to);
                    }
                    ++more;
                    if (key[q] <= top) {
                        atomicAdd(occ + slot, 1u);
                        placed = true;
                    }
                }
            }
            placed = __syncthreads_or(placed);
            const bool full = s_ns != 0;
            if (!full) dups += more;
            if (!full && placed) {
                for (int i = tid; i < kLgSlots; i += kLgRepThreads)
                    if (occ[i]) atomicAdd(A.dup + lg_place(A.skey, 0, np - 1, tab[i] - 1), occ[i]);
            }
            __syncthreads();  // before the table is cleared again
            if (full) {
                ++bits;
                part <<= 1;
                continue;
            }
            while (bits > 0 && (part & 1)) {
                part >>= 1;
                --bits;
            }
            if (bits == 0) break;
            part |= 1;
        }
    }
    settle();
    dups = __reduce_add_sync(0xffffffffu, dups);
    if ((tid & 31) == 0 && dups) atomicAdd(&A.h->direct_dups, dups);
}

// ------------------------------------------------------------------ tree ---
// The other component at component c's best edge.
__device__ __forceinline__ uint32_t lg_other(const LgArgs &A, uint32_t c) {
    const uint32_t uv = __ldcg(A.buv + c), a = __ldcg(A.comp + (uv >> 16)), b = __ldcg(A.comp + (uv & 0xffffu));
    return a == c ? b : a;
}

// Edges of equal keys meet at one component in their millions (two distances
// between 20,000 points: 10^8 edges for two components), so an atomic is only
// made by an edge that comes before the one found so far: the tree of that
// cloud takes 0.55 ms, 13.0 with every edge's atomics.
__device__ __forceinline__ void lg_first(uint32_t *best, uint32_t uv) {
    if (uv < __ldcg(best)) atomicMin(best, uv);
}
__device__ __forceinline__ void lg_less(unsigned long long *best, uint64_t key) {
    if (key < __ldcg(best)) atomicMin(best, (unsigned long long)key);
}
__device__ __forceinline__ void lg_offer(const LgArgs &A, uint64_t key, uint32_t uv, uint32_t cu, uint32_t cv) {
    if (key == __ldcg(A.best + cu)) lg_first(A.buv + cu, uv);
    if (key == __ldcg(A.best + cv)) lg_first(A.buv + cv, uv);
}

// First row and column of 128 x 128 tile w of the upper triangle (T tiles a
// side), row-major.
__device__ __forceinline__ void lg_tile(int64_t w, int64_t T, int &u0, int &v0) {
    const float b = float(2 * T + 1);
    int64_t r = int64_t((b - sqrtf(b * b - 8.0f * float(w))) * 0.5f);
    r = r < 0 ? 0 : r > T - 1 ? T - 1 : r;
    while (r > 0 && r * T - r * (r - 1) / 2 > w) --r;
    while (r < T - 1 && (r + 1) * T - (r + 1) * r / 2 <= w) ++r;
    u0 = int(r) * 128;
    v0 = int(r + w - (r * T - r * (r - 1) / 2)) * 128;
}

// The tree's edges between equal points, (a, v) for the first a of each group
// of them and its others: the points by a hash table of their coordinates, in
// the candidates' place (for clouds with more zeros than the list has room
// for; a round over all keys did the same: the tree of 20,000 points of two
// kinds 1.2 ms, 0.55 this way; of 50,000 with 2,500 equal 13.3, 0.87).
// False when a wait ran out.
__device__ __noinline__ bool lg_join_equal(const LgArgs &A, int *s_ok) {
    const int n = A.n, lane = threadIdx.x & 31;
    const int gthreads = gridDim.x * kLgTreeThreads, gtid = blockIdx.x * kLgTreeThreads + threadIdx.x;
    uint32_t slots = 2;
    while (slots < 2u * uint32_t(n)) slots *= 2;  // two tables of at most 2^17, m > 2^22 entries of room
    uint32_t *tab = A.cand, *low = A.cand + slots;
    for (uint32_t i = uint32_t(gtid); i < 2 * slots; i += uint32_t(gthreads)) tab[i] = 0xffffffffu;
    if (!grid_barrier(A.h, s_ok, A.spin_limit)) return false;
    // by bits, the two zeros alike: whatever is not a number ends in a status anyway
    auto bits = [&](int v, int k) {
        const uint32_t b = __float_as_uint(A.pts[int64_t(v) * A.ld + k]);
        return b << 1 ? b : 0u;
    };
    for (int v = gtid; v < n; v += gthreads) {
        uint32_t x = 0;
        for (int k = 0; k < A.d; ++k) {
            x = (x ^ bits(v, k)) * 0x9E3779B1u;
            x ^= x >> 15;
        }
        uint32_t at = x & (slots - 1);
        for (;;) {  // at most half the slots fill
            uint32_t old = __ldcg(tab + at);
            if (old == 0xffffffffu) old = atomicCAS(tab + at, 0xffffffffu, uint32_t(v));
            if (old == 0xffffffffu) break;
            int k = 0;
            while (k < A.d && bits(int(old), k) == bits(v, k)) ++k;
            if (k == A.d) break;
            at = (at + 1) & (slots - 1);
        }
        A.buv[v] = at;
        lg_first(low + at, uint32_t(v));
    }
    if (!grid_barrier(A.h, s_ok, A.spin_limit)) return false;
    for (int v0 = gtid - lane; v0 < n; v0 += gthreads) {
        const int v = v0 + lane;
        uint32_t a = uint32_t(v);
        if (v < n) {
            a = __ldcg(low + A.buv[v]);
            A.buv[v] = 0xffffffffu;
            A.comp[v] = A.parent[v] = a;
        }
        const bool take = a != uint32_t(v);
        const unsigned who = __ballot_sync(0xffffffffu, take);
        if (!who) continue;
        uint32_t j = 0;
        if (lane == 0) j = atomicAdd(&A.h->lg_tree, uint32_t(__popc(who)));
        j = __shfl_sync(0xffffffffu, j, 0) + __popc(who & ((1u << lane) - 1u));
        if (take && j < uint32_t(n)) {
            A.tkey[j] = 0;
            A.tuv[j] = (a << 16) | uint32_t(v);
        }
    }
    return grid_barrier(A.h, s_ok, A.spin_limit);
}

// Boruvka's rounds, a grid barrier between the steps of a round: every
// component's smallest key leaving it; of the edges with that key the first
// in (u, v); components hooked along them; components renamed.  Rounds on the
// list come first: it holds every edge below the threshold, so the smallest
// it has for a component is the smallest of all.  When it joins nothing more,
// rounds on all keys: a warp reads 128 columns by 32 rows, four rows at a
// time, against the best keys it knows of its rows' and columns' components;
// only an edge that betters one is looked at further (a few in a thousand).
__global__ void __launch_bounds__(kLgTreeThreads, 2) k_large_tree(const LgArgs A) {
    __shared__ int s_ok;
    const int n = A.n, tid = threadIdx.x, lane = tid & 31;
    const int gthreads = gridDim.x * kLgTreeThreads, gtid = blockIdx.x * kLgTreeThreads + tid;
    Header *h = A.h;
    if (lg_all_equal(A)) {
        for (int j = gtid; j < n - 1; j += gthreads) {
            A.tkey[j] = 0;
            A.tuv[j] = uint32_t(j) + 1;  // (0, j + 1)
        }
        if (gtid == 0) {
            h->lg_tree = uint32_t(n - 1);
            h->lg_rounds = 1;
        }
        return;
    }
    for (int v = gtid; v < n; v += gthreads) {
        A.comp[v] = A.parent[v] = uint32_t(v);
        A.best[v] = kNone;
        A.buv[v] = 0xffffffffu;
    }
    if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
    const uint32_t listed = __ldcg(&h->lg_list), list = listed <= A.lcap ? listed : 0u;
    uint32_t joined = 0, rounds = 0, passes = 0;
    uint32_t live = uint32_t(gtid) < list ? (list - gtid - 1) / gthreads + 1 : 0u;  // entries of this thread
    const uint64_t first = __ldcg(&h->lg_first);
    bool on_list = list > 0;
    if (__ldcg(&h->lg_lo) != 0) {  // the list has no zeros: equal points first
        if (!lg_join_equal(A, &s_ok)) return;
        joined = __ldcg(&h->lg_tree);
    }
    const int64_t T = (n + 127) / 128, tiles = T * (T + 1) / 2;
    const int warps = gthreads >> 5, gwarp = gtid >> 5;
    while (joined < uint32_t(n - 1)) {
        ++rounds;
        if (on_list) {
            // the shortest edges first: nearly every component has one among
            // them, and what is left then betters few (all at once: the first
            // round's two atomics per entry took most of the search)
            for (uint32_t j = 0; j < live; j += 4) {
                uint64_t k[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) k[q] = j + q < live ? A.lkey[gtid + size_t(j + q) * gthreads] : kNone;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (k[q] >= first) continue;
                    const uint32_t uv = A.luv[gtid + size_t(j + q) * gthreads];
                    const uint32_t cu = __ldcg(A.comp + (uv >> 16)), cv = __ldcg(A.comp + (uv & 0xffffu));
                    if (cu == cv) continue;
                    if (k[q] < __ldcg(A.best + cu)) atomicMin(A.best + cu, (unsigned long long)k[q]);
                    if (k[q] < __ldcg(A.best + cv)) atomicMin(A.best + cv, (unsigned long long)k[q]);
                }
            }
            if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
            // the others; a thread's entries, every gthreads-th, lose those
            // within a component
            const uint32_t had = live;
            live = 0;
            for (uint32_t j = 0; j < had; j += 4) {
                uint64_t k[4], bu[4], bv[4];
                uint32_t uv[4], cu[4], cv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const size_t i = gtid + size_t(j + q) * gthreads;
                    uv[q] = j + q < had ? A.luv[i] : 0u;
                    k[q] = j + q < had ? A.lkey[i] : kNone;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    cu[q] = __ldcg(A.comp + (uv[q] >> 16));
                    cv[q] = __ldcg(A.comp + (uv[q] & 0xffffu));
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    bu[q] = __ldcg(A.best + cu[q]);
                    bv[q] = __ldcg(A.best + cv[q]);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (cu[q] == cv[q]) continue;  // past the end too: an edge of vertex 0 with itself
                    if (k[q] < bu[q]) atomicMin(A.best + cu[q], (unsigned long long)k[q]);
                    if (k[q] < bv[q]) atomicMin(A.best + cv[q], (unsigned long long)k[q]);
                    if (live < j + q) {
                        const size_t i = gtid + size_t(live) * gthreads;
                        A.luv[i] = uv[q];
                        A.lkey[i] = k[q];
                    }
                    ++live;
                }
            }
            if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
            for (uint32_t j = 0; j < live; j += 4) {
                uint64_t k[4], bu[4], bv[4];
                uint32_t uv[4], cu[4], cv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const size_t i = gtid + size_t(j + q) * gthreads;
                    uv[q] = j + q < live ? A.luv[i] : 0u;
                    k[q] = j + q < live ? A.lkey[i] : 0u;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    cu[q] = __ldcg(A.comp + (uv[q] >> 16));
                    cv[q] = __ldcg(A.comp + (uv[q] & 0xffffu));
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    bu[q] = __ldcg(A.best + cu[q]);
                    bv[q] = __ldcg(A.best + cv[q]);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (cu[q] == cv[q]) continue;
                    if (k[q] == bu[q]) lg_first(A.buv + cu[q], uv[q]);
                    if (k[q] == bv[q]) lg_first(A.buv + cv[q], uv[q]);
                }
            }
        } else {
            ++passes;
            // first a sixteenth of the rows, for bounds that few edges better
            // in the pass over all keys (without them nearly every row of the
            // first tiles took the long way: 6.8 ms instead of 2.7 at 30,000
            // points in eight clusters)
            for (int64_t w = gwarp; w < tiles; w += warps) {
                int u0, v0;
                lg_tile(w, T, u0, v0);
                uint32_t cv[4];
                uint64_t mv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = v0 + q * 32 + lane;
                    cv[q] = v < n ? __ldcg(A.comp + v) : 0xffffffffu;
                    mv[q] = kNone;
                }
                for (int i = 0; i < 8; i += 4) {
                    uint64_t key[4][4];
                    uint32_t cu[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int u = u0 + (i + r) * 16 + int(w & 15);
                        cu[r] = u < n ? __ldcg(A.comp + u) : 0xffffffffu;
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int u = u0 + (i + r) * 16 + int(w & 15);
                        const int64_t e0 = edge_index(n, u, 0);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int v = v0 + q * 32 + lane;
                            key[r][q] = u < v && v < n && cu[r] != cv[q] ? __ldcg(A.mat + e0 + v) : kNone;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        uint64_t mine = kNone;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint64_t k = key[r][q];
                            mv[q] = k < mv[q] ? k : mv[q];
                            mine = k < mine ? k : mine;
                        }
                        const uint32_t mh = __reduce_min_sync(0xffffffffu, uint32_t(mine >> 32));
                        const uint32_t ml =
                            __reduce_min_sync(0xffffffffu, uint32_t(mine >> 32) == mh ? uint32_t(mine) : 0xffffffffu);
                        const uint64_t mn = (uint64_t(mh) << 32) | ml;
                        if (lane == r && mn != kNone && mn < __ldcg(A.best + cu[r]))
                            atomicMin(A.best + cu[r], (unsigned long long)mn);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (mv[q] != kNone && mv[q] < __ldcg(A.best + cv[q])) atomicMin(A.best + cv[q], (unsigned long long)mv[q]);
            }
            if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
            for (int64_t w = gwarp; w < 4 * tiles; w += warps) {
                int u0, v0;
                lg_tile(w >> 2, T, u0, v0);
                u0 += int(w & 3) * 32;
                if (u0 >= n - 1 || u0 >= v0 + 127) continue;
                // bounds: a key at or below what others found so far, then
                // only keys below what this warp saw (its edges come in
                // (u, v) order, so a later equal key is no better)
                uint32_t cv[4];
                uint64_t bv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int v = v0 + q * 32 + lane;
                    cv[q] = v < n ? __ldcg(A.comp + v) : 0xffffffffu;
                    bv[q] = v < n ? __ldcg(A.best + cv[q]) : 0u;
                    if (bv[q] != kNone && v < n) ++bv[q];
                }
                // rows and columns of one component have nothing to offer
                const uint32_t c0 = __shfl_sync(0xffffffffu, cv[0], 0);
                bool alike = true;
#pragma unroll
                for (int q = 0; q < 4; ++q) alike &= cv[q] == c0 || v0 + q * 32 + lane >= n;
                alike = __all_sync(0xffffffffu, alike);
                const int ul = u0 + lane;
                const uint32_t cul = ul < n ? __ldcg(A.comp + ul) : 0xffffffffu;
                uint64_t bul = ul < n ? __ldcg(A.best + cul) : 0u;
                if (bul != kNone && ul < n) ++bul;
                if (alike && __all_sync(0xffffffffu, cul == c0 || ul >= n)) continue;
                // whole tiles off the diagonal need no look at u < v < n
                const bool inner = u0 + 31 < v0 && v0 + 127 < n;
                const uint64_t *line = A.mat + (edge_index(n, u0, 0) + v0 + lane);
                uint32_t rowc = 0xffffffffu, colc = 0xffffffffu;  // row u0 + lane's edge: column; the columns': rows
                for (int i0 = 0; i0 < 32; i0 += 4) {
                    uint64_t key[4][4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int u = u0 + i0 + r;
                        const uint32_t cu = __shfl_sync(0xffffffffu, cul, i0 + r);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int v = v0 + q * 32 + lane;
                            key[r][q] = cu != cv[q] && (inner || (u < v && v < n)) ? __ldcs(line + q * 32) : kNone;
                        }
                        line += n - u - 2;
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        // by the high words first: a pass over all keys is
                        // bound by the instructions per key otherwise
                        const uint32_t bh = __shfl_sync(0xffffffffu, uint32_t(bul >> 32), i0 + r);
                        bool near = false;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t ch = uint32_t(bv[q] >> 32);
                            near |= uint32_t(key[r][q] >> 32) <= (bh > ch ? bh : ch);
                        }
                        if (!__any_sync(0xffffffffu, near)) continue;
                        const uint64_t bu = __shfl_sync(0xffffffffu, bul, i0 + r);
                        bool hit = false;
#pragma unroll
                        for (int q = 0; q < 4; ++q) hit |= key[r][q] < bu || key[r][q] < bv[q];
                        if (!__any_sync(0xffffffffu, hit)) continue;
                        const uint32_t cu = __shfl_sync(0xffffffffu, cul, i0 + r);
                        // the row's smallest key and the first edge that has it
                        uint64_t mine = kNone;
                        uint32_t at = 0xffffffffu;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (key[r][q] < mine) {
                                mine = key[r][q];
                                at = uint32_t(q * 32 + lane);
                            }
                        const uint32_t hi = uint32_t(mine >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
                        const uint32_t lo = hi == mh ? uint32_t(mine) : 0xffffffffu;
                        const uint32_t ml = __reduce_min_sync(0xffffffffu, lo);
                        const uint64_t mn = (uint64_t(mh) << 32) | ml;
                        at = __reduce_min_sync(0xffffffffu, mine == mn ? at : 0xffffffffu);
                        if (mn < bu) {
                            if (lane == 0) lg_less(A.best + cu, mn);
                            if (cul == cu && mn < bul) bul = mn;
                            if (lane == i0 + r) rowc = at;
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            if (key[r][q] < bv[q]) {
                                bv[q] = key[r][q];
                                lg_less(A.best + cv[q], bv[q]);
                                colc = (colc & ~(0xffu << (8 * q))) | uint32_t(i0 + r) << (8 * q);
                            }
                        }
                    }
                }
                // the edges that bettered a row's component, and the last
                // that bettered a column's (it has that column's smallest
                // key), with one addition to the counter (one per row and 32
                // columns: clouds of many equal keys waited for it alone)
                uint32_t total = 0, at[5];
                bool has[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    has[q] = q < 4 ? ((colc >> (8 * q)) & 0xffu) != 0xffu : rowc != 0xffffffffu;
                    const unsigned who = __ballot_sync(0xffffffffu, has[q]);
                    at[q] = total + __popc(who & ((1u << lane) - 1u));
                    total += __popc(who);
                }
                if (total == 0) continue;
                uint32_t j = 0;
                if (lane == 0) j = atomicAdd(&h->lg_cand, total);
                j = __shfl_sync(0xffffffffu, j, 0);
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    if (!has[q] || j + at[q] >= A.ccap) continue;
                    const int u = q < 4 ? u0 + int((colc >> (8 * q)) & 0xffu) : u0 + lane;
                    A.cand[j + at[q]] = uint32_t(edge_index(n, u, v0 + (q < 4 ? q * 32 + lane : int(rowc))));
                }
            }
            if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
            const uint32_t cands = __ldcg(&h->lg_cand);
            if (gtid == 0) h->lg_offers += cands;
            const bool whole = cands > A.ccap;  // the list does not hold them all: every edge instead
            const int64_t len = whole ? A.m : int64_t(cands);
            for (int64_t i = gtid; i < len; i += gthreads) {
                const int64_t e = whole ? i : int64_t(__ldcg(A.cand + i));
                uint32_t u, v;
                edge_uv(e, n, u, v);
                const uint32_t cu = __ldcg(A.comp + u), cv = __ldcg(A.comp + v);
                if (cu != cv) lg_offer(A, __ldcg(A.mat + e), (u << 16) | v, cu, cv);
            }
        }
        if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
        // hook: of two components that chose the same edge the smaller stays
        for (int c0 = gtid - lane; c0 < n; c0 += gthreads) {
            const uint32_t c = uint32_t(c0 + lane);
            bool take = false;
            uint32_t o = 0;
            if (c < uint32_t(n) && __ldcg(A.comp + c) == c && __ldcg(A.buv + c) != 0xffffffffu) {
                o = lg_other(A, c);
                take = !(__ldcg(A.buv + o) != 0xffffffffu && lg_other(A, o) == c && c < o);
            }
            const unsigned who = __ballot_sync(0xffffffffu, take);
            if (!who) continue;
            uint32_t j = 0;
            if (lane == 0) j = atomicAdd(&h->lg_tree, uint32_t(__popc(who)));
            j = __shfl_sync(0xffffffffu, j, 0) + __popc(who & ((1u << lane) - 1u));
            if (take) {
                A.parent[c] = o;
                if (j < uint32_t(n)) {
                    A.tkey[j] = __ldcg(A.best + c);
                    A.tuv[j] = __ldcg(A.buv + c);
                }
            }
        }
        if (gtid == 0) h->lg_cand = 0;
        if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
        for (int v = gtid; v < n; v += gthreads) {
            uint32_t r = __ldcg(A.comp + v);
            for (int i = 0;; ++i) {
                const uint32_t p = __ldcg(A.parent + r);
                if (p == r) break;
                if (i > n) {  // a cycle: never, with one order of the edges
                    set_status(h, PH0_EINTERNAL);
                    break;
                }
                const uint32_t g = __ldcg(A.parent + p);
                if (g != p) A.parent[r] = g;  // path halving (only moves toward the root)
                r = g;
            }
            A.comp[v] = r;
            A.best[v] = kNone;
            A.buv[v] = 0xffffffffu;
        }
        const uint32_t now = __ldcg(&h->lg_tree);
        if (!grid_barrier(h, &s_ok, A.spin_limit)) return;
        if (now == joined) {
            if (!on_list) {  // keys that are not numbers
                if (gtid == 0) set_status(h, PH0_EINTERNAL);
                break;
            }
            on_list = false;
        }
        joined = now;
    }
    if (gtid == 0) {
        h->lg_rounds = rounds;
        h->lg_passes = passes;
    }
}

// The tree's edges in order: runs sorted by a CTA each (bitonic), then every
// edge's place from binary searches in the other runs.
__global__ void __launch_bounds__(1024) k_large_runs(const LgArgs A) {
    __shared__ uint64_t s_k[kLgRun];
    __shared__ uint32_t s_u[kLgRun];
    const int base = blockIdx.x * kLgRun, tid = threadIdx.x;
    const uint32_t have = A.h->lg_tree;
    for (int i = tid; i < kLgRun; i += 1024) {
        const uint32_t g = uint32_t(base + i);
        const bool in = g < uint32_t(A.n - 1) && g < have;
        s_k[i] = in ? A.tkey[g] : kNone;
        s_u[i] = in ? A.tuv[g] : 0xffff0000u | (g & 0xffffu);  // missing after an error: no edge, all different
    }
    for (int kk = 2; kk <= kLgRun; kk <<= 1)
        for (int j = kk >> 1; j > 0; j >>= 1) {
            __syncthreads();
            const int i = ((tid & ~(j - 1)) << 1) | (tid & (j - 1)), o = i | j;
            const uint64_t a = s_k[i], b = s_k[o];
            const uint32_t ua = s_u[i], ub = s_u[o];
            if (lg_before(b, ub, a, ua) == ((i & kk) == 0)) {
                s_k[i] = b;
                s_k[o] = a;
                s_u[i] = ub;
                s_u[o] = ua;
            }
        }
    __syncthreads();
    for (int i = tid; i < kLgRun && base + i < A.n; i += 1024) {
        A.tkey[base + i] = s_k[i];
        A.tuv[base + i] = s_u[i];
    }
}

// A warp per edge, a lane per run (at most 32 up to 65,535 points).
__global__ void __launch_bounds__(256) k_large_merge(const LgArgs A) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, np = A.n - 1;
    if (i >= np) return;
    const uint64_t k = A.tkey[i];
    const uint32_t uv = A.tuv[i];
    const int start = lane * kLgRun;
    int lo = start, hi = start + kLgRun < np ? start + kLgRun : np;
    if (lane == i / kLgRun) lo = hi = i;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (lg_before(A.tkey[mid], A.tuv[mid], k, uv)) lo = mid + 1;
        else hi = mid;
    }
    const int rank = __reduce_add_sync(0xffffffffu, start < np ? uint32_t(lo - start) : 0u);
    if (lane == 0) {
        A.skey[rank] = k;  // rank < np: places among np edges
        A.suv[rank] = uv;
    }
}
static_assert(32 * kLgRun >= kMaxN - 1, "a lane per run");

// ---------------------------------------------------------- counts, bars ---
// s(e), t(e), order and a as in k_direct.cu.  cnt[s] counts the edges at s(e);
// those as long as a run of tree edges of one key but behind the run's last
// are counted apart, in late[end of the run] (a(p) takes them, where order(p)
// has them only from the run's end on).  The counts of the kLgHot longest tree
// edges, where nearly all edges up to the last one fall, are kept in shared
// memory; the others go to the L2 cache.
// An edge as long as a tree edge: its run comes from a table of the CTA
// (kLgRuns runs, by a hash of the key, filled as they are met), and most such
// edges are behind the run's last (copies of few points: the tree joins them
// in the rows of the first copies), which the table counts; the others are
// searched for in the run, and the gap between two of its edges is remembered
// with the edges counted there.  20,000 points of two kinds, whose 200M edges
// all come here: 0.8 ms; 64 with a search over the tree's edges and three
// atomics on the L2 cache's words for every edge.
struct LgRuns {
    // key (kNone: a free slot), first and end (in the high half) of a run,
    // number of its last edge (kUnknown until these are written), edges behind
    unsigned long long key[kLgRuns];
    uint32_t run[kLgRuns], last[kLgRuns], late[kLgRuns];
    static constexpr uint32_t kUnknown = 0xffffffffu;
    static_assert(kMaxN <= 65536, "places below 2^16");
};
struct LgGap {  // a thread's: key, (u, v) from and to, edges counted there, place
    uint64_t key = kNone;
    uint32_t from = 0, to = 0, n = 0;
    int s = 0;
    __device__ void flush(const LgArgs &A, uint32_t *s_cnt, int base) {
        if (n) atomicAdd(s >= base ? s_cnt + (s - base) : A.cnt + s, n);
        n = 0;
    }
};
// An edge as long as tree edge t (-1: not known, nor whether there is one)
// that is not known to lie behind its run; h, known: the key's slot in the
// table and its run's last edge.  Not inlined: the counting loop holds eight
// copies of what is, and most warps come by here now and then (20,000 random
// whole numbers on a line, all counts: 0.63 ms inlined, 0.46).
__device__ __noinline__ void lg_tie(const LgArgs &A, LgRuns *runs, uint32_t *s_cnt, LgGap &gap, uint64_t key, int64_t e,
                                    int t, uint32_t h, uint32_t known) {
    const int np = A.n - 1, base = np - (np < kLgHot ? np : kLgHot);
    int end;
    if (known != LgRuns::kUnknown) {
        __threadfence_block();
        const uint32_t run = *(volatile uint32_t *)&runs->run[h];
        t = int(run & 0xffffu);
        end = int(run >> 16);
    } else {
        if (t < 0) {
            t = lg_place(A.skey, 0, base, key);
            if (A.skey[t] != key) {
                atomicAdd(A.cnt + t, 1u);
                return;
            }
        }
        // the run's end: steps of 1, 2, 4, ... from its first
        end = t + 1;
        if (end < np && A.skey[end] == key) {
            int step = 1;
            while (end + step < np && A.skey[end + step] == key) {
                end += step;
                step *= 2;
            }
            int hi = end + step < np ? end + step : np;  // [end] is of the run, [hi] is not
            while (end + 1 < hi) {
                const int mid = (end + hi) >> 1;
                if (A.skey[mid] == key) end = mid;
                else hi = mid;
            }
            end = hi;
        }
        const uint32_t last = A.suv[end - 1], elast = uint32_t(edge_index(A.n, last >> 16, last & 0xffffu));
        if (atomicCAS(&runs->key[h], (unsigned long long)kNone, (unsigned long long)key) == kNone) {
            *(volatile uint32_t *)&runs->run[h] = uint32_t(t) | uint32_t(end) << 16;
            __threadfence_block();
            *(volatile uint32_t *)&runs->last[h] = elast;  // from now on the run is known
        }
        if (uint32_t(e) > elast) {
            atomicAdd(A.late + end, 1u);
            return;
        }
    }
    uint32_t u, v;
    edge_uv(e, A.n, u, v);
    const uint32_t uv = (u << 16) | v;
    if (key != gap.key || uv < gap.from || uv > gap.to) {
        gap.flush(A, s_cnt, base);
        int lo = t, hi = end - 1;  // suv[end - 1] >= uv
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (A.suv[mid] < uv) lo = mid + 1;
            else hi = mid;
        }
        gap.key = key;
        gap.s = lo;
        gap.from = lo > t ? A.suv[lo - 1] + 1 : 0u;
        gap.to = A.suv[lo];
    }
    ++gap.n;
}
// PREFIX (the early path): the keys counted are also kept for step 3, with
// the histogram of their partitions.
template <bool PREFIX>
__global__ void __launch_bounds__(kLgCountThreads, 2) k_large_count(const LgArgs A) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ uint32_t s_hist[PREFIX ? kLgParts : 1];
    if constexpr (PREFIX)
        for (int i = threadIdx.x; i < kLgParts; i += kLgCountThreads) s_hist[i] = 0;
    const int np = A.n - 1, hot = np < kLgHot ? np : kLgHot, base = np - hot, tid = threadIdx.x;
    uint64_t *s_key = reinterpret_cast<uint64_t *>(s_dyn);      // [hot]
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_key + hot);  // [hot]
    // where to look: the first hot key at or beyond each of kLgLut steps of
    // the way from the second to the last (a search over them all takes a warp
    // with a few keys to place 13 steps: 3.0 ms instead of 1.15 at 30,000
    // points in eight clusters, 450M keys)
    __shared__ uint16_t s_lut[kLgLut + 2];
    __shared__ LgRuns s_runs;
    for (int i = tid; i < kLgRuns; i += kLgCountThreads) {
        s_runs.key[i] = kNone;
        s_runs.last[i] = LgRuns::kUnknown;
        s_runs.late[i] = 0;
    }
    for (int i = tid; i < hot; i += kLgCountThreads) {
        s_key[i] = A.skey[base + i];
        s_cnt[i] = 0;
    }
    const int64_t gtid = int64_t(blockIdx.x) * kLgCountThreads + tid, gthreads = int64_t(gridDim.x) * kLgCountThreads;
    for (int64_t j = gtid; j < np; j += gthreads) {
        const unsigned long long p = A.kill_key[j];
        if (p < (unsigned long long)np) A.low[p] = A.kill_val[j];
    }
    if (lg_all_equal(A)) {
        for (int64_t j = gtid; j < np; j += gthreads) A.cnt[j] = 1;
        if (gtid == 0) {
            A.late[np] = uint32_t(A.m - np);
            A.dup[0] = A.h->direct_dups = uint32_t(A.m - 1);
            A.h->lg_keep = uint32_t(A.m);
        }
        return;
    }
    __syncthreads();
    // the steps go from the second key on: many tree edges may have the first,
    // zero, whose distance from the others would leave these in one step
    // (a tree that a wait's end left unfinished has kNone for its missing
    // edges: what is read past the last key must not count as one up to it)
    const uint64_t top = s_key[hot - 1] < kNone ? s_key[hot - 1] : kNone - 1, bottom = s_key[0];
    const uint64_t second = s_key[lg_place(s_key, 0, hot - 1, bottom < kNone ? bottom + 1 : kNone)];
    int shift = bitlen64(s_key[hot - 1] - second) - kLgLutBits;
    if (shift < 0) shift = 0;
    for (int i = tid; i < kLgLut + 2; i += kLgCountThreads) s_lut[i] = uint16_t(hot - 1);
    __syncthreads();
    for (int i = tid; i < hot; i += kLgCountThreads) {
        if (s_key[i] < second) continue;
        const int b = int((s_key[i] - second) >> shift);
        const int a = i > 0 && s_key[i - 1] >= second ? int((s_key[i - 1] - second) >> shift) : -1;
        for (int j = a + 1; j <= b; ++j) s_lut[j] = uint16_t(i);
    }
    __syncthreads();
    if constexpr (!PREFIX) lg_reps(A, uint32_t(gtid), uint32_t(gthreads));
    LgGap gap;
    auto tie = [&](uint64_t key, int64_t e, int t) {
        uint32_t h = (uint32_t(key >> 32) * 0x9E3779B9u + uint32_t(key) * 0x7F4A7C15u) >> 23, known = LgRuns::kUnknown;
        static_assert(kLgRuns == 512, "nine bits of the hash");
        for (int pr = 0; pr < 2; ++pr) {
            const uint64_t k = *(volatile uint64_t *)&s_runs.key[h];
            if (k == key) known = *(volatile uint32_t *)&s_runs.last[h];
            if (k == key || k == kNone) break;
            h = (h + 1) & (kLgRuns - 1);
        }
        if (known != LgRuns::kUnknown && uint32_t(e) > known) atomicAdd(&s_runs.late[h], 1u);
        else lg_tie(A, &s_runs, s_cnt, gap, key, e, t, h, known);
    };
    auto take = [&](uint64_t key, int64_t e) {
        if (key > top) return;
        if (key > bottom) {
            const int b = key > second ? int((key - second) >> shift) : 0;
            const int i = lg_place(s_key, s_lut[b], s_lut[b + 1], key);
            if (s_key[i] == key) tie(key, e, base + i);
            else atomicAdd(s_cnt + i, 1u);
        } else {
            tie(key, e, base == 0 ? 0 : -1);  // base 0: the first tree edge has the least key of all
        }
    };
    constexpr int kU = 8;
    for (int64_t b = int64_t(blockIdx.x) * kLgCountThreads; b < A.m; b += kU * gthreads) {
        const int64_t e0 = b + tid;
        uint64_t key[kU];
#pragma unroll
        for (int q = 0; q < kU; ++q) key[q] = e0 + q * gthreads < A.m ? __ldcs(A.mat + e0 + q * gthreads) : kNone;
#pragma unroll
        for (int q = 0; q < kU; ++q) take(key[q], e0 + q * gthreads);
        if constexpr (PREFIX) {
            uint32_t mine = 0;
#pragma unroll
            for (int q = 0; q < kU; ++q) mine += key[q] <= top;
            // an addition per warp (of 20,011 uniform points few warps have
            // any; one per CTA, with its barriers, took 0.93 ms instead of
            // 0.38 there, and 2.9 instead of 3.1 where a third are kept)
            if (!__any_sync(0xffffffffu, mine != 0)) continue;
            uint32_t at = lg_rank(mine, &A.h->lg_keep);
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                if (key[q] > top) continue;
                A.keep[at++] = key[q];
                atomicAdd(s_hist + hash_part(part_hash(key[q])), 1u);
            }
        }
    }
    gap.flush(A, s_cnt, base);
    __syncthreads();
    if constexpr (PREFIX)
        for (int i = tid; i < kLgParts; i += kLgCountThreads)
            if (s_hist[i]) atomicAdd(&A.h->phist[0][i], s_hist[i]);
    for (int i = tid; i < hot; i += kLgCountThreads)
        if (s_cnt[i]) atomicAdd(A.cnt + base + i, s_cnt[i]);
    for (int i = tid; i < kLgRuns; i += kLgCountThreads)
        if (s_runs.late[i]) atomicAdd(A.late + (s_runs.run[i] >> 16), s_runs.late[i]);
}

// Each CTA adds up the counts before its 1024 tree edges, then writes their
// bars; the last one to finish writes the bar that never dies.  order(p): the
// edges counted up to place p; a(p): those up to the end of p's run of equal
// keys and the late ones there, less the repeated ones.
__global__ void __launch_bounds__(1024) k_large_emit(const LgArgs A) {
    __shared__ uint32_t s_w[33], s_pre[2], s_upto[1025], s_beyond;
    __shared__ int s_last, s_end;
    const int tid = threadIdx.x, np = A.n - 1, base = blockIdx.x * 1024, p = base + tid;
    const int stop = base + 1024 < np ? base + 1024 : np;  // of this CTA's
    if (tid < 2) s_pre[tid] = 0;
    if (tid == 0) s_beyond = 0;
    __syncthreads();
    uint32_t so = 0, sa = 0;
    for (int i = tid; i < base; i += 1024) {
        const uint32_t c = A.cnt[i] + A.late[i];
        so += c;
        sa += c - A.dup[i];
    }
    so = __reduce_add_sync(0xffffffffu, so);
    sa = __reduce_add_sync(0xffffffffu, sa);
    if ((tid & 31) == 0) {
        atomicAdd(s_pre, so);
        atomicAdd(s_pre + 1, sa);
    }
    const uint64_t key = p < np ? A.skey[p] : kNone;
    int end = p + 1;  // of p's run
    if (end < np && A.skey[end] == key) {
        int hi = np;
        while (end < hi) {
            const int mid = (end + hi) >> 1;
            if (A.skey[mid] <= key) end = mid + 1;
            else hi = mid;
        }
    }
    if (p == stop - 1) s_end = end;
    __syncthreads();
    const uint32_t c = p < np ? A.cnt[p] + A.late[p] : 0u, a = p < np ? c - A.dup[p] : 0u;
    uint32_t total;
    const uint32_t order = s_pre[0] + block_scan<1024>(c, s_w, total) + c;
    s_upto[tid] = s_pre[1] + block_scan<1024>(a, s_w, total);
    if (tid == 0) s_upto[1024] = s_pre[1] + total;
    // the last run, beyond this CTA's places
    sa = 0;
    for (int i = stop + tid; i < s_end; i += 1024) sa += A.cnt[i] + A.late[i] - A.dup[i];
    sa = __reduce_add_sync(0xffffffffu, sa);
    if ((tid & 31) == 0 && sa) atomicAdd(&s_beyond, sa);
    __syncthreads();
    const uint32_t aval = p < np ? (end > stop ? s_upto[1024] + s_beyond : s_upto[end - base]) + A.late[end] : 0u;
    uint32_t low = 0;
    if (p < np) {
        const uint32_t uv = A.suv[p];
        low = A.low[p];
        ph0_bar b;
        b.u = int32_t(uv >> 16);
        b.v = int32_t(uv & 0xffffu);
        b.a = aval;
        b.low = int32_t(low);
        b.order = int64_t(order) - 1;
        b.death_sq = __longlong_as_double((long long)key);
        b.death = __dsqrt_rn(b.death_sq);
        A.bars[p] = b;
    }
    low = __reduce_xor_sync(0xffffffffu, low);
    if ((tid & 31) == 0) atomicXor(&A.h->inf_xor, low);  // starts as the XOR of 0..n-1 (k_reduce_init)
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&A.h->direct_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last || tid != 0) return;
    __threadfence();
    Header *h = A.h;
    uint32_t v = ld_volatile(&h->inf_xor);
    if (v >= uint32_t(A.n)) {  // only after a reported error
        set_status(h, PH0_EINTERNAL);
        v = 0;
    }
    h->inf_vertex = int32_t(v);
    h->kmin = A.skey[0];
    const int64_t keys = A.prefix ? int64_t(h->lg_keep) : A.m;
    h->n_distinct = keys - int64_t(h->direct_dups);
    h->sort_passes = 0;
    h->key_bits = make_plan(h->kmin, h->kmax).bits;
    h->windows = int32_t(h->lg_rounds);
    h->edges_scanned = A.m;
    h->sorted_edges = keys;
    h->direct = 1;
    if (A.inf) {
        ph0_inf_bar b;
        b.vertex = int32_t(v);
        b._pad = 0;
        b.birth = 0.0;
        b.death = __longlong_as_double(0x7ff0000000000000ll);  // +inf
        *A.inf = b;
    }
}

int large_nsub(int64_t m) {
    const int64_t per = (m + kLgParts - 1) / kLgParts;
    if (per <= kLgBucket + kLgBucket / 4) return 1;
    return int((per + kLgBucket - 1) / kLgBucket);
}

// The regions of this form within the sorts' (key, value and look-back
// buffers, candidate lists) and the reduction's.
LgArgs large_args(void *ws, const Layout &L, ph0_bar *bars, ph0_inf_bar *inf, uint32_t spin_limit, bool prefix,
                  size_t &zero, size_t &zero_end) {
    LgArgs A;
    const size_t n = size_t(L.n);
    A.m = L.m;
    A.n = int(L.n);
    A.pts = nullptr;
    A.ld = A.d = 0;
    A.nsub = large_nsub(L.m);
    A.mat = at<uint64_t>(ws, L.key[0]);
    // prefix: the kept keys in key[1], by partition in the value buffers, by
    // bucket in key[1] again; the records in place of the keys by edge, which
    // only the steps before read
    A.prefix = prefix;
    A.keep = at<uint64_t>(ws, L.key[1]);
    A.part = at<uint64_t>(ws, prefix ? L.val[0] : L.key[1]);
    A.bkt = at<uint64_t>(ws, prefix ? L.key[1] : L.val[0]);
    A.rep = at<LgRepeat>(ws, prefix ? L.key[0] : L.val[0]);
    const int64_t wcap = L.m < kMaxWindow ? L.m : kMaxWindow;
    A.lkey = at<uint64_t>(ws, L.candr);
    A.luv = at<uint32_t>(ws, L.cand[0]);
    A.lcap = uint32_t(wcap < kLgListRoom * L.n ? wcap : kLgListRoom * L.n);  // above lg_samples
    A.cand = at<uint32_t>(ws, L.cand[1]);
    A.ccap = uint32_t(wcap);
    A.comp = at<uint32_t>(ws, L.comp);
    A.parent = at<uint32_t>(ws, L.parent);
    A.best = at<unsigned long long>(ws, L.res);
    A.tkey = at<uint64_t>(ws, L.kill_key[1]);
    A.tuv = at<uint32_t>(ws, L.kill_val[1]);
    A.kill_key = at<unsigned long long>(ws, L.kill_key[0]);
    A.kill_val = at<uint32_t>(ws, L.kill_val[0]);
    size_t off = L.look[0];
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    const size_t nb = size_t(kLgParts) * size_t(A.nsub);
    zero = off;
    A.cnt = at<uint32_t>(ws, take(4 * n));
    A.late = at<uint32_t>(ws, take(4 * n));
    A.dup = at<uint32_t>(ws, take(4 * n));
    A.bcnt = at<uint32_t>(ws, take(4 * nb));
    A.bcur = at<uint32_t>(ws, take(4 * nb));
    zero_end = off;
    A.boff = at<uint32_t>(ws, take(4 * nb));
    A.poff = at<uint32_t>(ws, take(4 * (kLgParts + 1)));
    A.pcur = at<uint32_t>(ws, take(4 * kLgParts));
    A.buv = at<uint32_t>(ws, take(4 * n));
    A.skey = at<uint64_t>(ws, take(8 * n));
    A.suv = at<uint32_t>(ws, take(4 * n));
    A.low = at<uint32_t>(ws, take(4 * n));
    A.h = at<Header>(ws, L.hdr);
    A.bars = bars;
    A.inf = inf;
    A.spin_limit = spin_limit;
    // at least 8 * kMaxRadix bytes per 4096 edges, a byte per edge: the
    // regions take 36 n bytes and 12 per 5632 edges
    if (off > L.look[0] + 8 * size_t(L.tiles) * kMaxRadix) A.n = 0;
    return A;
}

cudaError_t launch_parts(const LgArgs &A, cudaStream_t s) {
    const cudaError_t e = smem_limit<move_smem(0)>(k_large_move<0>);
    if (e != cudaSuccess) return e;
    const int64_t moves = (A.m + kLgTile - 1) / kLgTile;
    const int ctas = 2048 / kLgThreads * sm_count();
    k_large_move<0><<<unsigned(moves < ctas ? moves : ctas), kLgThreads, move_smem(0), s>>>(A);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_dist(const float *pts, int64_t n, int32_t d, int64_t ld, uint64_t *key, uint32_t *val, Header *h,
                        cudaStream_t s, int split16, int tile, const int32_t *gate, bool wide, DistForm form);

// Up to the tree's edges in order: *records, n-1 of them ((u << 16) | v), for
// the reduction.
cudaError_t launch_large_tree(void *ws, const Layout &L, const float *pts, int64_t n, int32_t d, int64_t ld,
                              int split16, int tile, uint32_t spin_limit, bool prefix, const uint32_t **records,
                              cudaStream_t s, cudaEvent_t after_dist, cudaEvent_t after_part) {
    size_t zero, zero_end;
    LgArgs A = large_args(ws, L, nullptr, nullptr, spin_limit, prefix, zero, zero_end);
    if (A.n == 0) return cudaErrorInvalidValue;
    A.pts = pts;
    A.ld = ld;
    A.d = d;
    *records = A.suv;
    cudaError_t e = cudaMemsetAsync(at<char>(ws, L.hdr), 0, sizeof(Header), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(at<char>(ws, zero), 0, zero_end - zero, s);
    if (e == cudaSuccess)
        e = launch_dist(pts, n, d, ld, at<uint64_t>(ws, L.key[0]), nullptr, A.h, s, split16, tile, nullptr, false,
                        prefix ? kDistKeys : kDistHashed);
    if (e == cudaSuccess && after_dist) e = cudaEventRecord(after_dist, s);
    if (e == cudaSuccess) e = smem_limit<32768 * 4>(k_large_prep);
    if (e != cudaSuccess) return e;
    k_large_sample<<<unsigned((lg_samples(A.n) + 255) / 256), 256, 0, s>>>(A);  // into the list's place
    k_large_prep<<<1, 1024, 32768 * 4, s>>>(A);
    const int ctas = 2 * sm_count();
    if (prefix) k_large_list<<<unsigned(ctas), 1024, 0, s>>>(A);
    else if ((e = launch_parts(A, s)) != cudaSuccess) return e;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (after_part && (e = cudaEventRecord(after_part, s)) != cudaSuccess) return e;

    // fewer CTAs for small clouds (cheaper grid barriers): a warp per 128 columns by 32 rows
    const int64_t T = (n + 127) / 128, want = (T * (T + 1) * 2 * 32 + kLgTreeThreads - 1) / kLgTreeThreads;
    LgArgs args = A;
    void *params[] = {&args};
    e = cudaLaunchCooperativeKernel((const void *)k_large_tree, dim3(unsigned(want < ctas ? want : ctas)),
                                    dim3(kLgTreeThreads), params, 0, s);
    if (e != cudaSuccess) return e;
    k_large_runs<<<unsigned((n - 1 + kLgRun - 1) / kLgRun), 1024, 0, s>>>(A);
    k_large_merge<<<unsigned((n - 1 + 7) / 8), 256, 0, s>>>(A);
    return cudaGetLastError();
}

// The rest, after the reduction of the tree's edges (its pivots in kill_key,
// kill_val).
cudaError_t launch_large_bars(void *ws, const Layout &L, int64_t n, ph0_bar *bars, ph0_inf_bar *inf, bool prefix,
                              cudaStream_t s, cudaEvent_t after_counts) {
    size_t zero, zero_end;
    const LgArgs A = large_args(ws, L, bars, inf, 0, prefix, zero, zero_end);
    const int ctas = 2 * sm_count();
    const int hot = n - 1 < kLgHot ? int(n - 1) : kLgHot;
    const int64_t counts = (L.m + kLgCountThreads * 16 - 1) / (kLgCountThreads * 16);
    auto count = [&](auto kernel) {
        const cudaError_t r = smem_limit<size_t(kLgHot) * 12>(kernel);
        if (r != cudaSuccess) return r;
        kernel<<<unsigned(counts < ctas ? counts : ctas), kLgCountThreads, size_t(hot) * 12, s>>>(A);
        return cudaGetLastError();
    };
    cudaError_t e = prefix ? count(k_large_count<true>) : count(k_large_count<false>);
    if (e != cudaSuccess) return e;
    if (prefix) {
        k_large_places<<<1, 1024, 0, s>>>(A);
        if ((e = launch_parts(A, s)) != cudaSuccess) return e;
    }
    if (A.nsub > 1) {
        e = smem_limit<move_smem(1)>(k_large_move<1>);
        if (e != cudaSuccess) return e;
        k_large_sub<<<kLgParts * kLgSubCtas, kLgThreads, 0, s>>>(A);
        k_large_move<1><<<kLgParts * kLgSubCtas, kLgThreads, move_smem(1), s>>>(A);
    }
    e = smem_limit<size_t(kLgWords) * 4>(k_large_repeats);
    if (e != cudaSuccess) return e;
    k_large_repeats<<<unsigned(ctas), kLgRepThreads, size_t(kLgWords) * 4, s>>>(A);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (after_counts && (e = cudaEventRecord(after_counts, s)) != cudaSuccess) return e;
    k_large_emit<<<unsigned((n - 1 + 1023) / 1024), 1024, 0, s>>>(A);
    return cudaGetLastError();
}

}  // namespace ph0
