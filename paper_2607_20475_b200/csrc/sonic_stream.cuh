// Streaming kernel and merge kernel.
//
// The streaming kernel reads every logit of the rows of the streaming classes
// exactly once, applies the logit-processing prologue, and reduces each
// 8192-element tile either to an argmax (greedy rows) or to the complete set of
// elements at or above a tile cutoff (top-k rows), written to the tile's own
// slot of the workspace.  The merge kernel, a programmatic dependent launch with
// one CTA per row, combines a row's tile records and finishes the row (global
// top-k, truncation epilogue, token selection) or flags it for the exact kernel.
// The two correspond to the paper's Algorithms "Stage 1: Tile-Local Reduction
// Kernel" and "Stage 2: Cross-Tile Merge and Selection Kernel"; the selection
// itself is ours.
//
// (Calls with a grammar bitmask: sonic_mask.cuh.)  Structure of the streaming kernel: persistent CTAs (three per SM), each a
// producer warp plus eight consumer warps.  The producer takes tiles from a work
// queue, resolves each tile's row configuration and issues one bulk-TMA copy
// (cp.async.bulk, completion on an mbarrier) of the tile's logits into a ring of
// shared-memory stages, ahead of the consumers, so HBM requests stay in flight
// while the consumers compute.  Two builds: calls without sparse lists (histories,
// biases) carry no list code, which spares 80 to 100 bytes of spills per thread (with
// hardly any L1 left beside the ring they go to L2), and in bf16 the room of the
// fp32 tile that lists patch holds two more stages.  Measured (us per call): 128
// fp32 rows of 200003, k = 4096, 77.6 -> 68.4; 256 fp32 rows of 262144, k = 64,
// 59.6 -> 57.9 (4.6 TB/s); 160 fp32 verification rows of 131072 93.1 -> 91.3; 256
// bf16 rows of 262144, top-k 50, 57.9 -> 56.5.  Every mbarrier wait is bounded:
// on expiry the kernel records an error in the workspace header and returns.
//
// Exactness: a tile's cutoff t is a minimum of group maxima (of the G groups of
// one warp tile, or of all 8 G groups of the tile), so the tile holds elements
// >= t, and it emits EVERY finite element >= t.  With T the largest cutoff of
// the row, the emitted elements >= T are exactly the row's elements >= T.  If
// there are at least k of them the row's top-k is their top-k; otherwise the row
// is handed to the exact kernel.
#pragma once
#include "sonic_common.cuh"
#include "sonic_dense.cuh"

namespace sonic {

template <int DT> struct VecTraits;
template <> struct VecTraits<0> { static constexpr int VEC = 4, NV = 8, NSTAGE = 2, ELT = 4; };
template <> struct VecTraits<1> { static constexpr int VEC = 8, NV = 4, NSTAGE = 2, ELT = 2; };

constexpr int STREAM_CTA_THREADS = STREAM_THREADS + 32;      // eight consumer warps + the producer warp
#ifndef SONIC_WAIT_LIMIT
#define SONIC_WAIT_LIMIT (1u << 22)
#endif
constexpr unsigned int WAIT_LIMIT = SONIC_WAIT_LIMIT;        // try_wait rounds before a wait gives up (a test-only build shortens it)

// ---------------------------------------------------------------- mbarrier / bulk-copy primitives
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Announces `bytes` of a copy to the barrier's current phase without arriving on it (the arrival follows later).
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned int bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bounded wait for the phase with the given parity; false if it did not complete in time.
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned int parity) {
    const uint32_t addr = smem_u32(bar);
    for (unsigned int it = 0; it < WAIT_LIMIT; ++it) {
        unsigned int done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(addr), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
// One bulk copy global -> this CTA's shared memory; bytes and both addresses are multiples of 16.  The logits are
// read once, so the copy carries an evict-first L2 policy: the stream does not push the workspace (candidates,
// tile records) and the kernels' code out of L2.
__device__ __forceinline__ unsigned long long l2_evict_first_policy() {
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned int bytes, unsigned long long *bar,
                                          unsigned long long policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Element index of register slot s of a lane.
template <int DT>
__device__ __forceinline__ int slot_index(int wbase, int lane, int s) {
    constexpr int VEC = VecTraits<DT>::VEC;
    return wbase + (s / VEC) * 32 * VEC + lane * VEC + (s % VEC);
}

template <int THREADS>
struct MergeShared {
    int count;
    int tcnt[MAX_TILES + 1];                   // exclusive prefix of the tiles' candidate counts
    unsigned int tkey;
    int n_p, n_m, pick;
    int found;
    int wsum[THREADS / 32], wsum2[THREADS / 32];       // a block scan's warp totals
    int bracket[4];                            // the counting bins' answer: bin, count above it, count with it
    alignas(16) double scratch[THREADS];      // also read as int4
};


constexpr int MERGE_BUCKETS = 4096;           // buckets of the sort of larger candidate sets (16 KB behind the keys)
constexpr int RANK_SORT_MAX = 512;            // at most this many candidates: sort by rank counting
constexpr int WARP_EPILOGUE_MAX = 128;        // at most this many survivors of TopK: one warp finishes the row
struct WarpSync { __device__ __forceinline__ void operator()() const { __syncwarp(); } };

template <int NT, typename Sync, typename SH>
__device__ void merge_epilogue(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells);
template <int THREADS, typename SH>
__device__ void merge_epilogue_small(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells);

// Counting bins of the candidates of a large-k row: MERGE_GBINS bins of 2^MERGE_GSHIFT keys above the proven threshold
// (one binade of fp32 keys; whatever lies higher shares the top bin), kept in the scratch words of MergeShared.
constexpr int MERGE_GBINS = 2 * MERGE_THREADS, MERGE_GSHIFT = 13;

// The bin in which the count from the top reaches `need`, the count above it and the count with it (bin < 0: the
// bins hold fewer than `need`); thread t owns bins GBINS-1-2t and GBINS-2-2t.  Two barriers.
template <int THREADS>
__device__ __forceinline__ void merge_bins_find(MergeShared<THREADS> &sh, int tid, int need, int &bin, int &above, int &with) {
    constexpr int GBINS = MERGE_GBINS, BPT = GBINS / THREADS;
    static_assert(GBINS * 4 <= THREADS * 8, "the counting bins live in the scratch words");
    const int *ghist = reinterpret_cast<const int *>(sh.scratch);
    const int lane_ = tid & 31, warp_ = tid >> 5;
    int v[BPT], sum = 0;
#pragma unroll
    for (int j = 0; j < BPT; ++j) { v[j] = ghist[GBINS - 1 - (tid * BPT + j)]; sum += v[j]; }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane_ >= off) incl += o;
    }
    if (lane_ == 31) sh.wsum[warp_] = incl;
    if (tid == 0) sh.bracket[0] = -1;
    __syncthreads();
    int pre = incl - sum;
    for (int w = 0; w < warp_; ++w) pre += sh.wsum[w];
    if (pre < need && pre + sum >= need) {
        int run = pre;
#pragma unroll
        for (int j = 0; j < BPT; ++j) {
            if (run < need && run + v[j] >= need) { sh.bracket[0] = GBINS - 1 - (tid * BPT + j); sh.bracket[1] = run; sh.bracket[2] = run + v[j]; }
            run += v[j];
        }
    }
    __syncthreads();
    bin = sh.bracket[0]; above = sh.bracket[1]; with = sh.bracket[2];
    __syncthreads();
}

// Sorts up to 256 distinct 64-bit keys (zeros pad) in descending order, one warp, eight keys per lane.
__device__ __noinline__ void warp_sort_256(unsigned long long *a, int cnt, int lane) {
    unsigned long long k[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { const int e = j * 32 + lane; k[j] = (e < cnt) ? a[e] : 0ull; }
#pragma unroll
    for (int size = 2; size <= 256; size <<= 1) {
#pragma unroll
        for (int d = size >> 1; d > 0; d >>= 1) {
            if (d >= 32) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int o = j ^ (d >> 5);
                    if (o > j) {
                        const bool desc = (((j * 32) & size) == 0);
                        if ((k[j] < k[o]) == desc) { const unsigned long long t = k[j]; k[j] = k[o]; k[o] = t; }
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, k[j], d);
                    const int e = j * 32 + lane;
                    const bool take_max = (((e & size) == 0) == ((e & d) == 0));
                    k[j] = ((k[j] > o) == take_max) ? k[j] : o;
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) { const int e = j * 32 + lane; if (e < cnt) a[e] = k[j]; }
}

// Descending sort of n0 distinct 64-bit keys in buf (RANK_SORT_MAX < n0 <= MERGE_CAP), of which the first n are wanted:
// 4096 buckets by distance from the smallest, one counting pass, one scan, one scatter;
// what shares a bucket (a handful of keys for smooth values) is ranked by counting, a crowded bucket (ties of a
// low-precision value) is sorted by a warp.  Bound by barriers and shared-memory latency: 128 fp32 rows of 200003 with k = 4096
// 107 -> 75 us a call, 64 bf16 rows of 131072 with k = 1000 on an eighth of them 58.8 -> 55.5.  About 35 instructions per key in eight barrier-separated steps, where a
// bitonic sort of 4096 keys goes through 78 compare-exchange steps, 21 of them behind block barriers.  A bucket beyond
// 256 keys that the wanted ones reach into falls back to the bitonic sort.
template <int THREADS>
__device__ __forceinline__ void merge_bucket_sort(unsigned long long *buf, unsigned int *bins, const int n0, const int n, MergeShared<THREADS> &sh, int tid) {
    constexpr int NB = MERGE_BUCKETS, ITEMS = MERGE_CAP / THREADS, BPT = NB / THREADS, FEW = 64, WARP_MAX = 256;
    const int lane = tid & 31, warp = tid >> 5;
    unsigned long long key[ITEMS];
    uint32_t mx = 0u, mn = 0xFFFFFFFFu;
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        const int i = u * THREADS + tid;
        key[u] = (i < n0) ? buf[i] : 0ull;
        if (i < n0) { mx = max(mx, (uint32_t)(key[u] >> 32)); mn = min(mn, (uint32_t)(key[u] >> 32)); }
    }
    for (int i = tid; i < NB; i += THREADS) bins[i] = 0u;
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    if (lane == 0) { sh.wsum[warp] = (int)mx; sh.wsum2[warp] = (int)mn; }
    __syncthreads();
    if (tid == 0) { sh.count = 0; sh.found = 0; }                  // (behind the barrier: until then a warp may still be reading the caller's count)
    mx = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)sh.wsum[lane & (THREADS / 32 - 1)]);
    mn = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)sh.wsum2[lane & (THREADS / 32 - 1)]);
    // Bucket: 256 per octave of the distance above the smallest key.  The upper tail of a smooth distribution is dense at
    // its lower end and thins out exponentially, so an octave holds at most a quarter of the keys (8 per bucket of 8192),
    // and an outlier costs a few octaves of 16 instead of squashing everything else into a few buckets.
    const float y0 = fmaxf(unkey(mn), -1.7e38f);
    auto dist = [=](uint32_t key) -> int { return __float_as_int(fmaxf(fminf(unkey(key), 1.7e38f) - y0, 0.0f)) >> 15; };
    const int top = dist(mx);
    auto bucket = [=](unsigned long long k) -> int { return min(NB - 1, top - dist((uint32_t)(k >> 32))); };       // (monotone)
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        if (u * THREADS + tid < n0) atomicAdd(&bins[bucket(key[u])], 1u);
    }
    __syncthreads();
    // exclusive scan of the buckets, BPT consecutive ones per thread
    {
        unsigned int v[BPT], sum = 0u;
#pragma unroll
        for (int j = 0; j < BPT; j += 4) {
            const uint4 q = *reinterpret_cast<const uint4 *>(bins + tid * BPT + j);
            v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
            sum += (q.x + q.y) + (q.z + q.w);
        }
        unsigned int incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) { const unsigned int o = __shfl_up_sync(0xFFFFFFFFu, incl, off); if (lane >= off) incl += o; }
        __syncthreads();                                            // (every thread has read the warps' extremes)
        if (lane == 31) sh.wsum[warp] = (int)incl;
        __syncthreads();
        unsigned int run = incl - sum;
        for (int w = 0; w < warp; ++w) run += (unsigned int)sh.wsum[w];
#pragma unroll
        for (int j = 0; j < BPT; ++j) {
            if (v[j] > (unsigned int)FEW && run < (unsigned int)n) {
                if (v[j] > (unsigned int)WARP_MAX) sh.found = 1;
                else {
                    const int at = atomicAdd(&sh.count, 1);
                    reinterpret_cast<unsigned int *>(sh.scratch)[at] = run | (v[j] << 16);       // (more than MERGE_CAP / FEW never exist)
                }
            }
            if (run < (unsigned int)n && (unsigned int)n <= run + v[j]) sh.bracket[0] = (int)(run + v[j]);      // where the last wanted bucket ends
            const unsigned int t = v[j]; v[j] = run; run += t;
        }
#pragma unroll
        for (int j = 0; j < BPT; j += 4) *reinterpret_cast<uint4 *>(bins + tid * BPT + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        if (u * THREADS + tid < n0) buf[atomicAdd(&bins[bucket(key[u])], 1u)] = key[u];
    }
    __syncthreads();
    if (sh.found) {                                                 // the wanted buckets are in front now: the others are left out
        const int nw = sh.bracket[0], m = next_pow2(nw);
        for (int i = nw + tid; i < m; i += THREADS) buf[i] = 0ull;
        __syncthreads();
        bitonic_sort_desc_cta<THREADS>(buf, m, tid);
        return;
    }
    // bins[b] is now where bucket b ends: rank inside the bucket, for the wanted ones
    int to[ITEMS];
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        const int i = u * THREADS + tid;
        to[u] = -1;
        if (i < n0) {
            const unsigned long long k = buf[i];
            const int b = bucket(k), first = b ? (int)bins[b - 1] : 0, cnt = (int)bins[b] - first;
            if (first < n && cnt > 1 && cnt <= FEW) {
                int r = first;
#pragma unroll 4
                for (int t = first; t < first + cnt; ++t) r += (buf[t] > k) ? 1 : 0;
                to[u] = r;
            }
            key[u] = k;
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        if (to[u] >= 0) buf[to[u]] = key[u];
    }
    const int crowded = sh.count;
    for (int q = warp; q < crowded; q += THREADS / 32) {
        const unsigned int e = reinterpret_cast<const unsigned int *>(sh.scratch)[q];
        warp_sort_256(buf + (e & 0xFFFFu), (int)(e >> 16), lane);
    }
    __syncthreads();
}

// The rest of a top-k row once its candidates are in buf[0, Pn) (at most MERGE_CAP, distinct, in no order): the n best of
// them, sorted, then the outputs of sonic_topk or the truncation epilogue and the token.  bins: MERGE_BUCKETS words.
template <int THREADS, typename Sync>
__device__ void merge_finish(const KParams &P, const RowCfg &c, int row, unsigned long long *buf, unsigned int *bins, const int Pn, const int n,
                             MergeShared<THREADS> &sh, int tid, uint2 cells);

constexpr int SMALL_MAX = 128;                // candidates the short finish takes
// A top-k row whose at most SMALL_MAX candidates are in src (divide: before the temperature): everything that is left of it,
// with three block barriers.  Four threads per candidate count how many rank above it and how many have a smaller index;
// the weights (fp64) go to both orders; one warp does the cuts and the draw.
// list: 4 * SMALL_MAX words.
__device__ __forceinline__ void finish_small(const KParams &P, const RowCfg &c, int row, const unsigned long long *src, bool divide, int n,
                                             unsigned long long *list, int tid, uint2 cells, int draft, float q_draft) {
    unsigned long long *cand = list;                                // [SMALL_MAX] (value key after the temperature, ~index)
    unsigned long long *byrank = cand + SMALL_MAX;                  // [SMALL_MAX] the same in ranking order
    double *wr = reinterpret_cast<double *>(cand + 2 * SMALL_MAX);   // weights in ranking order
    unsigned long long *byidx = cand + 3 * SMALL_MAX;               // rank of the j-th candidate in index order
    const int lane = tid & 31;
    if (tid < SMALL_MAX) {
        unsigned long long v = (tid < n) ? src[tid] : 0ull;
        if (v && divide) v = ((unsigned long long)okey(div_tau(unkey((uint32_t)(v >> 32)), c.tau)) << 32) | (uint32_t)v;
        cand[tid] = v;
        byrank[tid] = 0ull; wr[tid] = 0.0; byidx[tid] = 0xFFFFull;
    }
    __syncthreads();
    {
        const int j = tid >> 2, part = tid & 3;
        const unsigned long long mine = cand[j];
        int rv = 0, ri = 0;
        uint32_t top = 0u;
#pragma unroll 4
        for (int u = part; u < (n + 1) / 2; u += 4) {              // (the four parts read 64 consecutive bytes)
            const ulonglong2 o = reinterpret_cast<const ulonglong2 *>(cand)[u];
            rv += (o.x > mine ? 1 : 0) + (o.y > mine ? 1 : 0);
            ri += ((uint32_t)o.x > (uint32_t)mine ? 1 : 0) + ((uint32_t)o.y > (uint32_t)mine ? 1 : 0);
            top = max(top, max((uint32_t)(o.x >> 32), (uint32_t)(o.y >> 32)));
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
            rv += __shfl_xor_sync(0xFFFFFFFFu, rv, off);
            ri += __shfl_xor_sync(0xFFFFFFFFu, ri, off);
            top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, off));
        }
        if (mine && part == 0) {
            byrank[rv] = mine;
            if (P.op == OP_TOPK) {
                if (rv < P.ktop) {
                    P.out_vals[(size_t)row * P.ktop + rv] = unkey((uint32_t)(mine >> 32));
                    P.out_idx[(size_t)row * P.ktop + rv] = (int)(~(uint32_t)mine);
                }
            } else {
                wr[rv] = exp((double)unkey((uint32_t)(mine >> 32)) - (double)unkey(top));
                byidx[ri] = (unsigned long long)rv;
            }
        }
    }
    if (P.op == OP_TOPK) return;
    __syncthreads();
    if (tid >= 32) return;
    // the ranking: four consecutive positions per lane
    const double M = (double)unkey((uint32_t)(byrank[0] >> 32));
    const int m = min(n, c.k);
    double cs[4], run = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) { const int j = lane * 4 + u; run += (j < m) ? wr[j] : 0.0; cs[u] = run; }
    double incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += up; }
    const double Z = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - run;
    auto first_hit = [&](int at) -> int {                           // first position from every lane's first hit among its four (4: none)
        const unsigned int b = __ballot_sync(0xFFFFFFFFu, at < 4);
        if (!b) return -1;
        const int l = __ffs(b) - 1;
        return l * 4 + __shfl_sync(0xFFFFFFFFu, at, l);
    };
    int keep = m;
    if (c.z & M_TOP_P) {
        const double target = (double)c.p * Z;
        int at = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u) if (lane * 4 + u < m && cs[u] + excl >= target) at = u;
        const int j = first_hit(at);
        if (j >= 0) keep = min(keep, j + 1);
    }
    if (c.z & M_MIN_P) {
        const double thr = M + log((double)c.theta);
        int at = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u) { const int j = lane * 4 + u; if (j < m && !((double)unkey((uint32_t)(byrank[j] >> 32)) >= thr)) at = u; }
        const int j = first_hit(at);
        if (j >= 0) keep = min(keep, j);
    }
    double W = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) if (((keep - 1) & 3) == u) W = cs[u] + excl;
    W = __shfl_sync(0xFFFFFFFFu, W, (keep - 1) >> 2);
    // index order: what is cut off weighs nothing
    int rk[4];
    double r4[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { rk[u] = (int)byidx[lane * 4 + u]; r4[u] = (rk[u] < keep) ? wr[rk[u] & (SMALL_MAX - 1)] : 0.0; }
    uint32_t flags = 0u;
    float p_draft = 0.0f;
    auto scan4 = [&]() -> double {                                  // cs: inclusive sums in index order; the total
        double r = 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) { r += r4[u]; cs[u] = r; }
        double in = r;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const double up = __shfl_up_sync(0xFFFFFFFFu, in, o); if (lane >= o) in += up; }
#pragma unroll
        for (int u = 0; u < 4; ++u) cs[u] += in - r;
        return __shfl_sync(0xFFFFFFFFu, in, 31);
    };
    double total = -1.0;
    if (P.op == OP_VERIFY && c.l < P.K) {
        double pd = 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) if (rk[u] < keep && draft >= 0 && (int)(~(uint32_t)byrank[rk[u] & (SMALL_MAX - 1)]) == draft) pd = r4[u];
        const unsigned int b = __ballot_sync(0xFFFFFFFFu, pd > 0.0);
        const double Pd = b ? __shfl_sync(0xFFFFFFFFu, pd, __ffs(b) - 1) / W : 0.0;
        p_draft = (float)Pd;
        if (Pd > 0.0 && cell_to_u(cells.x) * (double)q_draft <= Pd) flags |= F_ACCEPT;
        else {                                                      // residual max(0, p - q) over the support
            const float *q = P.draft_probs + ((size_t)c.b * P.K + c.l) * (size_t)P.V;
            float q4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) q4[u] = (rk[u] < keep) ? __ldg(q + (int)(~(uint32_t)byrank[rk[u] & (SMALL_MAX - 1)])) : 0.0f;
            double keep4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { keep4[u] = r4[u]; const double r = (rk[u] < keep) ? r4[u] / W - (double)q4[u] : 0.0; r4[u] = r > 0.0 ? r : 0.0; }
            total = scan4();
            if (!(total > 0.0)) {
#pragma unroll
                for (int u = 0; u < 4; ++u) r4[u] = keep4[u];
                total = -1.0;
            }
        }
    }
    if (total < 0.0) total = scan4();
    const double target = cell_to_u(cells.y) * total;
    int at = 4, lastpos = -1;
#pragma unroll
    for (int u = 3; u >= 0; --u) if (rk[u] < keep && cs[u] > target && r4[u] > 0.0) at = u;
#pragma unroll
    for (int u = 0; u < 4; ++u) if (rk[u] < keep) lastpos = u;
    int j = first_hit(at);
    if (j < 0) {                                                    // (rounding: the last survivor in index order)
        const unsigned int b = __ballot_sync(0xFFFFFFFFu, lastpos >= 0);
        const int l = 31 - __clz(b);
        j = l * 4 + __shfl_sync(0xFFFFFFFFu, lastpos, l);
    }
    if (lane == 0) {
        const int r = (int)byidx[j];
        emit_row(P, c, row, (int)(~(uint32_t)byrank[r]), (float)(wr[r] / W), flags, keep, p_draft);
    }
}

// The k-th largest of the n maxima in gmax (32-bit keys, n <= THREADS, zeros behind them up to the next multiple of four):
// every maximum counts those above it (up to four threads share one), the smallest with fewer than k above is the answer.
// red: THREADS / 32 words.  Whole CTA, one block barrier.
template <int THREADS>
__device__ __forceinline__ uint32_t kth_max(const unsigned int *gmax, unsigned int *red, int n, int k, int tid) {
    const int lg = n <= THREADS / 4 ? 2 : (n <= THREADS / 2 ? 1 : 0), part = tid & ((1 << lg) - 1);
    const uint32_t mine = ((tid >> lg) < n) ? gmax[tid >> lg] : 0u;
    int above = 0;
#pragma unroll 4
    for (int i = part; i < (n + 3) / 4; i += 1 << lg) {
        const uint4 o = reinterpret_cast<const uint4 *>(gmax)[i];
        above += (o.x > mine ? 1 : 0) + (o.y > mine ? 1 : 0) + (o.z > mine ? 1 : 0) + (o.w > mine ? 1 : 0);
    }
    if (lg > 0) above += __shfl_xor_sync(0xFFFFFFFFu, above, 1);
    if (lg > 1) above += __shfl_xor_sync(0xFFFFFFFFu, above, 2);
    const uint32_t t = __reduce_min_sync(0xFFFFFFFFu, (above < k && (tid >> lg) < n) ? mine : 0xFFFFFFFFu);
    if ((tid & 31) == 0) red[tid >> 5] = t;
    __syncthreads();
    return __reduce_min_sync(0xFFFFFFFFu, red[tid & (THREADS / 32 - 1)]);
}

// Row merge for top-k class rows (one CTA per row).  buf is MERGE_CAP 64-bit
// words of shared memory.  Returns false if the candidates cannot prove the
// row's answer.
template <int THREADS, typename Sync>
__device__ bool merge_topk_row(const KParams &P, const RowCfg &c, int row, int tiles,
                               unsigned long long *buf, unsigned int *bins, MergeShared<THREADS> &sh, int tid, uint2 cells) {
    Sync csync;
    const int cap_t = (int)(P.cand_stride / (unsigned)tiles);
    const TileRec *rec = P.tiles + (size_t)row * MAX_TILES;
    // tile records: the first warp takes one tile per lane; prefix of the counts and the largest cutoff by shuffles
    static_assert(MAX_TILES <= 32, "one tile record per lane of the first warp");
    if (tid < 32) {
        unsigned int cnt = 0u, tk = 0u;
        if (tid < tiles) {
            cnt = __ldcg(&rec[tid].cnt);
            tk = __ldcg(&rec[tid].tkey);
        }
        const bool over = __any_sync(0xFFFFFFFFu, cnt > (unsigned int)cap_t);     // a tile overflowed its slot
        int incl = (int)cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (tid >= off) incl += o;
        }
        tk = __reduce_max_sync(0xFFFFFFFFu, tk);
        sh.tcnt[tid + 1] = incl;                                   // lanes past the last tile repeat the total
        if (tid == 0) { sh.tcnt[0] = 0; sh.count = 0; sh.tkey = tk; sh.found = over ? 1 : 0; }
    }
    csync();
    if (sh.found) return false;
    const unsigned int tkey = sh.tkey;
    const bool complete = (tkey == KEY_NEG_INF);
    const bool strict = c.temp && !complete;            // keys are compared after the temperature division
    const uint32_t tykey = c.temp ? okey(div_tau(unkey(tkey), c.tau)) : tkey;
    const int total = sh.tcnt[tiles];
    // candidates are fetched eight per lane at a time (independent loads), then filtered and packed
    constexpr int GB = 8;
    // proven candidate -> its key after the temperature division (0 if it is not proven)
    auto proven_key = [&](unsigned long long cd, int j) -> unsigned long long {
        const uint32_t zk = (uint32_t)(cd >> 32);
        uint32_t yk = zk;
        if (c.temp) yk = okey(div_tau(unkey(zk), c.tau));
        const bool keep = (j < total) && (zk >= tkey) && !(strict && yk <= tykey);
        return keep ? (((unsigned long long)yk << 32) | (uint32_t)cd) : 0ull;
    };
    unsigned long long floor_key = 1ull;           // keys below it are left out (1: every proven candidate)
    // Large k: while the candidates are gathered they are also counted in 1024 bins of 8192 keys above the proven
    // threshold (one binade of fp32 keys; whatever lies higher shares the top bin).  The bin in which the count from
    // the top reaches k then brackets the k-th key without a pass of its own (GBINS ints in sh.scratch).
    constexpr int GBINS = MERGE_GBINS, GSHIFT = MERGE_GSHIFT;
    int *ghist = reinterpret_cast<int *>(sh.scratch);
    const uint32_t gbase = c.temp ? tykey : tkey;
    const bool use_bins = !complete && total > MERGE_CAP;
    auto gbin = [&](unsigned long long key) -> int {
        const uint32_t d = ((uint32_t)(key >> 32) - gbase) >> GSHIFT;
        return (int)min(d, (uint32_t)(GBINS - 1));
    };
    for (int attempt = 0; attempt < 2; ++attempt) {
        unsigned long long kmax = 0ull;
        if (use_bins) {
            for (int i = tid; i < GBINS; i += THREADS) ghist[i] = 0;
            csync();
        }
        // tile-major: a warp takes tiles w and w + NW together, its lanes the slots' entries (no search for the
        // tile of an entry; the loads of both tiles are in flight at once)
        constexpr int NW = THREADS / 32, HB = GB / 2;
        const int lane = tid & 31, warp = tid >> 5;
        for (int ta = warp; ta < tiles; ta += 2 * NW) {
            const int tb = ta + NW;
            const int na = sh.tcnt[ta + 1] - sh.tcnt[ta];
            const int nb = (tb < tiles) ? sh.tcnt[tb + 1] - sh.tcnt[tb] : 0;
            const bool single = tb >= tiles;            // no second tile for this warp: all load slots go to the first
            const unsigned long long *pa = P.cand + (size_t)row * P.cand_stride + (size_t)ta * cap_t;
            const unsigned long long *pb = P.cand + (size_t)row * P.cand_stride + (size_t)tb * cap_t;
            if (max(na, nb) <= 32) {
                // small k: a tile brings a dozen candidates, one per lane
                const unsigned long long ca = (lane < na) ? __ldcg(pa + lane) : 0ull;
                const unsigned long long cb = (lane < nb) ? __ldcg(pb + lane) : 0ull;
                const unsigned long long oa = proven_key(ca, lane < na ? 0 : total);
                const unsigned long long ob = proven_key(cb, lane < nb ? 0 : total);
                kmax = max(kmax, max(oa, ob));
                const unsigned int ma = __ballot_sync(0xFFFFFFFFu, oa >= floor_key);
                const unsigned int mb = __ballot_sync(0xFFFFFFFFu, ob >= floor_key);
                const int nk = __popc(ma) + __popc(mb);
                int base = 0;
                if (lane == 0 && nk) base = atomicAdd(&sh.count, nk);
                base = __shfl_sync(0xFFFFFFFFu, base, 0);
                const unsigned int below = (1u << lane) - 1u;
                if (oa >= floor_key) { const int pos = base + __popc(ma & below); if (pos < MERGE_CAP) buf[pos] = oa; if (use_bins) atomicAdd(&ghist[gbin(oa)], 1); }
                if (ob >= floor_key) { const int pos = base + __popc(ma) + __popc(mb & below); if (pos < MERGE_CAP) buf[pos] = ob; if (use_bins) atomicAdd(&ghist[gbin(ob)], 1); }
                continue;
            }
            for (int j0 = 0; j0 < max(na, nb); j0 += (single ? 32 * GB : 32 * HB)) {
                unsigned long long cd[GB];
#pragma unroll
                for (int u = 0; u < HB; ++u) {
                    const int j = j0 + u * 32 + lane, j2 = j + 32 * HB;
                    cd[u] = (j < na) ? __ldcg(pa + j) : 0ull;
                    cd[HB + u] = single ? ((j2 < na) ? __ldcg(pa + j2) : 0ull) : ((j < nb) ? __ldcg(pb + j) : 0ull);
                }
                // filter all of the batch, then reserve room with ONE shared-memory atomic per warp and batch
                // (every warp adds to the same counter: per-candidate or per-slot atomics would queue up there)
                unsigned long long out[GB];
                unsigned int km[GB];
                int nkeep = 0;
#pragma unroll
                for (int u = 0; u < GB; ++u) {
                    const int j = j0 + (u % HB) * 32 + lane + ((single && u >= HB) ? 32 * HB : 0);
                    const bool valid = (u < HB || single) ? (j < na) : (j < nb);
                    out[u] = proven_key(cd[u], valid ? 0 : total);
                    kmax = max(kmax, out[u]);
                    km[u] = __ballot_sync(0xFFFFFFFFu, out[u] >= floor_key);
                    nkeep += __popc(km[u]);
                }
                int base = 0;
                if (lane == 0 && nkeep) base = atomicAdd(&sh.count, nkeep);
                base = __shfl_sync(0xFFFFFFFFu, base, 0);
#pragma unroll
                for (int u = 0; u < GB; ++u) {
                    if (out[u] >= floor_key) {
                        const int pos = base + __popc(km[u] & ((1u << lane) - 1u));
                        if (pos < MERGE_CAP) buf[pos] = out[u];
                        if (use_bins) atomicAdd(&ghist[gbin(out[u])], 1);
                    }
                    base += __popc(km[u]);
                }
            }
        }
        csync();
        if (attempt == 1 || sh.count <= MERGE_CAP || sh.count < c.k) break;
        // More proven candidates than the buffer holds (large k): a key floor that keeps between k and MERGE_CAP of
        // them, then pack again.  The bins counted during the pass usually give it at once ...
        if (use_bins) {
            int b, above, with;
            merge_bins_find<THREADS>(sh, tid, c.k, b, above, with);
            if (b >= 0 && with <= MERGE_CAP) {
                floor_key = max(1ull, ((unsigned long long)gbase + ((unsigned long long)b << GSHIFT)) << 32);
                if (tid == 0) sh.count = 0;
                csync();
                continue;
            }
        }
        // ... otherwise a counting pass over the candidates in global memory, and an eight-way search if that leaves too many.
        unsigned long long *red = reinterpret_cast<unsigned long long *>(sh.scratch);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) kmax = max(kmax, __shfl_xor_sync(0xFFFFFFFFu, kmax, off));
        if ((tid & 31) == 0) red[tid >> 5] = kmax;
        csync();
        for (int w = 0; w < THREADS / 32; ++w) kmax = max(kmax, red[w]);
        csync();
        // every proven key is at least (cutoff key << 32): the search starts from the range the keys can span
        unsigned long long lo = max(1ull, (unsigned long long)(c.temp ? tykey : tkey) << 32), hi = kmax + 1ull;   // count(>= lo) >= k > count(>= hi) = 0
        bool bracketed = false;
        {
            // First a bracket from one counting pass: 2048 bins over the keys the proven candidates span, counted from
            // the top; the bin in which the count reaches k gives a floor that keeps at least k, and usually no more
            // than the buffer holds (the search below then has nothing left to do).
            int *hist = reinterpret_cast<int *>(buf);            // (what was packed so far is dropped: it is packed again below)
            int *redi = reinterpret_cast<int *>(sh.scratch);
            const uint32_t klo = (uint32_t)(lo >> 32), khi = (uint32_t)(kmax >> 32);
            const uint32_t span = khi - klo;
            const int shift = span < 2048u ? 0 : (32 - __clz(span)) - 11;
            for (int i = tid; i < 2048; i += THREADS) hist[i] = 0;
            csync();
            for (int ta = warp; ta < tiles; ta += 2 * NW) {
                const int tb = ta + NW;
                const int na = sh.tcnt[ta + 1] - sh.tcnt[ta];
                const int nb = (tb < tiles) ? sh.tcnt[tb + 1] - sh.tcnt[tb] : 0;
                const bool single = tb >= tiles;            // no second tile for this warp: all load slots go to the first
                const unsigned long long *pa = P.cand + (size_t)row * P.cand_stride + (size_t)ta * cap_t;
                const unsigned long long *pb = P.cand + (size_t)row * P.cand_stride + (size_t)tb * cap_t;
                for (int j0 = 0; j0 < max(na, nb); j0 += (single ? 32 * GB : 32 * HB)) {
                    unsigned long long cd[GB];
#pragma unroll
                    for (int u = 0; u < HB; ++u) {
                        const int j = j0 + u * 32 + lane, j2 = j + 32 * HB;
                        cd[u] = (j < na) ? __ldcg(pa + j) : 0ull;
                        cd[HB + u] = single ? ((j2 < na) ? __ldcg(pa + j2) : 0ull) : ((j < nb) ? __ldcg(pb + j) : 0ull);
                    }
#pragma unroll
                    for (int u = 0; u < GB; ++u) {
                        const int j = j0 + (u % HB) * 32 + lane + ((single && u >= HB) ? 32 * HB : 0);
                        const bool valid = (u < HB || single) ? (j < na) : (j < nb);
                        const unsigned long long out = proven_key(cd[u], valid ? 0 : total);
                        if (out >= lo) atomicAdd(&hist[(khi - (uint32_t)(out >> 32)) >> shift], 1);
                    }
                }
            }
            csync();
            static_assert(2048 % THREADS == 0, "bins per thread");
            constexpr int BPT = 2048 / THREADS;
            int v[BPT], s = 0;
#pragma unroll
            for (int j = 0; j < BPT; ++j) { v[j] = hist[tid * BPT + j]; s += v[j]; }
            int incl = s;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                if (lane >= off) incl += o;
            }
            if (lane == 31) redi[warp] = incl;
            if (tid == 0) redi[40] = -1;
            csync();
            int pre = incl - s;
            for (int w = 0; w < warp; ++w) pre += redi[w];
            if (pre < c.k && pre + s >= c.k) {
                int run = pre;
#pragma unroll
                for (int j = 0; j < BPT; ++j) {
                    if (run < c.k && run + v[j] >= c.k) { redi[40] = tid * BPT + j; redi[41] = run; redi[42] = run + v[j]; }
                    run += v[j];
                }
            }
            csync();
            const int b = redi[40], above = redi[41], kept = redi[42];
            csync();
            if (b >= 0) {
                // bin b holds the keys khi - ((b + 1) << shift) + 1 .. khi - (b << shift)
                const unsigned long long width = 1ull << shift;
                const unsigned long long down = (unsigned long long)(b + 1) * width - 1ull;
                const uint32_t kb = (down >= (unsigned long long)span) ? klo : khi - (uint32_t)down;
                lo = max(lo, (unsigned long long)kb << 32);                                    // count(>= lo) = kept >= k
                if (b > 0) hi = ((unsigned long long)(khi - (uint32_t)((unsigned long long)b * width) + 1u)) << 32;   // count(>= hi) = above < k
                (void)above;
                bracketed = kept <= MERGE_CAP;
            }
        }
        for (int it = 0; it < 24 && !bracketed && hi - lo > 1ull; ++it) {
            const unsigned long long step = (hi - lo) >> 3;
            unsigned long long th[7];
#pragma unroll
            for (int q = 0; q < 7; ++q) th[q] = (step > 0) ? lo + step * (q + 1) : min(hi - 1ull, lo + 1ull + q);
            int cnt[7] = {0, 0, 0, 0, 0, 0, 0};
            // one pass over the candidates, tile-major like the packing pass above
            for (int ta = warp; ta < tiles; ta += 2 * NW) {
                const int tb = ta + NW;
                const int na = sh.tcnt[ta + 1] - sh.tcnt[ta];
                const int nb = (tb < tiles) ? sh.tcnt[tb + 1] - sh.tcnt[tb] : 0;
                const bool single = tb >= tiles;            // no second tile for this warp: all load slots go to the first
                const unsigned long long *pa = P.cand + (size_t)row * P.cand_stride + (size_t)ta * cap_t;
                const unsigned long long *pb = P.cand + (size_t)row * P.cand_stride + (size_t)tb * cap_t;
                for (int j0 = 0; j0 < max(na, nb); j0 += (single ? 32 * GB : 32 * HB)) {
                    unsigned long long cd[GB];
#pragma unroll
                    for (int u = 0; u < HB; ++u) {
                        const int j = j0 + u * 32 + lane, j2 = j + 32 * HB;
                        cd[u] = (j < na) ? __ldcg(pa + j) : 0ull;
                        cd[HB + u] = single ? ((j2 < na) ? __ldcg(pa + j2) : 0ull) : ((j < nb) ? __ldcg(pb + j) : 0ull);
                    }
#pragma unroll
                    for (int u = 0; u < GB; ++u) {
                        const int j = j0 + (u % HB) * 32 + lane + ((single && u >= HB) ? 32 * HB : 0);
                        const bool valid = (u < HB || single) ? (j < na) : (j < nb);
                        const unsigned long long out = proven_key(cd[u], valid ? 0 : total);
#pragma unroll
                        for (int q = 0; q < 7; ++q) cnt[q] += (out >= th[q]) ? 1 : 0;
                    }
                }
            }
            int *redi = reinterpret_cast<int *>(sh.scratch);
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                cnt[q] = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned int)cnt[q]);
                if ((tid & 31) == 0) redi[(tid >> 5) * 8 + q] = cnt[q];
            }
            csync();
            bool done = false;
            bool fits = false;
            int tots[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
            for (int w = 0; w < THREADS / 32; ++w) {
                const int4 a4 = reinterpret_cast<const int4 *>(redi)[w * 2], b4 = reinterpret_cast<const int4 *>(redi)[w * 2 + 1];
                tots[0] += a4.x; tots[1] += a4.y; tots[2] += a4.z; tots[3] += a4.w;
                tots[4] += b4.x; tots[5] += b4.y; tots[6] += b4.z; tots[7] += b4.w;
            }
#pragma unroll
            for (int q = 6; q >= 0; --q) {                 // the highest threshold that still keeps k
                const int tot = tots[q];
                if (!done && tot >= c.k) {
                    lo = th[q];
                    if (q < 6) hi = th[q + 1];
                    done = true;
                    fits = tot <= MERGE_CAP;
                }
            }
            if (!done) hi = th[0];
            csync();
            if (fits) break;
        }
        floor_key = lo;
        if (tid == 0) sh.count = 0;
        csync();
    }
    csync();
    const int Pn = sh.count;
    if (Pn > MERGE_CAP) return false;
    int n;
    if (Pn >= c.k) n = c.k;
    else if (complete && P.op != OP_TOPK) n = Pn;
    else return false;
    merge_finish<THREADS, Sync>(P, c, row, buf, bins, Pn, n, sh, tid, cells);
    return true;
}

template <int THREADS, typename Sync>
__device__ void merge_finish(const KParams &P, const RowCfg &c, int row, unsigned long long *buf, unsigned int *bins, const int Pn, const int n,
                             MergeShared<THREADS> &sh, int tid, uint2 cells) {
    Sync csync;
    if (Pn <= RANK_SORT_MAX) {
        // few candidates, one per thread: every warp sorts its 32 keys with shuffles, then a key's rank is its
        // place in its own run plus, for every other run, the number of keys there above it (a binary search
        // in the sorted run; keys are distinct, 0 pads the last run).  Two block barriers.
        static_assert(RANK_SORT_MAX <= THREADS, "one candidate per thread");
        unsigned long long *dst = buf + MERGE_CAP / 2;
        {
            int rank;
            const unsigned long long key = rank_keys<THREADS, Sync>(buf, Pn, tid, rank);
            if (key != 0ull) dst[rank] = key;
        }
        csync();
        for (int i = tid; i < n; i += THREADS) buf[i] = dst[i];       // only the n best are used from here on
        csync();
    } else merge_bucket_sort<THREADS>(buf, bins, Pn, n, sh, tid);

    if (P.op == OP_TOPK) {
        for (int j = tid; j < n; j += THREADS) {
            unsigned long long kv = buf[j];
            P.out_vals[(size_t)row * P.ktop + j] = unkey((uint32_t)(kv >> 32));
            P.out_idx[(size_t)row * P.ktop + j] = (int)(~(uint32_t)kv);
        }
        return;
    }
    if (n == 0) {
        if (tid == 0) emit_row(P, c, row, -1, 0.0f, F_NO_TOKEN, 0, 0.0f);
        return;
    }
    // small supports are finished by one warp without block barriers
    if (n <= WARP_EPILOGUE_MAX) {
        merge_epilogue_small<THREADS>(P, c, row, n, buf, sh, tid, cells);
    } else {
        merge_epilogue<THREADS, Sync>(P, c, row, n, buf, sh, tid, cells);
    }
}

// Truncation epilogue and token selection over the n best candidates, sorted in
// buf[0, n) (TopK already applied): TopP, MinP, index-order CDF, Philox draw,
// and for verification rows the accept test and the residual.  Three parts:
// the front (weights, cumulative sums, TopP / MinP: linear work), the index
// order of the survivors (quadratic rank counting, or a sort), and the tail
// (linear again).  Large supports run all three on the whole CTA; small ones
// run the linear parts on one warp, without block barriers, and only the
// quadratic part on all threads.
//
// shared-memory layout after the sort (n <= KFAST_SAMPLE = MERGE_CAP / 4):
//   buf[0, n)     sorted keys (value key << 32 | ~index)
//   w             weights exp(y - M) in ranking order
//   cs            cumulative sums (ranking order), later residual / CDF in index order
//   ik            (~index << 32 | ranking position), sorted descending = index ascending
struct EpiView {
    double *w, *cs;
    unsigned long long *ik;
    __device__ explicit EpiView(unsigned long long *buf)
        : w(reinterpret_cast<double *>(buf + KFAST_SAMPLE)), cs(reinterpret_cast<double *>(buf + 2 * KFAST_SAMPLE)),
          ik(buf + 3 * KFAST_SAMPLE) {}
};

// weights of the candidates (all threads of the caller's group)
template <int NT>
__device__ __forceinline__ void epilogue_weights(int n, unsigned long long *buf, int tid) {
    EpiView v(buf);
    const double M = (double)unkey((uint32_t)(buf[0] >> 32));
    for (int j = tid; j < n; j += NT) {
        double y = (double)unkey((uint32_t)(buf[j] >> 32));
        double wj = exp(y - M);
        v.w[j] = wj; v.cs[j] = wj;
    }
}

// cumulative sums and the TopP / MinP cuts; returns the surviving prefix length (also left in sh.n_p)
template <int NT, typename Sync, typename SH>
__device__ __forceinline__ int epilogue_truncate(const RowCfg &c, int n, unsigned long long *buf, SH &sh, int tid) {
    Sync csync;
    EpiView v(buf);
    const double M = (double)unkey((uint32_t)(buf[0] >> 32));
    block_inclusive_scan<NT, Sync>(v.cs, n, sh.scratch, tid);
    const double Z = v.cs[n - 1];
    if (c.z & M_TOP_P) {
        const double target = (double)c.p * Z;
        for (int j = tid; j < n; j += NT)
            if (v.cs[j] >= target && (j == 0 || v.cs[j - 1] < target)) sh.n_p = j + 1;
    }
    if (c.z & M_MIN_P) {
        const double thr = M + log((double)c.theta);
        for (int j = tid; j < n; j += NT) {
            bool in = (double)unkey((uint32_t)(buf[j] >> 32)) >= thr;
            bool prev_in = (j == 0) || ((double)unkey((uint32_t)(buf[j - 1] >> 32)) >= thr);
            if (!in && prev_in) sh.n_m = j;
        }
    }
    csync();
    n = min(n, min(sh.n_p, sh.n_m));
    csync();
    if (tid == 0) sh.n_p = n;
    csync();
    return n;
}

// The same for one warp and n <= WARP_EPILOGUE_MAX, in registers: a lane holds four consecutive weights, the
// cumulative sums come from one shuffle scan, the cuts from votes.  Leaves the surviving prefix length in sh.n_p
// and its total weight in cs[length - 1].
template <typename SH>
__device__ __forceinline__ void epilogue_truncate_warp(const RowCfg &c, int n, unsigned long long *buf, SH &sh, int lane) {
    static_assert(WARP_EPILOGUE_MAX <= 128, "four elements per lane");
    EpiView v(buf);
    const double M = (double)unkey((uint32_t)(buf[0] >> 32));
    double cs[4];
    double run = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int j = lane * 4 + u;
        run += (j < n) ? v.w[j] : 0.0;
        cs[u] = run;
    }
    double incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += up;
    }
    const double excl = incl - run;
#pragma unroll
    for (int u = 0; u < 4; ++u) cs[u] += excl;
    const double Z = __shfl_sync(0xFFFFFFFFu, incl, 31);
    // first position (ranking order) where a cut falls, from every lane's first hit among its four (4: none)
    auto first_hit = [&](int mine) -> int {
        const unsigned int m = __ballot_sync(0xFFFFFFFFu, mine < 4);
        if (!m) return -1;
        const int l = __ffs(m) - 1;
        return l * 4 + __shfl_sync(0xFFFFFFFFu, mine, l);
    };
    int keep = n;
    if (c.z & M_TOP_P) {
        const double target = (double)c.p * Z;
        int mine = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u) if (lane * 4 + u < n && cs[u] >= target) mine = u;
        const int j = first_hit(mine);
        if (j >= 0) keep = min(keep, j + 1);
    }
    if (c.z & M_MIN_P) {
        const double thr = M + log((double)c.theta);
        int mine = 4;
#pragma unroll
        for (int u = 3; u >= 0; --u) {
            const int j = lane * 4 + u;
            if (j < n && !((double)unkey((uint32_t)(buf[j] >> 32)) >= thr)) mine = u;          // first element below the threshold
        }
        const int j = first_hit(mine);
        if (j >= 0) keep = min(keep, j);
    }
    // total weight of the survivors: the cumulative sum at position keep - 1
    double mine = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) if (((keep - 1) & 3) == u) mine = cs[u];
    const double W = __shfl_sync(0xFFFFFFFFu, mine, (keep - 1) >> 2);
    if (lane == 0) { sh.n_p = keep; v.cs[keep - 1] = W; }     // the tail reads the survivors' total weight from there
    __syncwarp();
}

// survivors in vocabulary-index order
template <int NT, typename Sync>
__device__ __forceinline__ void epilogue_index_order(int n, unsigned long long *buf, int tid) {
    Sync csync;
    EpiView v(buf);
    if (n <= RANK_SORT_MAX) {
        // few survivors: each lands at the number of survivors with a smaller index; S threads share a survivor
        const int S = min(32, max(1, NT / next_pow2(n)));
        for (int j0 = 0; j0 < n; j0 += NT / S) {
            const int j = j0 + tid / S, seg = tid % S;
            const uint32_t mine = (j < n) ? (uint32_t)buf[j] : 0xFFFFFFFFu;      // ~index: larger means smaller index
            const int tlo = (int)(((long long)n * seg) / S), thi = (int)(((long long)n * (seg + 1)) / S);
            int pos = 0;
            int t = tlo;
            for (; t + 8 <= thi; t += 8) {
                uint32_t o[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) o[u] = (uint32_t)buf[t + u];
#pragma unroll
                for (int u = 0; u < 8; ++u) pos += (o[u] > mine) ? 1 : 0;
            }
            for (; t < thi; ++t) pos += ((uint32_t)buf[t] > mine) ? 1 : 0;
            for (int off = 1; off < S; off <<= 1) pos += __shfl_xor_sync(0xFFFFFFFFu, pos, off);
            if (seg == 0 && j < n) v.ik[pos] = ((unsigned long long)mine << 32) | (unsigned long long)j;
        }
        csync();
    } else {
        const int m2 = next_pow2(n);
        for (int j = tid; j < m2; j += NT)
            v.ik[j] = (j < n) ? ((buf[j] << 32) | (unsigned long long)j) : 0ull;
        csync();
        if constexpr (NT >= 64) bitonic_sort_desc_cta<NT>(v.ik, m2, tid);
        else bitonic_sort_desc<NT, Sync>(v.ik, m2, tid);
    }
}

// draw, verification, selection and the row's outputs
template <int NT, typename Sync, typename SH>
__device__ __forceinline__ void epilogue_tail(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells) {
    Sync csync;
    constexpr int THREADS = NT;
    EpiView v(buf);
    double *w = v.w, *cs = v.cs;
    unsigned long long *ik = v.ik;
    const double W = cs[n - 1];                 // still the ranking-order cumulative sums here
    csync();
    const uint32_t a_acc = cells.x, a_draw = cells.y;      // the row's Philox cells, drawn before the wait on the streaming kernel
    const double u_draw = cell_to_u(a_draw);
    uint32_t flags = 0;
    float p_draft = 0.0f;
    bool use_residual = false;
    if (P.op == OP_VERIFY && c.l < P.K) {
        const int d = P.draft_tokens[(size_t)c.b * P.K + c.l];
        const float *q = P.draft_probs + ((size_t)c.b * P.K + c.l) * (size_t)P.V;
        if (tid == 0) sh.pick = -1;
        csync();
        for (int j = tid; j < n; j += THREADS)
            if ((int)(~(uint32_t)(ik[j] >> 32)) == d) sh.pick = j;
        csync();
        double Pd = 0.0;
        if (sh.pick >= 0) Pd = w[(uint32_t)ik[sh.pick]] / W;
        double Q = (d >= 0 && d < P.V) ? (double)__ldg(q + d) : 0.0;
        bool accept = (Pd > 0.0) && (cell_to_u(a_acc) * Q <= Pd);
        p_draft = (float)Pd;
        if (accept) flags |= F_ACCEPT;
        csync();
        if (!accept) {        // (an accepted position's own token is never read: the request moves on with the draft)
            // residual max(0, p - q) over the support, in index order
            for (int j = tid; j < n; j += THREADS) {
                int idx = (int)(~(uint32_t)(ik[j] >> 32));
                double r = w[(uint32_t)ik[j]] / W - (double)__ldg(q + idx);
                cs[j] = r > 0.0 ? r : 0.0;
            }
            csync();
            block_inclusive_scan<THREADS, Sync>(cs, n, sh.scratch, tid);
            use_residual = cs[n - 1] > 0.0;
            csync();
        }
    }
    bool picked = false;
    if constexpr (NT == 32) {
        if (!use_residual) {
            // one warp, at most 128 survivors: the index-order cumulative weights stay in registers (a lane holds
            // four consecutive positions), the drawn position comes from a vote
            double csr[4];
            double run = 0.0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = tid * 4 + u;
                run += (j < n) ? w[(uint32_t)ik[j]] : 0.0;
                csr[u] = run;
            }
            double incl = run;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (tid >= o) incl += up;
            }
            const double excl = incl - run;
            const double target = u_draw * __shfl_sync(0xFFFFFFFFu, incl, 31);
            int mine = 4;
#pragma unroll
            for (int u = 3; u >= 0; --u) if (tid * 4 + u < n && csr[u] + excl > target) mine = u;
            const unsigned int m = __ballot_sync(0xFFFFFFFFu, mine < 4);
            int j = n - 1;
            if (m) { const int l = __ffs(m) - 1; j = l * 4 + __shfl_sync(0xFFFFFFFFu, mine, l); }
            if (tid == 0) sh.pick = j;
            picked = true;
            __syncwarp();
        }
    }
    if (!picked) {
        if (!use_residual) {
            for (int j = tid; j < n; j += THREADS) cs[j] = w[(uint32_t)ik[j]];
            csync();
            block_inclusive_scan<THREADS, Sync>(cs, n, sh.scratch, tid);
        }
        const double R = cs[n - 1];
        const double target = u_draw * R;
        if (tid == 0) sh.pick = n - 1;
        csync();
        for (int j = tid; j < n; j += THREADS)
            if (cs[j] > target && (j == 0 || !(cs[j - 1] > target))) sh.pick = j;
        csync();
    }
    if (tid == 0) {
        int j = sh.pick;
        int token = (int)(~(uint32_t)(ik[j] >> 32));
        float prob = (float)(w[(uint32_t)ik[j]] / W);
        emit_row(P, c, row, token, prob, flags, n, p_draft);
    }
}


// The draw of a sampling row with a large support (more survivors than the rank counting takes): the survivors are not
// brought into index order at all.  Their weights, as 2^-40 fixed-point integers, are added up per tile, then per 256 ids
// of the tile the target falls into, then per id of that range; each level is one pass over the survivors, a scan of
// at most 256 bins and a barrier.  Integer sums: the same token in every replay; against the exact index-order CDF the
// target moves by less than n * 2^-40 of the mass.
template <int NT, typename Sync, typename SH>
__device__ void epilogue_draw_large(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells) {
    Sync csync;
    static_assert(NT >= 256, "a thread per bin");
    EpiView v(buf);
    const double *w = v.w;
    const double W = v.cs[n - 1];                              // ranking-order cumulative sums: the support's mass
    unsigned int *blo = reinterpret_cast<unsigned int *>(v.ik), *bhi = blo + 256;      // (the index keys' place: unused on this path)
    unsigned long long *red = reinterpret_cast<unsigned long long *>(sh.scratch);
    const int lane = tid & 31, warp = tid >> 5;
    auto fixed = [&](int j) -> unsigned long long { return (unsigned long long)(w[j] * 1099511627776.0); };
    unsigned int range_lo = 0u;
    unsigned long long rest = 0ull;
    const int shifts[3] = {13, 8, 0};
    const unsigned int spans[3] = {(unsigned int)MAX_TILES << 13, 8192u, 256u};
#pragma unroll
    for (int level = 0; level < 3; ++level) {
        const int shift = shifts[level];
        const unsigned int span = spans[level];
        const int nb = (int)(span >> shift);                   // 32, 32, 256
        if (tid < 256) { blo[tid] = 0u; bhi[tid] = 0u; }
        csync();
        for (int j = tid; j < n; j += NT) {
            const unsigned int idx = ~(uint32_t)buf[j];
            const unsigned int d = idx - range_lo;
            const unsigned long long q = fixed(j);
            if (d < span && q) {
                const int b = (int)(d >> shift);
                const unsigned int lo = (unsigned int)q, hi = (unsigned int)(q >> 32);
                unsigned int carry = 0u;
                if (lo) { const unsigned int old = atomicAdd(&blo[b], lo); carry = (old + lo < old) ? 1u : 0u; }
                if (hi + carry) atomicAdd(&bhi[b], hi + carry);
            }
        }
        csync();
        // scan of the bins (a thread per bin, warps in order)
        const unsigned long long mine = (tid < nb) ? (((unsigned long long)bhi[tid] << 32) + blo[tid]) : 0ull;
        unsigned long long incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) red[warp] = incl;
        if (tid == 0) sh.pick = -1;
        csync();
        unsigned long long before = 0ull, total = 0ull;
        for (int wq = 0; wq < NT / 32; ++wq) { const unsigned long long t = red[wq]; before += (wq < warp) ? t : 0ull; total += t; }
        if (level == 0) rest = draw_target(total, cells.y);     // the support's mass in fixed point, and the draw's target in it
        const unsigned long long excl = before + incl - mine;
        if (mine > 0ull && excl <= rest && rest < excl + mine) { sh.pick = tid; red[32] = excl; }
        csync();
        int b = sh.pick;
        if (b < 0) {                                           // (rest < total always; kept for safety: the last bin with mass)
            if (mine > 0ull) atomicMax(&sh.pick, tid);
            csync();
            b = sh.pick;
            if (tid == b) red[32] = excl;
            csync();
        }
        const unsigned long long excl_b = red[32];
        rest = (rest > excl_b) ? rest - excl_b : 0ull;
        range_lo += (unsigned int)b << shift;
        csync();
    }
    // the survivor with that id
    if (tid == 0) sh.pick = 0;
    csync();
    for (int j = tid; j < n; j += NT)
        if (~(uint32_t)buf[j] == range_lo) sh.pick = j;
    csync();
    if (tid == 0) {
        const int j = sh.pick;
        emit_row(P, c, row, (int)(~(uint32_t)buf[j]), (float)(w[j] / W), 0u, n, 0.0f);
    }
}

template <int NT, typename Sync, typename SH>
__device__ void merge_epilogue(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells) {
    Sync csync;
    epilogue_weights<NT>(n, buf, tid);
    if (tid == 0) { sh.n_p = n; sh.n_m = n; sh.found = 0; sh.pick = -1; }
    csync();
    n = epilogue_truncate<NT, Sync>(c, n, buf, sh, tid);
    if (P.op == OP_SAMPLE && n > RANK_SORT_MAX) {
        epilogue_draw_large<NT, Sync>(P, c, row, n, buf, sh, tid, cells);
        return;
    }
    epilogue_index_order<NT, Sync>(n, buf, tid);
    epilogue_tail<NT, Sync>(P, c, row, n, buf, sh, tid, cells);
}

// Small supports: the linear parts on warp 0 (warp-level synchronisation only), the weights and the quadratic
// index ranking on the whole CTA.  Three block barriers in all.
template <int THREADS, typename SH>
__device__ void merge_epilogue_small(const KParams &P, const RowCfg &c, int row, int n, unsigned long long *buf, SH &sh, int tid, uint2 cells) {
    epilogue_weights<THREADS>(n, buf, tid);
    if (tid == 0) { sh.n_p = n; sh.n_m = n; sh.found = 0; sh.pick = -1; }
    __syncthreads();
    if (tid < 32) epilogue_truncate_warp(c, n, buf, sh, tid);
    __syncthreads();
    n = sh.n_p;
    epilogue_index_order<THREADS, BlockSync>(n, buf, tid);
    if (tid < 32) epilogue_tail<32, WarpSync>(P, c, row, n, buf, sh, tid, cells);
}

// Smallest of a warp tile's group maxima, L lanes per group (g: the lane's own maximum, or with half-lane groups
// the smaller of its two).  In tile mode a group without a finite element counts as +inf, i.e. takes no part.
template <int L>
__device__ __forceinline__ float warp_cutoff(float g, bool tile_mode) {
#pragma unroll
    for (int off = 1; off < L; off <<= 1) g = fmaxf(g, __shfl_xor_sync(0xFFFFFFFFu, g, off));
    if (tile_mode && g == -CUDART_INF_F) g = CUDART_INF_F;
#pragma unroll
    for (int off = L; off < 32; off <<= 1) g = fminf(g, __shfl_xor_sync(0xFFFFFFFFu, g, off));
    return g;
}

// What the producer hands to the consumers with each stage.
struct StageMeta {
    RowCfg cfg;
    int row, tile;
    int skip;                                  // the row belongs to the exact kernel: nothing was loaded
    int patch;                                 // 0 none, 1 the producer filtered the lists into hits[], 2 consumers scan the lists
    int npen, nbias;                           // hits of this tile
    int hb;                                    // which hit buffer holds them
    int stop;                                  // no more tiles for this CTA (nothing else in the entry is valid)
    int bad;                                   // the producer met a list id outside [0, V)
};
struct Hit { int li; int payload; };           // element within the tile; history count, or the bias as float bits

// Stages of the ring: two tiles of fp32 take 64 KB, and so do four of bf16, or two and the fp32 tile that sparse lists patch.
template <int DT, bool LISTS> constexpr int STREAM_STAGES = (DT == 1 && !LISTS) ? 4 : 2;

template <int DT, bool LISTS>
struct StreamShared {
    static constexpr int NSTAGE = STREAM_STAGES<DT, LISTS>;
    unsigned long long full[NSTAGE];           // producer -> consumers: stage described and copy issued (one arrival + the copy's bytes)
    unsigned long long empty[NSTAGE];          // consumers -> producer: stage free (one arrival per consumer warp)
    StageMeta meta[NSTAGE];
    // per-stage scratch of the consumer warps (a fast warp may already be on the next tile, in the other stage)
    alignas(16) float tw[NSTAGE][STREAM_WARPS];
    unsigned int ncand[NSTAGE];
    unsigned long long best[NSTAGE][STREAM_WARPS];
    unsigned int kmin[NSTAGE][STREAM_WARPS], nfin[NSTAGE][STREAM_WARPS];     // dense rows
    // hit lists: one buffer more than stages, so that the producer fills the next tile's while both stages are busy
    Hit pen[LISTS ? NSTAGE + 1 : 1][LISTS ? HIT_PEN_CAP : 1];
    Hit bias[LISTS ? NSTAGE + 1 : 1][LISTS ? HIT_BIAS_CAP : 1];
};

template <int DT, bool LISTS>
__global__ void __launch_bounds__(STREAM_CTA_THREADS, 3)
sonic_stream_kernel(const KParams P, const int tiles, const int nitems, const int chunk, const int cap_t) {     // cap_t: candidate slots per tile, CAND_CAP / tiles
    constexpr int VEC = VecTraits<DT>::VEC, NV = VecTraits<DT>::NV, NSTAGE = STREAM_STAGES<DT, LISTS>;
    constexpr int ELT = VecTraits<DT>::ELT;
    constexpr int STAGE_BYTES = CTA_TILE * ELT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // layout: NSTAGE raw stages | fp32 conversion tile (bf16 with lists only) | control
    unsigned char *stages = smem_raw;
    float *conv = reinterpret_cast<float *>(smem_raw + NSTAGE * STAGE_BYTES);      // bf16 with lists only
    StreamShared<DT, LISTS> &sh = *reinterpret_cast<StreamShared<DT, LISTS> *>(smem_raw + NSTAGE * STAGE_BYTES + (DT == 1 && LISTS ? CTA_TILE * 4 : 0));
    ConsumerSync csync;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    KERNEL_T0(0);
    if (tid == 0) {
        for (int s = 0; s < NSTAGE; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], STREAM_WARPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (blockIdx.x == 0 && tid == 0) P.error[WS_FAILED_ROWS] = 0u;     // this call's count of rows the merge kernel cannot prove
    __syncthreads();
    pdl_launch_dependents();                   // the merge kernel may start launching; it waits for this grid to finish

    if (warp == STREAM_WARPS) {
        // ------------------------------------------------------------ producer warp
        // The (row, tile) items are handed out through a counter in the workspace, so CTAs that become resident
        // late (the SMs may be shared with the exact kernel) find less or no work instead of holding back a fixed
        // share.  Per tile the
        // producer (1) waits for a free stage, describes the tile and issues its bulk copy, then (2) prepares
        // the NEXT tile while the ring is busy.  On a new row that means one round of global loads (parameters
        // and sparse lists, kept in registers for the row's other tiles); on every tile, picking the list
        // entries that fall into it and writing them to a hit buffer, so that the consumers patch only what is
        // there, each warp only its own part of the tile.
        static_assert(SONIC_MAX_VOCAB <= (1 << 18), "packed history entries hold an 18-bit id");
        constexpr int HPL = FILTER_HIST / 32;      // packed history entries per lane
        struct Prep { int patch, npen, nbias; };
        RowCfg c_next;
        uint32_t packed[HPL];                      // id | count << 18; 0 = no entry
        int b_id = -1;
        float b_val = 0.0f;
        int row_patch = 0, cached_row = -1, row_bad = 0;
        auto load_row = [&](int row) {
            if (!LISTS) {
                c_next = resolve_cfg(P, row, fetch_cfg(P, row));
                cached_row = row;
                return;
            }
            const int req = (P.op == OP_VERIFY) ? row / (P.K + 1) : row;
            const int *hid = P.hist_ids ? P.hist_ids + (size_t)req * P.hist_stride : nullptr;
            const int *hct = P.hist_counts ? P.hist_counts + (size_t)req * P.hist_stride : nullptr;
            const int *bid = P.bias_ids ? P.bias_ids + (size_t)req * P.bias_stride : nullptr;
            const float *bvl = P.bias_vals ? P.bias_vals + (size_t)req * P.bias_stride : nullptr;
            // the first round of loads goes out before the first use (the lengths arrive with the parameters:
            // bound by the strides); the second half of a long history follows in a round of its own
            constexpr int HALF = HPL / 2;
            const CfgRaw raw = fetch_cfg(P, row);
            int id[HALF], ct[HALF];
#pragma unroll
            for (int u = 0; u < HALF; ++u) {
                const int t = lane + 32 * u;
                id[u] = -1; ct[u] = 0;
                if (hid && hct && t < P.hist_stride) { id[u] = __ldg(hid + t); ct[u] = __ldg(hct + t); }
            }
            int b0 = -1; float v0 = 0.0f;
            if (bid && bvl && lane < P.bias_stride) { b0 = __ldg(bid + lane); v0 = __ldg(bvl + lane); }
            c_next = resolve_cfg(P, row, raw);
            cached_row = row;
            row_patch = 0;
            row_bad = 0;
            if (c_next.cls == CLS_EXACT || !(c_next.hist_len > 0 || c_next.bias_len > 0)) return;
            row_patch = 2;
            if (c_next.hist_len > FILTER_HIST || c_next.bias_len > FILTER_BIAS) return;
            bool bad = false, big = false;
            auto pack = [&](int t, int i, int cnt) -> uint32_t {
                if (t >= c_next.hist_len) return 0u;
                if (i < 0 || i >= P.V) { bad = true; return 0u; }
                if (cnt > FILTER_COUNT_MAX) { big = true; return 0u; }
                return (cnt > 0) ? ((uint32_t)i | ((uint32_t)cnt << 18)) : 0u;
            };
#pragma unroll
            for (int u = 0; u < HALF; ++u) packed[u] = pack(lane + 32 * u, id[u], ct[u]);
#pragma unroll
            for (int u = 0; u < HALF; ++u) packed[HALF + u] = 0u;
            if (c_next.hist_len > 32 * HALF) {
#pragma unroll
                for (int u = 0; u < HALF; ++u) {
                    const int t = lane + 32 * (HALF + u);
                    id[u] = -1; ct[u] = 0;
                    if (t < c_next.hist_len) { id[u] = __ldg(hid + t); ct[u] = __ldg(hct + t); }
                }
#pragma unroll
                for (int u = 0; u < HALF; ++u) packed[HALF + u] = pack(lane + 32 * (HALF + u), id[u], ct[u]);
            }
            b_id = -1; b_val = 0.0f;
            if (lane < c_next.bias_len) {
                if (b0 < 0 || b0 >= P.V) bad = true;
                else { b_id = b0; b_val = v0; }
            }
            row_bad = __any_sync(0xFFFFFFFFu, bad) ? 1 : 0;
            if (__any_sync(0xFFFFFFFFu, big)) return;          // a count too large to pack: consumers scan
            row_patch = 1;
        };
        auto prepare = [&](int row, int tile, int hb) -> Prep {
            if (row != cached_row) load_row(row);
            Prep r{row_patch, 0, 0};
            if (!LISTS || row_patch != 1) return r;
            const int first = tile * CTA_TILE;
#pragma unroll
            for (int u = 0; u < HPL; ++u) {
                const unsigned int li = (packed[u] & 0x3FFFFu) - (unsigned int)first;
                const bool hit = packed[u] != 0u && li < (unsigned int)CTA_TILE;
                const unsigned int hm = __ballot_sync(0xFFFFFFFFu, hit);
                if (hit) {
                    const int pos = r.npen + __popc(hm & ((1u << lane) - 1u));
                    if (pos < HIT_PEN_CAP) { sh.pen[hb][pos].li = (int)li; sh.pen[hb][pos].payload = (int)(packed[u] >> 18); }
                }
                r.npen += __popc(hm);
            }
            {
                const unsigned int li = (unsigned int)(b_id - first);
                const bool hit = b_id >= 0 && li < (unsigned int)CTA_TILE;
                const unsigned int hm = __ballot_sync(0xFFFFFFFFu, hit);
                if (hit) {
                    const int pos = __popc(hm & ((1u << lane) - 1u));
                    sh.bias[hb][pos].li = (int)li; sh.bias[hb][pos].payload = __float_as_int(b_val);
                }
                r.nbias = __popc(hm);
            }
            if (r.npen > HIT_PEN_CAP) r.patch = 2;             // crowded tile: the consumers scan the lists
            return r;
        };
        const unsigned long long l2_policy = l2_evict_first_policy();
        // Work queue: one counter of items.  A CTA first asks for `chunk` consecutive items (seven eighths of an
        // even share: a contiguous run like a static split would give it) and then for single items, each
        // requested one tile ahead (lane 0 keeps the raw result of the atomic until it is needed, so nothing
        // waits for it).  The single items even out the tail and whatever CTAs that started late did not take.
        unsigned int *queue = P.error + WS_QUEUE;
        int run_lo = nitems, run_hi = nitems, nxt_raw = nitems;
        if (lane == 0) run_lo = (int)atomicAdd(queue, (unsigned int)chunk);
        run_lo = __shfl_sync(0xFFFFFFFFu, run_lo, 0);
        run_hi = min(run_lo + chunk, nitems);
        if (lane == 0 && run_lo < nitems) nxt_raw = (int)atomicAdd(queue, 1u);
        auto current_item = [&]() -> int { return run_lo < run_hi ? run_lo : -1; };
        auto advance = [&]() {
            ++run_lo;
            if (run_lo >= run_hi) {
                run_lo = __shfl_sync(0xFFFFFFFFu, nxt_raw, 0);
                run_hi = min(run_lo + 1, nitems);
                if (lane == 0 && run_lo < nitems) nxt_raw = (int)atomicAdd(queue, 1u);
            }
        };
        int n = 0;
        Prep p_next{0, 0, 0};
        int item = current_item();
        bool prepared = false;
        // lane 0: the tile's bulk copy, with the arrival on full[s] (arrive == true) or with the bytes announced only
        // (the arrival then follows once the stage's description is written)
        auto issue_copy = [&](int row, int tile, int s, bool arrive) {
            const int first = tile * CTA_TILE;
            const int elems = min(CTA_TILE, ((P.V - first) + VEC - 1) / VEC * VEC);
            const unsigned int bytes = (unsigned int)elems * ELT;
            const unsigned char *src = reinterpret_cast<const unsigned char *>(P.logits) +
                                       ((size_t)row * (size_t)P.row_stride + (size_t)first) * ELT;
            if (arrive) mbar_arrive_expect_tx(&sh.full[s], bytes); else mbar_expect_tx(&sh.full[s], bytes);
#ifdef SONIC_TEST_WITHHOLD
            // test-only build: the bytes of one chosen tile are announced but its copy is never issued, so the waits
            // on this stage run out (consumers, then the producer) and the call reports it
            if (__ldcg(&P.error[WS_TEST_WITHHOLD]) == (unsigned int)(row * tiles + tile) + 1u) return;
#endif
            bulk_load(stages + (size_t)s * STAGE_BYTES, src, bytes, &sh.full[s], l2_policy);
        };
        // The CTA's first tile is requested at once, before its row's parameters and lists are known (they take two
        // rounds of global loads): the copy's latency hides behind them.  (A row of the cluster kernel's class gets
        // a copy nobody reads: such rows are rare.)
        if (item >= 0 && lane == 0) issue_copy(item / tiles, item % tiles, 0, false);
        for (;; ++n) {
            const int s = n % NSTAGE;
            if (n >= NSTAGE) {
                // the consumers have left tile n - NSTAGE: its stage and its hit buffer are free
                if (!mbar_wait(&sh.empty[s], ((n / NSTAGE) - 1) & 1)) {
                    if (lane == 0) atomicOr(P.error, ERR_TIMEOUT);
                    for (int i = n - NSTAGE; i < n; ++i) (void)mbar_wait(&sh.full[i % NSTAGE], (i / NSTAGE) & 1);       // copies under way
                    return;
                }
            }
            if (item < 0) {                            // out of work: tell the consumers
                if (lane == 0) { sh.meta[s].stop = 1; mbar_arrive(&sh.full[s]); }
                break;
            }
            const int row = item / tiles, tile = item - row * tiles;
            if (!prepared) {                           // the CTA's first tile: nothing was prepared ahead
                p_next = prepare(row, tile, n % (NSTAGE + 1));
                prepared = true;
            }
            const RowCfg c = c_next;
            const Prep pr = p_next;
            const int bad_now = row_bad;
            advance();
            const int nxt = current_item();
            __syncwarp();                              // the hit buffer's entries, written by all lanes, precede the arrival
            if (lane == 0) {
                StageMeta &m = sh.meta[s];
                m.cfg = c; m.row = row; m.tile = tile; m.skip = (c.cls == CLS_EXACT) ? 1 : 0;
                m.patch = pr.patch; m.npen = pr.npen; m.nbias = pr.nbias; m.hb = n % (NSTAGE + 1);
                m.stop = 0;
                m.bad = bad_now;
                if (n == 0 || c.cls == CLS_EXACT) mbar_arrive(&sh.full[s]);     // (the first tile's copy is under way; nothing is copied for rows of the cluster kernel's class)
                else issue_copy(row, tile, s, true);
            }
            __syncwarp();
            // hit buffer (n + 1) % (NSTAGE + 1) was last used by tile n - NSTAGE, which the consumers have left
            if (nxt >= 0) p_next = prepare(nxt / tiles, nxt % tiles, (n + 1) % (NSTAGE + 1));
            item = nxt;
        }
        return;
    }

    // ---------------------------------------------------------------- consumer warps
    for (int n = 0;; ++n) {
        const int s = n % NSTAGE;
        if (!mbar_wait(&sh.full[s], (n / NSTAGE) & 1)) {
            if (lane == 0) atomicOr(P.error, ERR_TIMEOUT);
            return;
        }
        if (sh.meta[s].stop) { KERNEL_T1(0); break; }
        const int row = sh.meta[s].row, tile = sh.meta[s].tile;
        const int tile_base = tile * CTA_TILE;
        const int wbase = tile_base + warp * WARP_TILE;
        const StageMeta &meta = sh.meta[s];
        if (meta.skip) {
            // a row of the cluster kernel: counted, its status word initialised
            if (tile == 0 && tid == 0) { P.rs[row].status = 0u; atomicAdd(&P.error[WS_NEXACT], 1u); }
        } else {
            const RowCfg c = meta.cfg;
            RowState *rs = P.rs + row;
            TileRec *rec = P.tiles + (size_t)row * MAX_TILES + tile;
            // Every per-row word of the workspace is initialised by the call that reads it: the tile's flags here
            // (before any barrier of this tile), the row's status word and, for rows of the histogram path, the
            // row's control block and its histogram by the CTA of the row's first tile.
            if (tid == 0) {
                rec->flags = meta.bad ? TILE_BADID : 0u;
                if (tile == 0) rs->status = 0u;
            }
            if (c.cls == CLS_DENSE && tile == 0) {
                uint4 *h = reinterpret_cast<uint4 *>(P.hist + (size_t)row * DBINS);
                for (int i = tid; i < DBINS / 2; i += STREAM_THREADS) h[i] = make_uint4(0u, 0u, 0u, 0u);
                if (tid == 0) {
                    DenseRow *dr = P.drow + row;
                    dr->nmembers = 0u;
                    dr->kmin = 0xFFFFFFFFu; dr->kmax = 0u; dr->overflow = 0u; dr->state = 0u;
                    P.dlist[atomicAdd(&P.error[WS_NDENSE], 1u)] = row;
                }
            }
            unsigned char *stage = stages + (size_t)s * STAGE_BYTES;
            const bool tail = tile_base + CTA_TILE > P.V;
            const int patch = LISTS ? meta.patch : 0;
            const bool patched = patch != 0;
            float *ptile = (DT == 0) ? reinterpret_cast<float *>(stage) : conv;    // fp32 view the sparse lists patch

            float e[EPL];
            auto read_raw = [&]() {
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const int li = warp * WARP_TILE + j * 32 * VEC + lane * VEC;
                    const uint4 raw = *reinterpret_cast<const uint4 *>(stage + (size_t)li * ELT);
                    const uint32_t r[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                    for (int q = 0; q < VEC; ++q) {
                        if (DT == 0) e[j * VEC + q] = __uint_as_float(r[q]);
                        else e[j * VEC + q] = __uint_as_float((q & 1) ? (r[q >> 1] & 0xFFFF0000u) : (r[q >> 1] << 16));
                    }
                }
            };
            auto read_f32 = [&](const float *src) {
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const float *p = src + warp * WARP_TILE + j * 32 * VEC + lane * VEC;
#pragma unroll
                    for (int q = 0; q < VEC; q += 4) {
                        const float4 v = *reinterpret_cast<const float4 *>(p + q);
                        e[j * VEC + q] = v.x; e[j * VEC + q + 1] = v.y; e[j * VEC + q + 2] = v.z; e[j * VEC + q + 3] = v.w;
                    }
                }
            };
            auto widen = [&]() {                      // bf16 only: the warp's part of the tile as fp32 in shared memory
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    float *p = conv + warp * WARP_TILE + j * 32 * VEC + lane * VEC;
#pragma unroll
                    for (int q = 0; q < VEC; q += 4)
                        *reinterpret_cast<float4 *>(p + q) = make_float4(e[j * VEC + q], e[j * VEC + q + 1], e[j * VEC + q + 2], e[j * VEC + q + 3]);
                }
            };
            if (patch == 1) {
                // the producer listed this tile's entries: every warp patches its own part, no block-wide barrier
                if (DT == 1) { read_raw(); widen(); }
                __syncwarp();
                for (int h = lane; h < meta.npen; h += 32) {
                    const Hit x = sh.pen[meta.hb][h];
                    if (x.li / WARP_TILE == warp) ptile[x.li] = apply_penalties(ptile[x.li], x.payload, c);
                }
                __syncwarp();
                for (int h = lane; h < meta.nbias; h += 32) {
                    const Hit x = sh.bias[meta.hb][h];
                    if (x.li / WARP_TILE == warp) ptile[x.li] = __fadd_rn(ptile[x.li], __int_as_float(x.payload));
                }
                __syncwarp();
                read_f32(ptile);
            } else if (patch == 2) {
                // long or crowded lists: all consumer threads scan them together
                if (DT == 1) { read_raw(); widen(); csync(); }
                const int req = (P.op == OP_VERIFY) ? row / (P.K + 1) : row;
                const int *hid = P.hist_ids + (size_t)req * P.hist_stride;
                const int *hct = P.hist_counts + (size_t)req * P.hist_stride;
                bool bad = false;
                for (int t = tid; t < c.hist_len; t += STREAM_THREADS) {
                    const int id = __ldg(hid + t);
                    if (id < 0 || id >= P.V) { bad = true; continue; }
                    const int li = id - tile_base;
                    if (li >= 0 && li < CTA_TILE) ptile[li] = apply_penalties(ptile[li], __ldg(hct + t), c);
                }
                csync();
                for (int t = tid; t < c.bias_len; t += STREAM_THREADS) {
                    const int id = __ldg(P.bias_ids + (size_t)req * P.bias_stride + t);
                    if (id < 0 || id >= P.V) { bad = true; continue; }
                    const int li = id - tile_base;
                    if (li >= 0 && li < CTA_TILE) ptile[li] = __fadd_rn(ptile[li], __ldg(P.bias_vals + (size_t)req * P.bias_stride + t));
                }
                if (bad) atomicOr(&rec->flags, TILE_BADID);          // (ordered after the first thread's store by the barriers above)
                csync();
                read_f32(ptile);
            } else {
                read_raw();
            }
            if (tail) {
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const int first = wbase + j * 32 * VEC + lane * VEC;
#pragma unroll
                    for (int q = 0; q < VEC; ++q) if (first + q >= P.V) e[j * VEC + q] = -CUDART_INF_F;
                }
            }
            if (c.div_all) {
#pragma unroll
                for (int q = 0; q < EPL; ++q) e[q] = div_tau(e[q], c.tau);
            }

            // per-vector maxima, half maxima, lane maximum
            float mv[NV];
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                float m = e[j * VEC];
#pragma unroll
                for (int q = 1; q < VEC; ++q) m = fmaxf(m, e[j * VEC + q]);
                mv[j] = m;
            }
            float qm[4];                               // maxima of the lane's four quarters (8 elements each)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                qm[i] = mv[i * (NV / 4)];
#pragma unroll
                for (int j = 1; j < NV / 4; ++j) qm[i] = fmaxf(qm[i], mv[i * (NV / 4) + j]);
            }
            const float h0 = fmaxf(qm[0], qm[1]), h1 = fmaxf(qm[2], qm[3]);
            const float lm = fmaxf(h0, h1);

            if (c.cls == CLS_GREEDY || c.cls == CLS_DENSE) {
                if (c.cls == CLS_DENSE) {
                    // histogram path: the processed logits (already divided by the temperature) are kept as ordered
                    // keys for the later passes; per tile the smallest finite key and the number of finite elements
                    uint32_t kmn = 0xFFFFFFFFu;
                    unsigned int nf = 0u;
                    unsigned int *yk = P.ykeys + (size_t)row * ((size_t)P.ytiles * CTA_TILE) + tile_base + warp * WARP_TILE;
#pragma unroll
                    for (int j = 0; j < NV; ++j) {
#pragma unroll
                        for (int q4 = 0; q4 < VEC; q4 += 4) {
                            uint32_t kk[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                kk[u] = okey(e[j * VEC + q4 + u]);
                                const bool fin = kk[u] > KEY_NEG_INF;
                                nf += fin ? 1u : 0u;
                                kmn = fin ? min(kmn, kk[u]) : kmn;
                            }
                            *reinterpret_cast<uint4 *>(yk + j * 32 * VEC + lane * VEC + q4) = make_uint4(kk[0], kk[1], kk[2], kk[3]);
                        }
                    }
                    kmn = __reduce_min_sync(0xFFFFFFFFu, kmn);
                    nf = __reduce_add_sync(0xFFFFFFFFu, nf);
                    if (lane == 0) { sh.kmin[s][warp] = kmn; sh.nfin[s][warp] = nf; }
                }
                float wm = lm;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xFFFFFFFFu, wm, off));
                unsigned long long key = 0ull;
                if (wm > -CUDART_INF_F) {
                    int best = 0x7FFFFFFF;
                    if (lm == wm) {
                        // slots ascend: the last write is the lowest; only the first quarter that holds the maximum is searched
                        bool found = false;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if (!found && qm[i] == wm) {
                                found = true;
#pragma unroll
                                for (int q = (i + 1) * (EPL / 4) - 1; q >= i * (EPL / 4); --q)
                                    if (e[q] == wm) best = slot_index<DT>(wbase, lane, q);
                            }
                        }
                    }
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
                    key = ((unsigned long long)okey(wm) << 32) | (uint32_t)(~(uint32_t)best);
                }
                if (lane == 0) sh.best[s][warp] = key;
                csync();
                if (tid == 0) {
                    unsigned long long b = sh.best[s][0];
#pragma unroll
                    for (int w = 1; w < STREAM_WARPS; ++w) b = max(b, sh.best[s][w]);
                    rec->best = b;
                    if (c.cls == CLS_DENSE) {
                        unsigned int kmn = sh.kmin[s][0], nf = sh.nfin[s][0];
#pragma unroll
                        for (int w = 1; w < STREAM_WARPS; ++w) { kmn = min(kmn, sh.kmin[s][w]); nf += sh.nfin[s][w]; }
                        rec->minkey = kmn; rec->nfin = nf;
                    }
                }
            } else {
                // warp cutoff: minimum over G groups of the group maximum.  Tile cutoff: the largest of the eight
                // warp cutoffs (warp mode) or the smallest (tile mode: a minimum over all 8 G groups of the tile).
                // In tile mode a group without a finite element (masked, or past the row's end) does not take
                // part: it would drag the cutoff to -inf and the tile would emit everything it has.
                float g;
                const int G = c.G;
                const bool tmin = c.tile_min;
                switch (G) {                                   // (one straight-line butterfly per group count)
                case 0: g = -CUDART_INF_F; break;
                case 1: g = warp_cutoff<32>(lm, tmin); break;
                case 2: g = warp_cutoff<16>(lm, tmin); break;
                case 4: g = warp_cutoff<8>(lm, tmin); break;
                case 8: g = warp_cutoff<4>(lm, tmin); break;
                case 16: g = warp_cutoff<2>(lm, tmin); break;
                case 32: g = warp_cutoff<1>(lm, tmin); break;
                default: {                                     // 64: half-lane groups
                    const float a0 = (tmin && h0 == -CUDART_INF_F) ? CUDART_INF_F : h0;
                    const float a1 = (tmin && h1 == -CUDART_INF_F) ? CUDART_INF_F : h1;
                    g = warp_cutoff<1>(fminf(a0, a1), false);
                    break;
                }
                }
                if (lane == 0) sh.tw[s][warp] = g;
                if (tid == 0) { sh.ncand[s] = 0; rec->cnt = 0u; }          // (the warps add to the record after the barrier)
                csync();
                static_assert(STREAM_WARPS == 8, "the eight warp cutoffs are read as two 128-bit words");
                const float4 ta = *reinterpret_cast<const float4 *>(&sh.tw[s][0]);
                const float4 tb = *reinterpret_cast<const float4 *>(&sh.tw[s][4]);
                float t;
                if (tmin) {
                    t = fminf(fminf(fminf(ta.x, ta.y), fminf(ta.z, ta.w)), fminf(fminf(tb.x, tb.y), fminf(tb.z, tb.w)));
                    if (t == CUDART_INF_F) t = -CUDART_INF_F;          // no finite element in the tile: nothing to emit
                } else {
                    t = fmaxf(fmaxf(fmaxf(ta.x, ta.y), fmaxf(ta.z, ta.w)), fmaxf(fmaxf(tb.x, tb.y), fmaxf(tb.z, tb.w)));
                }
                // every finite element >= t goes to the tile's candidate slot; a warp reserves its share of the
                // slot with one shared-memory atomic and adds it to the tile record (no second barrier).
                // Most warps hold no candidate at all and leave after one vote.  The others mark their
                // candidates in a bit mask and fetch the values again from the tile in shared memory (a
                // candidate is neither masked nor past the row's end, so the tile holds its value).
                const float t2 = fmaxf(t, -CUDART_MAX_NORMAL_F);           // e >= t2  <=>  e >= t and e is not -inf
                if (__any_sync(0xFFFFFFFFu, lm >= t2)) {
                    // a quarter of the lanes' elements without a candidate anywhere in the warp is skipped by one vote
                    unsigned int cm = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (__any_sync(0xFFFFFFFFu, qm[i] >= t2)) {
#pragma unroll
                            for (int q = i * (EPL / 4); q < (i + 1) * (EPL / 4); ++q) cm |= (e[q] >= t2) ? (1u << q) : 0u;
                        }
                    }
                    const int cnt = __popc(cm);
                    int incl, total;
                    if (!__any_sync(0xFFFFFFFFu, cnt > 1)) {
                        // the usual case, at most one candidate per lane: positions from one vote
                        const unsigned int has = __ballot_sync(0xFFFFFFFFu, cnt > 0);
                        incl = __popc(has & (0xFFFFFFFFu >> (31 - lane)));
                        total = __popc(has);
                    } else {
                        incl = cnt;
#pragma unroll
                        for (int off = 1; off < 32; off <<= 1) {
                            const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
                            if (lane >= off) incl += o;
                        }
                        total = __shfl_sync(0xFFFFFFFFu, incl, 31);
                    }
                    unsigned int base = 0;
                    if (lane == 0) {
                        base = atomicAdd(&sh.ncand[s], (unsigned int)total);
                        atomicAdd(&rec->cnt, (unsigned int)total);      // zero before the call; the merge kernel clears it
                    }
                    base = __shfl_sync(0xFFFFFFFFu, base, 0);
                    if ((int)base + total <= cap_t) {
                        unsigned long long *dst = P.cand + (size_t)row * P.cand_stride + (size_t)tile * cap_t + base + (incl - cnt);
                        const int lbase = warp * WARP_TILE + lane * VEC;
                        while (cm) {
                            const int q = __ffs(cm) - 1;
                            cm &= cm - 1;
                            const int li = lbase + (q / VEC) * (32 * VEC) + (q % VEC);
                            float v;
                            if (DT == 0 || patched) v = ptile[li];
                            else v = __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(stage)[li] << 16);
                            if (c.div_all) v = div_tau(v, c.tau);
                            *dst++ = ((unsigned long long)okey(v) << 32) | (uint32_t)(~(uint32_t)(tile_base + li));
                        }
                    }
                }
                if (tid == 0) rec->tkey = okey(t);
            }

            // generic-proxy writes into the stage (in-place patches) precede the next bulk copy into it
            if (DT == 0 && patched) fence_async_proxy();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.empty[s]);
    }
}

// One CTA per row of the streaming classes: combines the tile records and
// finishes the row (global top-k, truncation epilogue, token selection, or the
// per-position verification result).  Rows it cannot prove are flagged for the
// cluster kernel.
__global__ void __launch_bounds__(MERGE_THREADS, 2)
sonic_merge_kernel(const KParams P, const int tiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ MergeShared<MERGE_THREADS> s_merge;
    const int row = blockIdx.x;
    const int tid = threadIdx.x;
    KERNEL_T0(1);
    const RowCfg c = load_cfg(P, row);         // inputs only: independent of the streaming kernel
    const bool other = (c.cls == CLS_EXACT || c.cls == CLS_DENSE);
    if (other && row != 0) return;
    // the row's two uniforms depend on the inputs alone: drawn here, while the streaming kernel may still be running
    uint2 cells = make_uint2(0u, 0u);
    if (P.op != OP_TOPK && c.cls == CLS_TOPK) draw_cells(P, c, cells.x, cells.y);
    pdl_wait_primary();                        // tile records and candidates of the streaming kernel
    // The next kernel of the call (stage 2 of the histogram path) does not wait for this grid: it needs the
    // streaming kernel's results only, and those are complete once every CTA here is past its wait (the first
    // row's CTA never leaves before it).  So it is let go after the wait, and runs beside the merges.
    pdl_launch_dependents();
    if (row == 0 && tid == 0) P.error[WS_QUEUE] = 0u;    // the streaming kernel is done with its work counter
    if (other) return;
    if (__ldcg(&P.error[WS_ERROR]) & ERR_TIMEOUT) {
        // a bounded wait of the streaming kernel ran out (in this call or an earlier one on this workspace): the
        // tile records are not to be trusted, the row reports it instead of a token
        if (tid == 0) {
            if (P.op == OP_TOPK) { for (int j = 0; j < P.ktop; ++j) { P.out_vals[(size_t)row * P.ktop + j] = -CUDART_INF_F; P.out_idx[(size_t)row * P.ktop + j] = -1; } }
            else emit_row(P, c, row, -1, 0.0f, F_TIMEOUT, 0, 0.0f);
        }
        return;
    }
    RowState *rs = P.rs + row;
    const TileRec *recs = P.tiles + (size_t)row * MAX_TILES;
    const unsigned int tflags = (tid < tiles) ? __ldcg(&recs[tid].flags) : 0u;
    const bool badid = __syncthreads_or((int)(tflags & TILE_BADID)) != 0;
    if (c.bad || badid) {
        if (tid == 0) emit_row(P, c, row, -1, 0.0f, F_BADPARAM, 0, 0.0f);
        return;
    }
    if (c.cls == CLS_GREEDY) {
        if (tid < 32) {
            unsigned long long best = (tid < tiles) ? __ldcg(&recs[tid].best) : 0ull;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
            if (tid == 0) {
                if (P.op == OP_TOPK) {
                    // k == 1: a row of nothing but -inf still has a first element
                    P.out_vals[row] = best ? unkey((uint32_t)(best >> 32)) : -CUDART_INF_F;
                    P.out_idx[row] = best ? (int)(~(uint32_t)best) : 0;
                } else if (best == 0ull) {
                    emit_row(P, c, row, -1, 0.0f, F_NO_TOKEN, 0, 0.0f);
                } else {
                    const int token = (int)(~(uint32_t)best);
                    uint32_t flags = 0;
                    float pd = 0.0f;
                    if (P.op == OP_VERIFY && c.l < P.K) {
                        const bool acc = P.draft_tokens[(size_t)c.b * P.K + c.l] == token;
                        if (acc) { flags |= F_ACCEPT; pd = 1.0f; }
                    }
                    emit_row(P, c, row, token, 1.0f, flags, 1, pd);
                }
            }
        }
        return;
    }
    const bool ok = merge_topk_row<MERGE_THREADS, BlockSync>(P, c, row, tiles, reinterpret_cast<unsigned long long *>(smem_raw), reinterpret_cast<unsigned int *>(smem_raw + MERGE_CAP * 8), s_merge, tid, cells);
    if (tid == 0 && !ok) { rs->status = ST_FAILED; atomicAdd(&P.error[WS_FAILED_ROWS], 1u); }
    KERNEL_T1(1);
}

}  // namespace sonic
