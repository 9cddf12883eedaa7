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
// Structure of the streaming kernel: persistent CTAs (three per SM), each a
// producer warp plus eight consumer warps.  The producer takes tiles from a work
// queue, resolves each tile's row configuration and issues one bulk-TMA copy
// (cp.async.bulk, completion on an mbarrier) of the tile's logits into a ring of
// two shared-memory stages, one tile ahead of the consumers, so HBM requests
// stay in flight while the consumers compute.  Every mbarrier wait is bounded:
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
// low-precision value) is sorted by a warp.  About 35 instructions per key in eight barrier-separated steps, where a
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
    if (tid == 0) { sh.count = 0; sh.found = 0; }
    __syncthreads();
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
            const unsigned int t = v[j]; v[j] = run; run += t;
        }
#pragma unroll
        for (int j = 0; j < BPT; j += 4) *reinterpret_cast<uint4 *>(bins + tid * BPT + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
    __syncthreads();
    if (sh.found) {
        const int m = next_pow2(n0);
        for (int i = n0 + tid; i < m; i += THREADS) buf[i] = 0ull;
        __syncthreads();
        bitonic_sort_desc_cta<THREADS>(buf, m, tid);
        return;
    }
#pragma unroll
    for (int u = 0; u < ITEMS; ++u) {
        if (u * THREADS >= n0) break;
        if (u * THREADS + tid < n0) buf[atomicAdd(&bins[bucket(key[u])], 1u)] = key[u];
    }
    __syncthreads();
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
    // Small k: the k-th largest of the maxima of the row's warp tiles is a value that k elements reach and few more do (75
    // of 2^18 for k = 64), all of them candidates.  bins: the maxima.
    const int groups = tiles * STREAM_WARPS;
    const bool tight = 2 * c.k <= groups && c.k <= 100;
    static_assert(MAX_TILES * STREAM_WARPS * 2 == THREADS, "two threads per maximum at most");
    if (tight && tid < MAX_TILES * STREAM_WARPS) bins[tid] = (tid < groups) ? __ldcg(&P.wmax[(size_t)row * MAX_TILES * STREAM_WARPS + tid]) : 0u;
    csync();
    if (sh.found) return false;
    unsigned int tkey = sh.tkey;
    if (tight && tkey != KEY_NEG_INF) {
        const uint32_t kth = kth_max<THREADS>(bins, reinterpret_cast<unsigned int *>(sh.wsum), groups, c.k, tid);
        // (with a temperature a hair less: a value just below the bound may become equal to it when divided)
        float t = unkey(kth);
        if (c.temp) t -= fmaxf(fabsf(t) * 4.76837158203125e-07f, 1e-37f);
        if (kth > KEY_NEG_INF) tkey = max(tkey, okey(t));
    }
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
    if (Pn <= SMALL_MAX && n > 0) {
        int draft = -1;
        float q_draft = 0.0f;
        if (P.op == OP_VERIFY && c.l < P.K) {
            draft = __ldg(P.draft_tokens + (size_t)c.b * P.K + c.l);
            if (draft < 0 || draft >= P.V) draft = -1;
            if (draft >= 0) q_draft = __ldg(P.draft_probs + ((size_t)c.b * P.K + c.l) * (size_t)P.V + draft);
        }
        finish_small(P, c, row, buf, false, Pn, reinterpret_cast<unsigned long long *>(bins), tid, cells, draft, q_draft);
        return true;
    }
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
    int row, tile, slot;                       // slot: the row's parameters and lists
    int skip;                                  // the row belongs to another kernel: nothing to do
    int stop;                                  // no more tiles for this CTA (nothing else in the entry is valid)
    int next_row, next_tile;                   // the tile that follows (-1: none)
};
struct Hit { int id; int payload; };           // a bias entry: token, value bits
struct RowSlot {                               // a row's parameters and lists
    RowCfg cfg;
    int patch;                                 // 0 no lists, 1 they are here, 2 consumers scan them in global memory
    int bad;                                   // a list id outside [0, V)
    int off[MAX_TILES + 1];                    // the history entries of tile t: list[off[t], off[t + 1])
    uint32_t list[FILTER_HIST];                // id | count << 18
    Hit bias[FILTER_BIAS];
};

template <int DT>
struct StreamShared {
    static constexpr int NSTAGE = VecTraits<DT>::NSTAGE;
    unsigned long long full[NSTAGE];           // producer -> consumers: stage described and copy issued (one arrival + the copy's bytes)
    unsigned long long empty[NSTAGE];          // consumers -> producer: stage free (one arrival per consumer warp)
    StageMeta meta[NSTAGE];
    // per-stage results of the consumer warps, which the producer turns into the tile's record once all of them are done
    alignas(16) float tw[NSTAGE][STREAM_WARPS];
    unsigned int ncand[NSTAGE], badid[NSTAGE];
    unsigned long long best[NSTAGE][STREAM_WARPS];       // greedy rows: argmax; top-k rows: cutoff key << 32 | key of the warp's maximum
    unsigned int kmin[NSTAGE][STREAM_WARPS], nfin[NSTAGE][STREAM_WARPS];     // dense rows
    RowSlot slot[NSTAGE + 1];                  // the rows of the tiles in the ring and of the one that is prepared
};

template <int DT>
__global__ void __launch_bounds__(STREAM_CTA_THREADS, 3)
sonic_stream_kernel(const KParams P, const int tiles, const int nitems, const int chunk, const int cap_t) {     // cap_t: candidate slots per tile, CAND_CAP / tiles
    constexpr int VEC = VecTraits<DT>::VEC, NV = VecTraits<DT>::NV, NSTAGE = VecTraits<DT>::NSTAGE;
    constexpr int ELT = VecTraits<DT>::ELT;
    constexpr int STAGE_BYTES = CTA_TILE * ELT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // layout: NSTAGE raw stages | fp32 conversion tile (bf16 only) | control
    unsigned char *stages = smem_raw;
    float *conv = reinterpret_cast<float *>(smem_raw + NSTAGE * STAGE_BYTES);      // bf16 only
    StreamShared<DT> &sh = *reinterpret_cast<StreamShared<DT> *>(smem_raw + NSTAGE * STAGE_BYTES + (DT == 1 ? CTA_TILE * 4 : 0));
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
        // late (the SMs may be shared) find less or no work instead of holding back a fixed
        // share.  Per tile the producer waits for a free stage, requests the next tile at once, and only then writes the
        // record of the tile that left the stage and the description of the new one: what it does by itself is one warp's
        // serial work of several hundred cycles, which would otherwise lie between a stage's release and its next request.
        // On a new row one round of global loads brings the parameters and lists into a slot in shared memory.
        static_assert(SONIC_MAX_VOCAB <= (1 << 18), "packed history entries hold an 18-bit id");
        static_assert(CTA_TILE == 1 << 13, "tile of a token");
        constexpr int HALF = FILTER_HIST / 64;     // history entries per lane and round of loads
        int cached_row = -1, cur_slot = 0, cls_cur = CLS_GREEDY;
        auto load_row = [&](int row) {
            const int req = (P.op == OP_VERIFY) ? row / (P.K + 1) : row;
            const int *hid = P.hist_ids ? P.hist_ids + (size_t)req * P.hist_stride : nullptr;
            const int *hct = P.hist_counts ? P.hist_counts + (size_t)req * P.hist_stride : nullptr;
            const int *bid = P.bias_ids ? P.bias_ids + (size_t)req * P.bias_stride : nullptr;
            const float *bvl = P.bias_vals ? P.bias_vals + (size_t)req * P.bias_stride : nullptr;
            // the first round of loads goes out before the first use (the lengths arrive with the parameters:
            // bound by the strides); the second half of a long history follows in a round of its own
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
            const RowCfg c = resolve_cfg(P, row, raw);
            cached_row = row;
            cls_cur = c.cls;
            cur_slot = (cur_slot + 1) % (NSTAGE + 1);
            RowSlot &q = sh.slot[cur_slot];
            int patch = (c.hist_len > 0 || c.bias_len > 0) ? 1 : 0;
            if (c.hist_len > FILTER_HIST || c.bias_len > FILTER_BIAS) patch = 2;
            bool bad = false, big = false;
            if (patch == 1) {
                // the history by tile: count, offsets, place
                q.off[lane] = 0;
                __syncwarp();
                uint32_t e[2 * HALF];
                int at[2 * HALF];
                auto take = [&](int t, int i, int cnt, uint32_t &out, int &rank) {
                    out = 0u; rank = 0;
                    if (t >= c.hist_len) return;
                    if (i < 0 || i >= P.V) { bad = true; return; }
                    if (cnt > FILTER_COUNT_MAX) { big = true; return; }
                    if (cnt <= 0) return;
                    out = (uint32_t)i | ((uint32_t)cnt << 18);
                    rank = atomicAdd(&q.off[i >> 13], 1);
                };
#pragma unroll
                for (int u = 0; u < HALF; ++u) take(lane + 32 * u, id[u], ct[u], e[u], at[u]);
#pragma unroll
                for (int u = 0; u < HALF; ++u) { e[HALF + u] = 0u; at[HALF + u] = 0; }
                if (c.hist_len > 32 * HALF) {
#pragma unroll
                    for (int u = 0; u < HALF; ++u) {
                        const int t = lane + 32 * (HALF + u);
                        id[u] = -1; ct[u] = 0;
                        if (t < c.hist_len) { id[u] = __ldg(hid + t); ct[u] = __ldg(hct + t); }
                    }
#pragma unroll
                    for (int u = 0; u < HALF; ++u) take(lane + 32 * (HALF + u), id[u], ct[u], e[HALF + u], at[HALF + u]);
                }
                __syncwarp();
                const int cnt = q.off[lane];
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const int up = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += up; }
                q.off[lane] = incl - cnt;
                if (lane == 31) q.off[32] = incl;
                __syncwarp();
#pragma unroll
                for (int u = 0; u < 2 * HALF; ++u)
                    if (e[u]) q.list[q.off[(e[u] & 0x3FFFFu) >> 13] + at[u]] = e[u];
                Hit h;
                h.id = -1; h.payload = 0;
                if (lane < c.bias_len) {
                    if (b0 < 0 || b0 >= P.V) bad = true;
                    else { h.id = b0; h.payload = __float_as_int(v0); }
                }
                q.bias[lane] = h;
                bad = __any_sync(0xFFFFFFFFu, bad);
                if (__any_sync(0xFFFFFFFFu, big)) patch = 2;       // a count too large to pack: consumers scan
            }
            if (lane == 0) { q.cfg = c; q.patch = patch; q.bad = bad ? 1 : 0; }
            __syncwarp();
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
        // The next item, with its row's parameters and lists loaded.
        auto find_item = [&]() -> int {
            const int it = current_item();
            if (it >= 0 && it / tiles != cached_row) load_row(it / tiles);
            return it;
        };
        int item = current_item();
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
        // The record of a tile that every consumer warp has left: candidates, cutoff, argmax, bad list ids.
        auto retire = [&](int s) {
            const int row = sh.meta[s].row, tile = sh.meta[s].tile;
            if (sh.meta[s].skip) {
                // a row of the cluster kernel: counted, its status word initialised
                if (tile == 0 && lane == 0) { P.rs[row].status = 0u; atomicAdd(&P.error[WS_NEXACT], 1u); }
                return;
            }
            const RowSlot &q = sh.slot[sh.meta[s].slot];
            unsigned long long b = (lane < STREAM_WARPS) ? sh.best[s][lane] : 0ull;
            unsigned int kmn = 0xFFFFFFFFu, nf = 0u;
            if (q.cfg.cls == CLS_DENSE) {
                kmn = __reduce_min_sync(0xFFFFFFFFu, lane < STREAM_WARPS ? sh.kmin[s][lane] : 0xFFFFFFFFu);
                nf = __reduce_add_sync(0xFFFFFFFFu, lane < STREAM_WARPS ? sh.nfin[s][lane] : 0u);
            }
            if (lane < STREAM_WARPS && q.cfg.cls == CLS_TOPK) P.wmax[((size_t)row * MAX_TILES + tile) * STREAM_WARPS + lane] = (uint32_t)b;
#pragma unroll
            for (int off = STREAM_WARPS / 2; off > 0; off >>= 1) b = max(b, __shfl_xor_sync(0xFFFFFFFFu, b, off));
            if (lane == 0) {
                TileRec r;
                r.best = b; r.cnt = sh.ncand[s]; r.tkey = (unsigned int)(b >> 32);
                r.flags = (q.bad || sh.badid[s]) ? TILE_BADID : 0u;
                r.minkey = kmn; r.nfin = nf; r.pad = 0u;
                P.tiles[(size_t)row * MAX_TILES + tile] = r;
                if (tile == 0) P.rs[row].status = 0u;
            }
            __syncwarp();
        };
        int n = -1;
        for (;; ++n) {                                 // (round -1 only prepares the first tile)
            if (n >= 0) {
                const int s = n % NSTAGE;
                const bool skip = item >= 0 && cls_cur == CLS_EXACT;
                const int row = item / tiles, tile = item - row * tiles;
                if (n >= NSTAGE) {
                    // the consumers have left tile n - NSTAGE: its stage is free
                    if (!mbar_wait(&sh.empty[s], ((n / NSTAGE) - 1) & 1)) {
                        if (lane == 0) atomicOr(P.error, ERR_TIMEOUT);
                        return;
                    }
                    // (the first tiles' copies are under way; nothing is copied for rows of the cluster kernel's class)
                    if (item >= 0 && !skip && lane == 0) issue_copy(row, tile, s, false);
                    retire(s);
                }
                if (item < 0) {                            // out of work: tell the consumers
                    if (lane == 0) { sh.meta[s].stop = 1; mbar_arrive(&sh.full[s]); }
                    break;
                }
                advance();
                const int hint = current_item();           // the tile that follows
                if (lane == 0) {
                    if (n > 0 && n < NSTAGE && !skip) issue_copy(row, tile, s, false);
                    StageMeta &m = sh.meta[s];
                    m.row = row; m.tile = tile; m.slot = cur_slot; m.skip = skip ? 1 : 0;
                    m.stop = 0;
                    m.next_row = (hint >= 0) ? hint / tiles : -1;
                    m.next_tile = (hint >= 0) ? hint - m.next_row * tiles : -1;
                    sh.ncand[s] = 0u; sh.badid[s] = 0u;
                    mbar_arrive(&sh.full[s]);
                }
                __syncwarp();
            }
            item = find_item();
        }
        for (int i = max(0, n - NSTAGE + 1); i < n; ++i) {     // the last tiles
            if (!mbar_wait(&sh.empty[i % NSTAGE], (i / NSTAGE) & 1)) {
                if (lane == 0) atomicOr(P.error, ERR_TIMEOUT);
                return;
            }
            retire(i % NSTAGE);
        }
        return;
    }

    // ---------------------------------------------------------------- consumer warps
    // The grammar words of a warp tile (32 words, one coalesced load, handed to the lanes that need them by
    // shuffles later) are requested one tile ahead: each stage names the tile that follows it.
    uint32_t mword_pre = 0u;
    int pre_row = -1, pre_tile = -1;
    auto load_mask_words = [&](int row, int tile) -> uint32_t {
        const int w = ((tile * CTA_TILE + warp * WARP_TILE) >> 5) + lane;
        return (w < ((P.V + 31) >> 5)) ? __ldg(P.bitmask + (size_t)row * P.bitmask_stride + w) : 0u;
    };
    // What a warp carries from tile to tile of a row.  Top-k rows: the cutoff, taken from the CTA's first tile of the row
    // and kept for the tiles that follow (any cutoff is good as long as the tile's record names it; a tile then costs its
    // maxima and one vote, without a block barrier).  Greedy rows: what an element must reach to matter.
    int cut_row = -1, g_row = -1;
    float cut = 0.0f, g_thr = 0.0f;
    for (int n = 0;; ++n) {
        const int s = n % NSTAGE;
        if (!mbar_wait(&sh.full[s], (n / NSTAGE) & 1)) {
            if (lane == 0) atomicOr(P.error, ERR_TIMEOUT);
            return;
        }
        const StageMeta &meta = sh.meta[s];
        if (meta.stop) { KERNEL_T1(0); break; }
        const int row = meta.row, tile = meta.tile;
        const int tile_base = tile * CTA_TILE;
        uint32_t mword = 0xFFFFFFFFu;
        if (P.bitmask) {
            mword = (row == pre_row && tile == pre_tile) ? mword_pre : load_mask_words(row, tile);
            pre_row = meta.next_row; pre_tile = meta.next_tile;
            if (pre_row >= 0) mword_pre = load_mask_words(pre_row, pre_tile);
        }
        if (!meta.skip) {
            const unsigned char *stage = stages + (size_t)s * STAGE_BYTES;
            const RowSlot &slot = sh.slot[meta.slot];
            const bool masked = (slot.cfg.z & M_GRAMMAR) != 0;
            const bool tail = tile_base + CTA_TILE > P.V;
            const int patch = slot.patch;
            // word: which of the 32 consecutive elements from lane * 32 count.  Under a sparse mask (a grammar allows a few per
            // cent of the ids) a lane walks its word's few set bits instead of 32 elements.
            uint32_t word = masked ? mword : 0xFFFFFFFFu;
            if (tail) { const int left = P.V - tile_base - warp * WARP_TILE - lane * 32; if (left < 32) word &= left > 0 ? (1u << left) - 1u : 0u; }
            const bool sparse = masked && __all_sync(0xFFFFFFFFu, __popc(word) <= 8);
            float *ptile = (DT == 0) ? reinterpret_cast<float *>(stages + (size_t)s * STAGE_BYTES) : conv;    // fp32 view the sparse lists patch
            bool wide = DT == 0;                               // the warp's part is fp32 in ptile (else bf16 in the stage)
            const int lane0 = warp * WARP_TILE + lane * VEC;   // the lane's first element within the tile
            auto widen = [&]() {                               // bf16 only: the warp's part as fp32
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const uint4 raw = *reinterpret_cast<const uint4 *>(stage + (size_t)(lane0 + j * 32 * VEC) * ELT);
                    float *p = conv + lane0 + j * 32 * VEC;
                    *reinterpret_cast<float4 *>(p) = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u),
                                                                 __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xFFFF0000u));
                    *reinterpret_cast<float4 *>(p + 4) = make_float4(__uint_as_float(raw.z << 16), __uint_as_float(raw.z & 0xFFFF0000u),
                                                                     __uint_as_float(raw.w << 16), __uint_as_float(raw.w & 0xFFFF0000u));
                }
            };
            // penalties and biases commute with the mask (a masked logit stays -inf), so they are applied to the unmasked tile
            if (patch == 1) {
                // the producer listed this tile's entries: every warp patches its own part, if there are any in it
                // (that the mask allows)
                const int first = slot.off[tile], npen = slot.off[tile + 1] - first, nbias = slot.cfg.bias_len;
                auto mine = [&](int li) -> bool {                // (every lane calls it; li: element of the tile, or anything outside)
                    const uint32_t w = __shfl_sync(0xFFFFFFFFu, word, (li >> 5) & 31);
                    return (li >> 10) == warp && ((w >> (li & 31)) & 1u);
                };
                static_assert(WARP_TILE == 1024 && FILTER_BIAS == 32, "element -> warp; one bias entry per lane");
                bool any = false;
                for (int h0 = 0; h0 < npen; h0 += 32) {
                    const bool m = mine((h0 + lane < npen) ? (int)(slot.list[first + h0 + lane] & 0x3FFFFu) - tile_base : -1);
                    any = any || m;
                }
                int bli = -1;
                float bval = 0.0f;
                if (nbias > 0) {
                    const Hit h = slot.bias[lane];
                    bli = (h.id >= 0) ? h.id - tile_base : -1;
                    bval = __int_as_float(h.payload);
                    if (!mine(bli)) bli = -1;
                    any = any || bli >= 0;
                }
                if (__any_sync(0xFFFFFFFFu, any)) {
                    const RowCfg c = slot.cfg;
                    if (DT == 1) { widen(); wide = true; }
                    __syncwarp();
                    for (int h = lane; h < npen; h += 32) {
                        const uint32_t e = slot.list[first + h];
                        const int li = (int)(e & 0x3FFFFu) - tile_base;
                        if ((li >> 10) == warp) ptile[li] = apply_penalties(ptile[li], (int)(e >> 18), c);
                    }
                    __syncwarp();
                    if (bli >= 0) ptile[bli] = __fadd_rn(ptile[bli], bval);
                    __syncwarp();
                }
            } else if (patch == 2) {
                // long or crowded lists: all consumer threads scan them together
                const RowCfg c = slot.cfg;
                if (DT == 1) { widen(); wide = true; csync(); }
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
                if (bad) sh.badid[s] = 1u;
                csync();
            }

            if (slot.cfg.cls == CLS_DENSE) {
                // Histogram path: the processed logits (divided by the temperature) are kept as ordered keys for the later
                // passes; per tile the largest and smallest finite key and the number of finite elements.  The CTA of the
                // row's first tile initialises the row's control block and histogram and lists the row.
                if (tile == 0) {
                    uint4 *h = reinterpret_cast<uint4 *>(P.hist + (size_t)row * DBINS);
                    for (int i = tid; i < DBINS / 2; i += STREAM_THREADS) h[i] = make_uint4(0u, 0u, 0u, 0u);
                    if (tid == 0) {
                        DenseRow *dr = P.drow + row;
                        dr->ticket_h = 0u; dr->ticket_c = 0u; dr->ticket_r = 0u; dr->nmembers = 0u;
                        dr->kmin = 0xFFFFFFFFu; dr->kmax = 0u; dr->overflow = 0u; dr->state = 0u;
                        P.dlist[atomicAdd(&P.error[WS_NDENSE], 1u)] = row;
                    }
                }
                const bool divide = slot.cfg.div_all, all = !masked && !tail;
                const float tau = slot.cfg.tau;
                uint32_t kmx = 0u, kmn = 0xFFFFFFFFu;
                unsigned int nf = 0u;
                unsigned int *yk = P.ykeys + (size_t)row * ((size_t)P.ytiles * CTA_TILE) + tile_base;
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const int li = lane0 + j * 32 * VEC;
                    const uint32_t bits = all ? 0xFFFFFFFFu : __shfl_sync(0xFFFFFFFFu, word, (j * 32 * VEC + lane * VEC) >> 5) >> ((lane * VEC) & 31);
                    float v[VEC];
                    if (DT == 1 && !wide) {
                        const uint4 raw = *reinterpret_cast<const uint4 *>(stage + (size_t)li * ELT);
                        const uint32_t r[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                        for (int q = 0; q < VEC; ++q) v[q] = __uint_as_float((q & 1) ? (r[(q >> 1) & 3] & 0xFFFF0000u) : (r[(q >> 1) & 3] << 16));
                    } else {
#pragma unroll
                        for (int q = 0; q < VEC; q += 4) {
                            const float4 a = *reinterpret_cast<const float4 *>(ptile + li + q);
                            v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
                        }
                    }
#pragma unroll
                    for (int q4 = 0; q4 < VEC; q4 += 4) {
                        uint32_t kk[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            float y = ((bits >> (q4 + u)) & 1u) ? v[q4 + u] : -CUDART_INF_F;
                            if (divide) y = div_tau(y, tau);
                            kk[u] = okey(y);
                            const bool fin = kk[u] > KEY_NEG_INF;
                            nf += fin ? 1u : 0u;
                            kmn = fin ? min(kmn, kk[u]) : kmn;
                            kmx = fin ? max(kmx, kk[u]) : kmx;
                        }
                        *reinterpret_cast<uint4 *>(yk + li + q4) = make_uint4(kk[0], kk[1], kk[2], kk[3]);
                    }
                }
                kmx = __reduce_max_sync(0xFFFFFFFFu, kmx);
                kmn = __reduce_min_sync(0xFFFFFFFFu, kmn);
                nf = __reduce_add_sync(0xFFFFFFFFu, nf);
                if (lane == 0) { sh.best[s][warp] = (unsigned long long)kmx << 32; sh.kmin[s][warp] = kmn; sh.nfin[s][warp] = nf; }
                if (DT == 0 && patch != 0) fence_async_proxy();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.empty[s]);
                continue;
            }

            // Maxima of the lane's vectors.  ebits: which of its 32 elements count (allowed by the mask, inside the row).
            // raw: the lane's elements as they lie in the stage (not of a widened part): what is looked at again stays in registers
            float mv[NV];
            uint4 raw[NV];
            uint32_t ebits = 0xFFFFFFFFu;
            auto value = [&](int li) -> float {                // one element of the tile
                return (DT == 1 && !wide) ? __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(stage)[li] << 16) : ptile[li];
            };
            float h0 = -CUDART_INF_F, h1 = -CUDART_INF_F;      // maxima of the lane's two halves
            if (sparse) {
                for (uint32_t w = word; w; w &= w - 1u) {
                    const int b = __ffs(w) - 1;
                    const float v = value(warp * WARP_TILE + lane * 32 + b);
                    if (b < 16) h0 = fmaxf(h0, v); else h1 = fmaxf(h1, v);
                }
            } else if (!masked && !tail) {
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const int li = lane0 + j * 32 * VEC;
                    if (DT == 1 && !wide) {
                        // bf16 pairs: half an instruction per element
                        raw[j] = *reinterpret_cast<const uint4 *>(stage + (size_t)li * ELT);
                        const __nv_bfloat162 m = __hmax2(__hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[j].x), *reinterpret_cast<const __nv_bfloat162 *>(&raw[j].y)),
                                                         __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[j].z), *reinterpret_cast<const __nv_bfloat162 *>(&raw[j].w)));
                        const uint32_t u = *reinterpret_cast<const uint32_t *>(&m);
                        mv[j] = fmaxf(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
                    } else {
                        const float4 a = *reinterpret_cast<const float4 *>(ptile + li);
                        if (DT == 0) raw[j] = make_uint4(__float_as_uint(a.x), __float_as_uint(a.y), __float_as_uint(a.z), __float_as_uint(a.w));
                        mv[j] = fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w));
                        if (VEC == 8) {
                            const float4 b = *reinterpret_cast<const float4 *>(ptile + li + 4);
                            mv[j] = fmaxf(mv[j], fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
                        }
                    }
                }
            } else {
                ebits = 0u;
#pragma unroll
                for (int j = 0; j < NV; ++j) {
                    const int li = lane0 + j * 32 * VEC;
                    const uint32_t bits = (__shfl_sync(0xFFFFFFFFu, word, (j * 32 * VEC + lane * VEC) >> 5) >> ((lane * VEC) & 31)) & ((1u << VEC) - 1u);
                    ebits |= bits << (j * VEC);
                    float v[VEC];
                    if (DT == 0 || !wide) {
                        raw[j] = *reinterpret_cast<const uint4 *>(stage + (size_t)li * ELT);
                        const uint32_t r[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
                        for (int q = 0; q < VEC; ++q) v[q] = DT == 0 ? __uint_as_float(r[q & 3]) : __uint_as_float((q & 1) ? (r[(q >> 1) & 3] & 0xFFFF0000u) : (r[(q >> 1) & 3] << 16));
                    } else {
#pragma unroll
                        for (int q = 0; q < VEC; q += 4) {
                            const float4 a = *reinterpret_cast<const float4 *>(ptile + li + q);
                            v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
                        }
                    }
                    mv[j] = -CUDART_INF_F;
#pragma unroll
                    for (int q = 0; q < VEC; ++q) mv[j] = ((bits >> q) & 1u) ? fmaxf(mv[j], v[q]) : mv[j];
                }
            }
            if (!sparse) {
#pragma unroll
                for (int j = 0; j < NV / 2; ++j) { h0 = fmaxf(h0, mv[j]); h1 = fmaxf(h1, mv[NV / 2 + j]); }
            }
            const float lm = fmaxf(h0, h1);
            // The elements of the lane's vectors whose maximum reaches t, one vector after the other (rare: read again):
            // f(value, index within the tile) for those that reach t.
            auto visit = [&](float t, auto f) {
                if (sparse) {
#pragma unroll 1
                    for (uint32_t w = word; w; w &= w - 1u) {
                        const int li = warp * WARP_TILE + lane * 32 + __ffs(w) - 1;
                        const float v = value(li);
                        if (v >= t) f(v, li);
                    }
                    return;
                }
                unsigned int vm = 0u;
#pragma unroll
                for (int j = 0; j < NV; ++j) vm |= (mv[j] >= t) ? (1u << j) : 0u;
#pragma unroll 1
                while (vm) {
                    const int j = __ffs(vm) - 1, li = lane0 + j * 32 * VEC;
                    vm &= vm - 1u;
                    const uint32_t bits = ebits >> (j * VEC);
#pragma unroll
                    for (int q = 0; q < VEC; q += 4) {
                        float4 a;
                        if (DT == 1 && !wide) {
                            const uint2 r = *reinterpret_cast<const uint2 *>(stage + (size_t)(li + q) * ELT);
                            a = make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
                        } else a = *reinterpret_cast<const float4 *>(ptile + li + q);
                        if (a.x >= t && ((bits >> q) & 1u)) f(a.x, li + q);
                        if (a.y >= t && ((bits >> (q + 1)) & 1u)) f(a.y, li + q + 1);
                        if (a.z >= t && ((bits >> (q + 2)) & 1u)) f(a.z, li + q + 2);
                        if (a.w >= t && ((bits >> (q + 3)) & 1u)) f(a.w, li + q + 3);
                    }
                }
            };

            if (slot.cfg.cls == CLS_GREEDY) {
                // The argmax of the processed logits, lowest index first.  Only elements at or above the largest so far can
                // matter (with a temperature: above a hair less, since the division may make them equal).
                if (row != g_row) { g_row = row; g_thr = -CUDART_MAX_NORMAL_F; }
                unsigned long long best = 0ull;
                if (__any_sync(0xFFFFFFFFu, lm >= g_thr)) {
                    const bool temp = slot.cfg.temp;
                    const float tau = slot.cfg.tau;
                    if (lm >= g_thr) visit(g_thr, [&](float z, int li) {
                        const uint32_t key = okey(temp ? div_tau(z, tau) : z);
                        best = max(best, ((unsigned long long)key << 32) | (uint32_t)(~(uint32_t)(tile_base + li)));
                    });
                    __syncwarp();
                    const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(best >> 32));
                    const uint32_t lo = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(best >> 32) == hi ? (uint32_t)best : 0u);
                    best = ((unsigned long long)hi << 32) | lo;
                    const float z = unkey(__reduce_max_sync(0xFFFFFFFFu, okey(lm)));
                    g_thr = fmaxf(g_thr, temp ? z - fmaxf(fabsf(z) * 4.76837158203125e-07f, 1e-37f) : z);
                }
                if (lane == 0) sh.best[s][warp] = best;
            } else {
                const int G = slot.cfg.G;
                const bool tmin = slot.cfg.tile_min;
                // warp cutoff: minimum over G groups of the group maximum.  Tile cutoff: the largest of the eight warp cutoffs
                // (warp mode) or the smallest (tile mode: a minimum over all 8 G groups of the tile).  In tile mode a group
                // without a finite element (masked, or past the row's end) does not take part: it would drag the cutoff
                // to -inf and the tile would emit everything it has.
                auto group_cutoff = [&]() -> float {
                    switch (G) {                               // (one straight-line butterfly per group count)
                    case 0: return -CUDART_INF_F;
                    case 1: return warp_cutoff<32>(lm, tmin);
                    case 2: return warp_cutoff<16>(lm, tmin);
                    case 4: return warp_cutoff<8>(lm, tmin);
                    case 8: return warp_cutoff<4>(lm, tmin);
                    case 16: return warp_cutoff<2>(lm, tmin);
                    case 32: return warp_cutoff<1>(lm, tmin);
                    default: {                                 // 64: half-lane groups
                        const float a0 = (tmin && h0 == -CUDART_INF_F) ? CUDART_INF_F : h0;
                        const float a1 = (tmin && h1 == -CUDART_INF_F) ? CUDART_INF_F : h1;
                        return warp_cutoff<1>(fminf(a0, a1), false);
                    }
                    }
                };
                // (many groups, many candidates: a cutoff per tile keeps them down)
                float t = cut;
                if (row != cut_row || G > 8) {
                    const float g = group_cutoff();
                    if (lane == 0) sh.tw[s][warp] = g;
                    csync();
                    static_assert(STREAM_WARPS == 8, "the eight warp cutoffs are read as two 128-bit words");
                    const float4 ta = *reinterpret_cast<const float4 *>(&sh.tw[s][0]);
                    const float4 tb = *reinterpret_cast<const float4 *>(&sh.tw[s][4]);
                    if (tmin) {
                        t = fminf(fminf(fminf(ta.x, ta.y), fminf(ta.z, ta.w)), fminf(fminf(tb.x, tb.y), fminf(tb.z, tb.w)));
                        if (t == CUDART_INF_F) t = -CUDART_INF_F;          // no finite element in the tile: nothing to emit
                    } else {
                        t = fmaxf(fmaxf(fmaxf(ta.x, ta.y), fmaxf(ta.z, ta.w)), fmaxf(fmaxf(tb.x, tb.y), fmaxf(tb.z, tb.w)));
                    }
                    // (a tile that bounds nothing leaves the cutoff to the next one)
                    cut = t;
                    cut_row = (t > -CUDART_INF_F) ? row : -1;
                } else if (__popc(__ballot_sync(0xFFFFFFFFu, lm >= t)) > 28) {
                    // far more candidates than the cutoff was meant for (values that depend on the position): the warp takes
                    // a cutoff of its own for this tile
                    t = fmaxf(t, group_cutoff());
                    if (t == CUDART_INF_F) t = cut;
                }
                const uint32_t wk = __reduce_max_sync(0xFFFFFFFFu, okey(lm));
                if (lane == 0) sh.best[s][warp] = ((unsigned long long)okey(t) << 32) | wk;
                // every finite element >= t goes to the tile's candidate slot
                const float t2 = fmaxf(t, -CUDART_MAX_NORMAL_F);           // e >= t2  <=>  e >= t and e is not -inf
                const unsigned int cand = __ballot_sync(0xFFFFFFFFu, lm >= t2);
                if (cand) {
                    unsigned long long *dst = P.cand + (size_t)row * P.cand_stride + (size_t)tile * cap_t;
                    auto put = [&](unsigned int pos, float z, int li) {
                        if ((int)pos < cap_t) dst[pos] = ((unsigned long long)okey(z) << 32) | (uint32_t)(~(uint32_t)(tile_base + li));
                    };
                    if (sparse) {
                        if (lm >= t2) visit(t2, [&](float z, int li) { put(atomicAdd(&sh.ncand[s], 1u), z, li); });
                    } else {
                        // Every lane marks its candidates in a bit mask, a quarter of its elements at a time (a quarter without
                        // one anywhere in the warp is skipped by a vote); one reservation for the warp.  The marked values are
                        // fetched again from the tile.
                        unsigned int cm = 0u;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float qm = mv[i * NV / 4];
                            if (NV == 8) qm = fmaxf(qm, mv[i * NV / 4 + 1]);
                            if (__any_sync(0xFFFFFFFFu, qm >= t2)) {
#pragma unroll
                                for (int j = i * NV / 4; j < (i + 1) * NV / 4; ++j) {
                                    const uint32_t r[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
                                    if (DT == 1 && wide) {
                                        const float4 a = *reinterpret_cast<const float4 *>(ptile + lane0 + j * 32 * VEC);
                                        const float4 b = *reinterpret_cast<const float4 *>(ptile + lane0 + j * 32 * VEC + (VEC == 8 ? 4 : 0));
                                        cm |= ((a.x >= t2 ? 1u : 0u) | (a.y >= t2 ? 2u : 0u) | (a.z >= t2 ? 4u : 0u) | (a.w >= t2 ? 8u : 0u)) << (j * VEC);
                                        cm |= ((b.x >= t2 ? 16u : 0u) | (b.y >= t2 ? 32u : 0u) | (b.z >= t2 ? 64u : 0u) | (b.w >= t2 ? 128u : 0u)) << (j * VEC);
                                    } else {
#pragma unroll
                                        for (int q = 0; q < VEC; ++q) {
                                            const float v = DT == 0 ? __uint_as_float(r[q & 3]) : __uint_as_float((q & 1) ? (r[(q >> 1) & 3] & 0xFFFF0000u) : (r[(q >> 1) & 3] << 16));
                                            cm |= (v >= t2) ? (1u << (j * VEC + q)) : 0u;
                                        }
                                    }
                                }
                            }
                        }
                        cm &= ebits;
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
                            for (int off = 1; off < 32; off <<= 1) { const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off); if (lane >= off) incl += o; }
                            total = __shfl_sync(0xFFFFFFFFu, incl, 31);
                        }
                        unsigned int base = 0u;
                        if (lane == 0) base = atomicAdd(&sh.ncand[s], (unsigned int)total);
                        base = __shfl_sync(0xFFFFFFFFu, base, 0) + (unsigned int)(incl - cnt);
                        while (cm) {
                            const int b = __ffs(cm) - 1, li = lane0 + (b / VEC) * (32 * VEC) + (b % VEC);
                            cm &= cm - 1u;
                            put(base++, value(li), li);
                        }
                    }
                }
                __syncwarp();
            }

            // generic-proxy writes into the stage (in-place patches) precede the next bulk copy into it
            if (DT == 0 && patch != 0) fence_async_proxy();
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
