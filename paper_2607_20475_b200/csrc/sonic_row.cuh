// Row kernel: one thread-block cluster per row does the whole row - load, logit processing, selection, truncation,
// draw, verification - in one launch, the processed row staying in distributed shared memory.
//
// What bounds a row is not its bytes (a 131072-entry bf16 row is 0.26 MB, 0.04 us at the copy rate) but the chain of
// steps that depend on each other, and inside a step the instructions per element (8192 elements on one SM cost 64 cycles
// per instruction).  A kernel boundary costs 3-4 us of that chain (the next kernel finds its row, its parameters and
// its keys again through dependent global loads); an exchange through distributed shared memory with a cluster barrier
// costs about 1 us and nothing is read twice.  So a row is spread over as many CTAs as its length and the number of rows
// allow (up to 16), and every row-wide step is one exchange:
//
//   load      one bulk copy per CTA, under way while the row's parameters and lists are read
//   process   penalties, biases, mask, temperature; fp32 values to shared memory, maxima
//   greedy    the largest (value, index) of the CTAs: done
//   top-k, small k    every warp (or part of a warp) publishes its maximum to all CTAs; the k-th largest of these
//             maxima is a value that at least k elements reach, and few more do (53 of 131072 for k = 50): those go to
//             CTA 0, which ranks them and finishes the row                                             (2 exchanges)
//   top-k, larger k   the same bound from a histogram of the lanes' maxima                            (4 exchanges)
//   top-p     the weights' own bits are the bins: 256 by exponent and leading mantissa bits, then 256 more inside the bin
//             where the mass from the top reaches p; its elements go to CTA 0, which finds the exact cut, the support's
//             mass and the CTA the draw falls into; that CTA finds the element                         (5 exchanges)
//   others    (min-p, no truncation): the cut is known from the maximum, one exchange of masses, then the draw
//
// A bin too crowded for CTA 0 is one value's ties almost always (low-precision logits): those are counted and ordered by
// index; anything else is split again over the (value, index) pairs it holds until it fits.  Every row is finished here,
// whatever its values.
// What it measured, against the chain of kernels of large calls (us per call): a bf16 row of 131072 with top-k 50, top-p
// 0.9 13.6 (25.5); 32 bf16 rows of 100003 with top-p or min-p only 49.3 (73.9); 37 fp32 rows of 50021 of every kind 36.4
// (64.3).  Its stalls are instruction fetch (8.1 of 23.1 cycles between two instructions of a warp, four rows of four kinds), barriers
// (3.6), loads (2.5) and fences (2.4): serial code, not bytes.
// Masses are integers, 2^-44 of the largest weight: sums do not depend on the order, replays are bit-identical.
#pragma once
#include <cooperative_groups.h>
#include "sonic_common.cuh"
#include "sonic_dense.cuh"
#include "sonic_stream.cuh"

namespace sonic {
namespace cgr = cooperative_groups;

constexpr int ROW_THREADS = 512;
constexpr int ROW_WARPS = ROW_THREADS / 32;
constexpr int ROW_CMIN = 4, ROW_CMAX = 16;        // CTAs per cluster
constexpr int ROW_SLICE_MAX = 16384;              // elements per CTA, at most (64 KB as fp32)
constexpr int ROW_UNIT = ROW_WARPS * 128;         // a slice is a multiple of this: every warp owns whole groups of 128
constexpr int ROW_BINS = 256;                     // bins of a level
constexpr int ROW_COPIES = 8;                     // copies of the bins, by lane: ties of one value share a bin, and atomics of
                                                  // a warp on one address take their turns (8 cycles each)
constexpr int ROW_XBINS = 128;                    // bins of a level over (value, index) pairs (exchanged as 64-bit words)
constexpr int ROW_LAND = 2944;                    // elements CTA 0 can receive
constexpr int ROW_MEMBERS = ROW_THREADS;          // ... of a top-p row's crossing bin (one per thread)
constexpr int ROW_GMAX = 256;                     // group maxima that are exchanged directly (a thread of kth_max counts half of them;
                                                  // with 512 it counts all: 8 bf16 rows of 50021 with k = 64 23 us, 15 with 256)
constexpr int ROW_DIRECT = 88;                    // largest k they serve: 108 of 256 groups' elements reach the bound then, give or take 8,
                                                  // and 128 are what the short finish takes (k = 100 reaches 127 and lies with the maxima of the lanes:
                                                  // 8 fp32 rows of 50021 23 -> 17 us)
constexpr int ROW_KMAX = 2048;                    // largest top-k finished from gathered elements
static_assert(ROW_SLICE_MAX * 4 >= MERGE_CAP * 8, "the epilogue's buffers take the values' place in CTA 0");
static_assert(ROW_KMAX <= KFAST_SAMPLE, "the epilogue's layout");
static_assert(ROW_THREADS == MERGE_THREADS, "the merge epilogue runs on the row kernel's CTAs");
static_assert(ROW_WARPS == ROW_CMAX, "half a warp: a lane per warp of the CTA, and per CTA of the cluster");

// CTA 0 -> all.  again: 0 finished, 1 split the part [lo, hi] (need: what it has to bring), 2 masses at or above cutc.
// tie_cta >= 0: the cut falls among the ties of the value with key cutc >> 32 (row_tie_cut).
constexpr int RB_DONE = 0, RB_SPLIT = 1, RB_MASS = 2;
constexpr unsigned int RB_ACCEPT = 1u, RB_REJECT = 2u;
struct RowBcast {
    unsigned long long cutc, W, rest, need, lo, hi;
    unsigned int owner, support, flags;
    int again;
    float p_draft;
    int tie_cta;
    unsigned int tie_in, pad;
};

struct RowShared {
    unsigned long long full;                      // mbarrier of the bulk copy
    unsigned int late[ROW_CMAX];                  // per CTA: its copy never came
    ulonglong2 ex1[ROW_CMAX];                     // per CTA: {max key << 32 | ~min finite key, best element or draft key}
    ulonglong2 above[ROW_CMAX];                   // CTA 0: per CTA {mass, number | members << 32}: what lies above the gathered part; its members
    unsigned long long sum[2][ROW_CMAX];          // per CTA: exact masses that go with a level (total; above the first level's bin)
    ulonglong2 span[ROW_CMAX];                    // splits: per CTA {smallest, largest} element of the part
    double resid[ROW_CMAX][3];
    RowBcast bc;
    unsigned int land_n, land_min, land_max;      // CTA 0: elements received, their smallest and largest key
    unsigned int cross_bin;
    double cross_before, cross_in;
    unsigned long long red64[ROW_WARPS], warp2[ROW_WARPS];       // (a search's scratch: both)
    unsigned int red32[ROW_WARPS];
    double redd[3][ROW_WARPS];                    // (a search's scratch: two rows)
    unsigned long long cta_mass[ROW_CMAX];
    union {
        unsigned int gmax[ROW_GMAX];              // group maxima of all CTAs (keys)
        unsigned long long bins[ROW_BINS];        // the CTA's own bins, folded
        unsigned long long list[ROW_THREADS];     // CTA 0: what it ranks
        MergeShared<ROW_THREADS> merge;
    };
};

// Dynamic shared memory: values | bins received | bins, landing zone | mask words | control.  The raw bf16 part is copied to
// the place of the two bin areas (and expanded before they are used); the landing zone takes the bins' place and 7 KB more
// (nobody sends to it before every CTA has folded its bins).  Every access names the array itself, so that it is compiled
// as a shared-memory access: through pointers kept in a structure they were generic loads and atomics, several times slower.
constexpr int ROW_OFF_RX = ROW_SLICE_MAX * 4, ROW_OFF_H = ROW_OFF_RX + ROW_CMAX * ROW_BINS * 4, ROW_OFF_MASK = ROW_OFF_H + ROW_LAND * 8,
              ROW_OFF_CTL = ROW_OFF_MASK + ROW_SLICE_MAX / 8, ROW_DYN_SMEM = ROW_OFF_CTL + (int)sizeof(RowShared);
static_assert(ROW_LAND * 8 >= ROW_BINS * ROW_COPIES * 8 && ROW_OFF_MASK - ROW_OFF_RX >= ROW_SLICE_MAX * 2, "areas share their place");
static_assert(ROW_XBINS * 8 <= ROW_BINS * 4, "bins received");
static_assert(ROW_CMAX * ROW_BINS >= MERGE_BUCKETS, "the sort's buckets take the place of the bins received");
static_assert(ROW_DYN_SMEM + 1024 <= 233472 / 2, "two CTAs per SM");
extern __shared__ __align__(128) unsigned char row_smem[];
__device__ __forceinline__ float *row_y() { return reinterpret_cast<float *>(row_smem); }                                       // [slice] the CTA's part of the row
__device__ __forceinline__ float *row_rx() { return reinterpret_cast<float *>(row_smem + ROW_OFF_RX); }                         // [ROW_CMAX][ROW_BINS]
__device__ __forceinline__ unsigned int *row_h() { return reinterpret_cast<unsigned int *>(row_smem + ROW_OFF_H); }              // [2][ROW_BINS][ROW_COPIES]
__device__ __forceinline__ unsigned long long *row_land() { return reinterpret_cast<unsigned long long *>(row_smem + ROW_OFF_H); }      // [ROW_LAND]
__device__ __forceinline__ uint32_t *row_mask() { return reinterpret_cast<uint32_t *>(row_smem + ROW_OFF_MASK); }               // [slice / 32]
__device__ __forceinline__ RowShared &row_sh() { return *reinterpret_cast<RowShared *>(row_smem + ROW_OFF_CTL); }

__device__ __forceinline__ void cl_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_sync() { cl_arrive(); cl_wait(); }
template <typename T> __device__ __forceinline__ T *cl_map(T *p, int rank) { return cgr::this_cluster().map_shared_rank(p, rank); }

__device__ __forceinline__ unsigned long long row_comp(uint32_t key, int idx) {
    return ((unsigned long long)key << 32) | (uint32_t)(~(uint32_t)idx);
}
__device__ __forceinline__ unsigned long long row_elem(float y, int idx) { return row_comp(okey(y), idx); }

// Running context of a row in one CTA.  Values past the row's end are NaN: they fail every comparison.
struct RowCtx {
    int rank, ncta, slice, base;                  // base: vocabulary index of the part's first element
    int tid, lane, warp, wlo, wn;                 // the warp's elements: [wlo, wlo + wn)
    float Mf;                                     // row maximum
};

// The bound of a row's small top-k where its quotient by the temperature is far from the ordinary (subnormal, overflowing, or none).
// Ordinary quotients that are equal come from values within 2^-22 of each other; with the exact bound on that path as well a bf16 row of
// 131072 takes 13.8 instead of 13.0 us.  (One division and two searches for a neighbour: code that runs once, fetched cold.)
__device__ __noinline__ float row_bound_before_div(float t, float tau) {
    const float low = first_finite_quotient(tau);
    return t > low ? fmaxf(bound_before_div(t, tau), low) : low;
}

// Four elements at a time over the warp's part, index order across the lanes: f(value, vocabulary index).
template <typename F>
__device__ __forceinline__ void row_each(const RowCtx &x, F f) {
#pragma unroll 2
    for (int i = x.wlo + x.lane * 4; i < x.wlo + x.wn; i += 128) {
        const float4 v = *reinterpret_cast<const float4 *>(row_y() + i);
        f(v.x, x.base + i); f(v.y, x.base + i + 1); f(v.z, x.base + i + 2); f(v.w, x.base + i + 3);
    }
}

// ---------------------------------------------------------------- weights
// An element's weight exp(y - M) as qweight has it (the same operations, before the conversion).
__device__ __forceinline__ float row_w(float y, float Mf) {
    const float d = __fsub_rn(y, Mf);
    const float L1 = 1.44269502162933349609375f;        // fp32(log2 e)
    const float L2 = 1.925963033500011e-08f;            // log2 e - L1
    float w;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(fmaf(d, L1, d * L2)));
    return w;
}
// ... as an integer, 2^-44 of the largest.  The weight of a NaN (past the row's end) converts to 2^63: every sum takes elements
// of at least vmin alone, which a NaN is not.
constexpr double ROW_Q1 = 17592186044416.0;              // 2^44
__device__ __forceinline__ unsigned long long row_q(float w) { return __float2ull_rz(w * 17592186044416.0f); }
// Weights below 2^-41 count as nothing (their fixed-point value was 0 before it was refined to 2^-44).
constexpr uint32_t ROW_WMIN = (127u - 41u) << 23;

// What takes part in a row's truncation: values of at least vmin (all finite ones, or -inf too), and with `cut` only the
// elements at or above `base`.
struct RowSel {
    unsigned long long base, lo, hi;              // [lo, hi]: the part of the row a split has narrowed a selection down to
    float vmin;
    bool cut;
};
__device__ __forceinline__ bool row_in(const RowSel &s, float y, int idx) {
    return y >= s.vmin && (!s.cut || row_elem(y, idx) >= s.base);
}

// ---------------------------------------------------------------- levels
// A level: every CTA adds its elements to ROW_COPIES copies of the bins, folds them, sends them to all CTAs, and after one
// cluster barrier every CTA adds up what it received and finds the bin where the running total from bin 0 reaches the target.
__device__ __forceinline__ void row_zero_bins(const RowCtx &x) {
    for (int i = x.tid; i < ROW_BINS * ROW_COPIES * 2 / 4; i += ROW_THREADS) reinterpret_cast<uint4 *>(row_h())[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
}
// A weight's 24 mantissa bits as two 12-bit halves: two 32-bit reductions without a return value, exact sums (a part has at
// most 2^14 elements).
__device__ __forceinline__ void row_add_weight(uint32_t bits, int bin, int lane) {
    const uint32_t mant = (bits & 0x7FFFFFu) | 0x800000u;
    unsigned int *h = row_h() + bin * ROW_COPIES + (lane & (ROW_COPIES - 1));
    atomicAdd(h, mant & 0xFFFu);
    atomicAdd(h + ROW_BINS * ROW_COPIES, mant >> 12);
}
// Folds the bins and sends them to all CTAs as floats (they decide where to look; the exact sums stay behind in sh.bins).
// oct(bin): for weights, the octave below 2 that the bin's weights lie in; counts: WEIGHTS == false.  Needs a block barrier
// before, a cluster barrier after.
template <bool WEIGHTS, typename OF>
__device__ __forceinline__ void row_fold(const RowCtx &x, bool wait, OF oct) {
    RowShared &sh = row_sh();
    const int bin = x.tid >> 1, word = x.tid & 1;
    static_assert(ROW_BINS * 2 == ROW_THREADS && ROW_COPIES == 8, "two threads per bin, eight copies");
    const uint4 a = reinterpret_cast<const uint4 *>(row_h() + word * ROW_BINS * ROW_COPIES + bin * ROW_COPIES)[0];
    const uint4 b = reinterpret_cast<const uint4 *>(row_h() + word * ROW_BINS * ROW_COPIES + bin * ROW_COPIES)[1];
    const unsigned int mine = (a.x + a.y) + (a.z + a.w) + (b.x + b.y) + (b.z + b.w), other = __shfl_xor_sync(0xFFFFFFFFu, mine, 1);
    unsigned long long s = word ? ((unsigned long long)mine << 12) + other : mine + ((unsigned long long)other << 12);
    if (WEIGHTS) {
        const int up = 21 - oct(bin);                               // mantissa * 2^(-octave - 23), in units of 2^-44
        s = up >= 0 ? s << up : s >> -up;
    } else s = word ? other : mine;
    if (word == 0) sh.bins[bin] = s;
    const float f = (float)s;
    if (wait) cl_wait();                                            // (every CTA has read the last level's bins)
    float *rx = row_rx() + x.rank * ROW_BINS + bin;
    for (int r = word; r < x.ncta; r += 2) *cl_map(rx, r) = f;
}
// The received bins: the bin where the running total reaches `want` (clipped to the total), the total before it and the
// bin's own.  Two block barriers.  Returns false if the total is below `want`.  next: another level follows - arrives at the
// cluster barrier once the received bins are read, the next row_fold waits there before it sends.
__device__ __forceinline__ bool row_cross(const RowCtx &x, bool next, double want, int &bin, double &before, double &in_bin) {
    RowShared &sh = row_sh();
    float v = 0.0f;
    if (x.tid < ROW_BINS) {
#pragma unroll
        for (int r = 0; r < ROW_CMAX; ++r) v += (r < x.ncta) ? row_rx()[r * ROW_BINS + x.tid] : 0.0f;
    }
    if (next) cl_arrive();
    double incl = (double)v;
    if (x.tid < ROW_BINS) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const double up = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (x.lane >= o) incl += up; }
        if (x.lane == 31) sh.redd[0][x.warp] = incl;
    }
    __syncthreads();
    double pre = 0.0, all = 0.0;
#pragma unroll
    for (int w = 0; w < ROW_BINS / 32; ++w) { const double t = sh.redd[0][w]; if (w < x.warp) pre += t; all += t; }
    const double need = fmin(want, all);
    if (x.tid < ROW_BINS) {
        // (the same additions on both sides of a bin's edge: exactly one bin has need in (lo, hi])
        const double hi = pre + incl, up = __shfl_up_sync(0xFFFFFFFFu, hi, 1), lo = x.lane ? up : pre;
        if (lo < need && need <= hi) { sh.cross_bin = x.tid; sh.cross_before = lo; sh.cross_in = (double)v; }
    }
    __syncthreads();
    bin = (int)sh.cross_bin; before = sh.cross_before; in_bin = sh.cross_in;
    return all >= want;
}
// Exact sum of the CTA's own bins below `n`, in every thread of warp 0 (the others: undefined).  One block barrier.
__device__ __forceinline__ unsigned long long row_sum_bins(const RowCtx &x, int n) {
    RowShared &sh = row_sh();
    if (x.tid < ROW_BINS) {
        const unsigned long long t = dense_warp_sum(x.tid < n ? sh.bins[x.tid] : 0ull);
        if (x.lane == 0) sh.red64[x.warp] = t;
    }
    __syncthreads();
    unsigned long long s = 0ull;
    if (x.warp == 0) {
#pragma unroll
        for (int w = 0; w < ROW_BINS / 32; ++w) s += sh.red64[w];
    }
    return s;
}

// Splits the part [s.lo, s.hi]: ROW_XBINS bins over the (key, index) pairs it spans, by mass or by count, exact.  `need`
// counts from the top of the part.  Each call divides the span by 128, so ten calls end in a part of one element.
__device__ __noinline__ void row_split(const RowCtx &ctx, RowSel &sel, bool by_mass, unsigned long long &need, unsigned long long &in_part) {
    const RowCtx x = ctx;                                           // (copies: through the references every access would go to memory)
    RowSel s = sel;
    RowShared &sh = row_sh();
    unsigned long long mn = ~0ull, mx = 0ull;
    row_each(x, [&](float y, int idx) {
        const unsigned long long c = row_elem(y, idx);
        if (row_in(s, y, idx) && c >= s.lo && c <= s.hi) { mn = min(mn, c); mx = max(mx, c); }
    });
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, off));
        mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    }
    if (x.lane == 0) { sh.red64[x.warp] = mn; sh.warp2[x.warp] = mx; }
    row_zero_bins(x);
    if (x.tid < x.ncta) {
        for (int w = 0; w < ROW_WARPS; ++w) { mn = min(mn, sh.red64[w]); mx = max(mx, sh.warp2[w]); }
        *cl_map(&sh.span[x.rank], x.tid) = make_ulonglong2(mn, mx);
    }
    cl_sync();
    mn = ~0ull; mx = 0ull;
    for (int r = 0; r < x.ncta; ++r) { mn = min(mn, sh.span[r].x); mx = max(mx, sh.span[r].y); }
    const int shift = max(0, 64 - __clzll((long long)(mx - mn)) - 7);
    const float Mf = x.Mf;
    unsigned int *h = row_h();
    row_each(x, [&](float y, int idx) {
        const unsigned long long c = row_elem(y, idx);
        if (row_in(s, y, idx) && c >= mn && c <= mx) {
            const int d = (int)((mx - c) >> shift);
            const unsigned long long q = by_mass ? row_q(row_w(y, Mf)) : 1ull;
            // 64 bits as two words: the low word's old value reveals a carry
            const unsigned int lo = (unsigned int)q, hi = (unsigned int)(q >> 32);
            unsigned int carry = 0u;
            if (lo) { const unsigned int old = atomicAdd(&h[d], lo); carry = (old + lo < old) ? 1u : 0u; }
            if (hi + carry) atomicAdd(&h[ROW_XBINS + d], hi + carry);
        }
    });
    __syncthreads();
    {
        const int d = x.tid & (ROW_XBINS - 1);
        const unsigned long long v = ((unsigned long long)h[ROW_XBINS + d] << 32) + h[d];
        for (int r = x.tid / ROW_XBINS; r < x.ncta; r += ROW_THREADS / ROW_XBINS) *cl_map(reinterpret_cast<unsigned long long *>(row_rx()) + x.rank * ROW_XBINS + d, r) = v;
    }
    cl_sync();
    // every warp: four bins per lane
    unsigned long long v[4], run = 0ull;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        v[u] = 0ull;
        for (int r = 0; r < x.ncta; ++r) v[u] += reinterpret_cast<const unsigned long long *>(row_rx())[r * ROW_XBINS + x.lane * 4 + u];
        run += v[u];
    }
    const unsigned long long incl = dense_warp_scan(run, x.lane), all = __shfl_sync(0xFFFFFFFFu, incl, 31), want = max(1ull, min(need, all));
    const unsigned int hit = __ballot_sync(0xFFFFFFFFu, incl >= want);
    const int l = hit ? __ffs(hit) - 1 : 31;
    unsigned long long before = incl - run, in = 0ull;
    int at = 0;
    bool found = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (!found) { if (before + v[u] >= want) { found = true; at = u; in = v[u]; } else before += v[u]; }
    }
    const int d = __shfl_sync(0xFFFFFFFFu, x.lane * 4 + at, l);
    before = __shfl_sync(0xFFFFFFFFu, before, l);
    in_part = __shfl_sync(0xFFFFFFFFu, in, l);
    need = want > before ? want - before : 1ull;
    s.hi = mx - ((unsigned long long)d << shift);
    const unsigned long long down = (1ull << shift) - 1ull;
    s.lo = (s.hi - mn > down) ? s.hi - down : mn;
    sel = s;
    __syncthreads();                                                // (red64, the bins: used again)
}

// Room for `mine` elements of every lane in CTA 0's landing zone: one remote atomic per warp that sends anything.
__device__ __forceinline__ unsigned int row_room(const RowCtx &x, unsigned int mine, bool &any) {
    unsigned int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const unsigned int up = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (x.lane >= o) incl += up; }
    const unsigned int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    any = total != 0u;
    unsigned int pos = 0u;
    if (any) {
        if (x.lane == 0) pos = atomicAdd(cl_map(&row_sh().land_n, 0), total);
        pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + incl - mine;
    }
    return pos;
}
// The warps' sums of a mass, a number and a number of members -> this CTA's entry of CTA 0's sh.above (block barrier inside).
__device__ __forceinline__ void row_send_above(const RowCtx &x, unsigned long long m, unsigned int n, unsigned int members, unsigned long long more) {
    RowShared &sh = row_sh();
    m = dense_warp_sum(m);
    const unsigned int both = __reduce_add_sync(0xFFFFFFFFu, n | (members << 16));      // (a warp has at most 1024 elements)
    if (x.lane == 0) { sh.warp2[x.warp] = m; sh.red32[x.warp] = both; }
    __syncthreads();
    if (x.warp == 0) {
        m = dense_warp_sum(x.lane < ROW_WARPS ? sh.warp2[x.lane] : 0ull);
        const unsigned int t = x.lane < ROW_WARPS ? sh.red32[x.lane] : 0u;
        n = __reduce_add_sync(0xFFFFFFFFu, t & 0xFFFFu);
        members = __reduce_add_sync(0xFFFFFFFFu, t >> 16);
        if (x.lane == 0) *cl_map(&sh.above[x.rank], 0) = make_ulonglong2(m + more, (unsigned long long)n | ((unsigned long long)members << 32));
    }
}
// Elements of a level's bin (their weights' bits, shifted, equal `code`) to CTA 0, and their number and that of the elements
// above; `more`: the exact mass above (warp 0).  One pass marks the bin's elements in a bit per element of the lane, the few
// that are marked are then fetched again.  The caller's cluster barrier completes it.
__device__ __forceinline__ void row_gather_bin(const RowCtx &x, const RowSel &s, int shift, int code, unsigned long long more) {
    RowShared &sh = row_sh();
    const float Mf = x.Mf;
    unsigned int an = 0u, hits = 0u;
    int bit = 0;
    static_assert(ROW_SLICE_MAX / ROW_THREADS <= 32, "a bit per element of a lane");
    row_each(x, [&](float y, int idx) {
        const int d = (int)((0x3FFFFFFFu - __float_as_uint(row_w(y, Mf))) >> shift);
        const bool in = y >= s.vmin && d <= code && (!s.cut || row_elem(y, idx) >= s.base);
        an += (in && d < code) ? 1u : 0u;
        hits |= (in && d == code) ? (1u << bit) : 0u;
        ++bit;
    });
    const unsigned int mine = (unsigned int)__popc(hits);
    bool any;
    unsigned int pos = row_room(x, mine, any);
    if (any) {
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
        unsigned long long *land = cl_map(row_land(), 0);
        while (hits) {
            const int b = __ffs(hits) - 1, li = x.wlo + (b >> 2) * 128 + x.lane * 4 + (b & 3);
            hits &= hits - 1u;
            const unsigned long long c = row_elem(row_y()[li], x.base + li);
            mn = min(mn, (uint32_t)(c >> 32)); mx = max(mx, (uint32_t)(c >> 32));
            if (pos < (unsigned int)ROW_MEMBERS) land[pos] = c;
            ++pos;
        }
        __syncwarp();
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (x.lane == 0) { atomicMin(cl_map(&sh.land_min, 0), mn); atomicMax(cl_map(&sh.land_max, 0), mx); }
    }
    row_send_above(x, 0ull, an, mine, more);
}
// Elements of the part [s.lo, s.hi] to CTA 0; mass and number of those above it.  MASS: also when the part is empty.
__device__ __noinline__ void row_gather_part(const RowCtx &ctx, const RowSel &sel) {
    const RowCtx x = ctx;
    const RowSel s = sel;
    RowShared &sh = row_sh();
    const float Mf = x.Mf;
    unsigned long long am = 0ull;
    unsigned int an = 0u, mine = 0u;
    row_each(x, [&](float y, int idx) {
        const unsigned long long c = row_elem(y, idx);
        if (row_in(s, y, idx) && c >= s.lo) {
            if (c > s.hi) { am += row_q(row_w(y, Mf)); ++an; } else ++mine;
        }
    });
    bool any;
    unsigned int pos = row_room(x, mine, any);
    if (any) {
        uint32_t mn = 0xFFFFFFFFu, mx = 0u;
        unsigned long long *land = cl_map(row_land(), 0);
        row_each(x, [&](float y, int idx) {
            const unsigned long long c = row_elem(y, idx);
            if (row_in(s, y, idx) && c >= s.lo && c <= s.hi) {
                mn = min(mn, (uint32_t)(c >> 32)); mx = max(mx, (uint32_t)(c >> 32));
                if (pos < (unsigned int)ROW_MEMBERS) land[pos] = c;
                ++pos;
            }
        });
        __syncwarp();
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (x.lane == 0) { atomicMin(cl_map(&sh.land_min, 0), mn); atomicMax(cl_map(&sh.land_max, 0), mx); }
    }
    row_send_above(x, am, an, mine, 0ull);
}
// Mass and number of the elements at or above cutc.
__device__ __noinline__ void row_mass_above(const RowCtx &ctx, float vmin, unsigned long long cutc) {
    const RowCtx x = ctx;
    const float Mf = x.Mf;
    unsigned long long am = 0ull;
    unsigned int an = 0u;
    const uint32_t ckey = (uint32_t)(cutc >> 32);
    const float cy = fmaxf(unkey(ckey), vmin);
    const bool whole = (uint32_t)cutc == 0u;                        // the cut is a value: every element of it is in
    row_each(x, [&](float y, int idx) {
        const unsigned long long q = row_q(row_w(y, Mf));
        bool in = y >= cy;
        if (!whole) in = in && row_elem(y, idx) >= cutc;
        am += in ? q : 0ull;
        an += in ? 1u : 0u;
    });
    row_send_above(x, am, an, 0u, 0ull);
}
// CTA 0's word to all, then a cluster barrier (bc: the same in every thread of CTA 0).
__device__ __forceinline__ void row_broadcast(const RowCtx &x, const RowBcast &bc) {
    RowShared &sh = row_sh();
    if (x.rank == 0) {
        if (x.tid == 0) { sh.land_n = 0u; sh.land_min = 0xFFFFFFFFu; sh.land_max = 0u; }
        if (x.tid < x.ncta) *cl_map(&sh.bc, x.tid) = bc;
    }
    cl_sync();
}

// Top-k selection by count: bins uniform in M - y.  lane_max: only the lanes' maxima are counted (k of them at or above a
// bin mean at least k elements there, and with many more lanes than k hardly more): 1/16 to 1/32 of the work.
// Returns the number of elements (or maxima) above the bin and in it; false if there are fewer than k in all.
__device__ __forceinline__ int row_count_bin(float y, float Mf, float scale) {
    return (int)fminf(__fmul_rn(__fsub_rn(Mf, y), scale), (float)(ROW_BINS - 1));
}
__device__ __forceinline__ bool row_level_count(const RowCtx &x, const RowSel &s, bool lane_max, float lmax, uint32_t kmin, int k, float &scale,
                                                int &bin, unsigned int &above, unsigned int &inside) {
    row_zero_bins(x);
    // the row's finite range, 128 units below the maximum at most
    const float spread = (okey(x.Mf) >= kmin) ? fminf(__fsub_rn(x.Mf, unkey(kmin)), 128.0f) : 0.0f;
    const float Mf = x.Mf;
    scale = (spread > 0.0f) ? fminf(__fdividef((float)(ROW_BINS - 2), spread), 16384.0f) : 32.0f;
    const float sc = scale;
    unsigned int *h = row_h() + (x.lane & (ROW_COPIES - 1));
    if (lane_max) {
        if (lmax >= s.vmin) atomicAdd(&h[row_count_bin(lmax, Mf, sc) * ROW_COPIES], 1u);
    } else {
        row_each(x, [&](float y, int idx) {
            const int b = row_count_bin(y, Mf, sc);
            if (row_in(s, y, idx)) atomicAdd(&h[b * ROW_COPIES], 1u);
        });
    }
    __syncthreads();
    row_fold<false>(x, false, [](int) { return 0; });
    cl_sync();
    double before, in_bin;
    const bool enough = row_cross(x, false, (double)k, bin, before, in_bin);
    above = (unsigned int)before; inside = (unsigned int)in_bin;
    return enough;
}
// Everything in that bin or above it to CTA 0.
__device__ __forceinline__ void row_gather_count(const RowCtx &x, const RowSel &s, float scale, int bin, unsigned long long floorc) {
    const float Mf = x.Mf, limit = (bin == ROW_BINS - 1) ? CUDART_INF_F : (float)(bin + 1);       // (int)min(u, 255) <= bin  <=>  u < bin + 1
    unsigned int mine = 0u;
    auto in = [&](float y, int idx) -> bool {
        const float u = __fmul_rn(__fsub_rn(Mf, y), scale);
        return y >= s.vmin && !(u >= limit && limit < CUDART_INF_F) && (floorc == 0ull || row_elem(y, idx) >= floorc);
    };
    row_each(x, [&](float y, int idx) { mine += in(y, idx) ? 1u : 0u; });
    bool any;
    unsigned int pos = row_room(x, mine, any);
    if (any && mine) {
        unsigned long long *land = cl_map(row_land(), 0);
        row_each(x, [&](float y, int idx) {
            if (in(y, idx)) { if (pos < (unsigned int)ROW_LAND) land[pos] = row_elem(y, idx); ++pos; }
        });
    }
    __syncwarp();
}

template <typename T>
__device__ __forceinline__ T row_lane_scan(T v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const T up = __shfl_up_sync(0xFFFFFFFFu, v, o); if (lane >= o) v += up; }
    return v;
}
// The element, in index order, at which the running weight of the CTA's part first exceeds `rest`: the warp whose part it
// is, then that part spread over the whole CTA (one or two consecutive elements per thread).  wf(value, index) -> weight,
// T integer or fp64; wtot: 2 * ROW_WARPS words.  f(index, weight) is called by one thread of the CTA (for the last element of
// positive weight if rounding keeps the sum below `rest`; not at all if there is none).  Three block barriers.
template <typename T, typename WF, typename F>
__device__ __forceinline__ void row_find(const RowCtx &x, T rest, T *wtot, WF wf, F f) {
    T s = T(0);
    row_each(x, [&](float y, int idx) { s += wf(y, idx); });
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
    __syncthreads();
    if (x.lane == 0) wtot[x.warp] = s;
    __syncthreads();
    const T tw = (x.lane < ROW_WARPS) ? wtot[x.lane] : T(0);
    T incl = row_lane_scan<T>(tw, x.lane);
    const unsigned int pos = __ballot_sync(0xFFFFFFFFu, tw > T(0)), hit = __ballot_sync(0xFFFFFFFFu, tw > T(0) && incl > rest);
    if (!pos) return;
    const int w = hit ? __ffs(hit) - 1 : 31 - __clz(pos);           // (no hit: floating-point sums, past the end by rounding)
    rest -= __shfl_sync(0xFFFFFFFFu, incl - tw, w);
    const int per = (x.wn > ROW_THREADS) ? 2 : 1, li = w * x.wn + x.tid * per;
    const bool mine = x.tid * per < x.wn;
    const T a = mine ? wf(row_y()[li], x.base + li) : T(0), b = (mine && per == 2) ? wf(row_y()[li + 1], x.base + li + 1) : T(0);
    incl = row_lane_scan<T>(a + b, x.lane);
    if (x.lane == 31) wtot[ROW_WARPS + x.warp] = incl;
    __syncthreads();
    const T t2 = (x.lane < ROW_WARPS) ? wtot[ROW_WARPS + x.lane] : T(0), i2 = row_lane_scan<T>(t2, x.lane);
    const T hi = incl + __shfl_sync(0xFFFFFFFFu, i2 - t2, x.warp), lo = hi - (a + b);
    // the first element in index order that takes the sum beyond `rest`, else the last of positive weight
    const unsigned int over = __ballot_sync(0xFFFFFFFFu, t2 > T(0) && i2 > rest), some = __ballot_sync(0xFFFFFFFFu, t2 > T(0));
    const unsigned int mh = __ballot_sync(0xFFFFFFFFu, a + b > T(0) && hi > rest), mp = __ballot_sync(0xFFFFFFFFu, a + b > T(0));
    if (x.warp != (over ? __ffs(over) - 1 : 31 - __clz(some))) return;
    if (x.lane == (mh ? __ffs(mh) - 1 : 31 - __clz(mp))) {
        const bool first = a > T(0) && (lo + a > rest || !(b > T(0)));
        f(x.base + li + (first ? 0 : 1), first ? a : b);
    }
}

// Ranks the n <= ROW_THREADS elements CTA 0 has received: the thread's element and its weight in descending order (0 past
// the end).
__device__ __forceinline__ void row_rank(const RowCtx &x, int n, unsigned long long &c, unsigned long long &w) {
    unsigned long long *comp = &row_sh().list[0];
    comp[x.tid] = (x.tid < n) ? row_land()[x.tid] : 0ull;
    __syncthreads();
    int rank;
    const unsigned long long key = rank_keys<ROW_THREADS, BlockSync>(comp, n, x.tid, rank);
    __syncthreads();                                                // every search has read the runs
    if (key) comp[rank] = key;
    __syncthreads();
    c = (x.tid < n) ? comp[x.tid] : 0ull;
    w = c ? row_q(row_w(unkey((uint32_t)(c >> 32)), x.Mf)) : 0ull;
}

// The cut of this CTA's part when the cut falls among the ties of one value, by index: all of them are in before CTA
// `tie_cta`, none behind it, its own first `tie_in` there.  (Called by the whole CTA; block barriers in that CTA alone.)
__device__ __forceinline__ unsigned long long row_tie_cut(const RowCtx &x, const RowSel &s, uint32_t v, int tie_cta, unsigned int tie_in) {
    if (x.rank != tie_cta) return ((unsigned long long)v + (x.rank > tie_cta ? 1ull : 0ull)) << 32;
    RowShared &sh = row_sh();
    const float vy = unkey(v);
    row_find<unsigned int>(x, tie_in - 1u, reinterpret_cast<unsigned int *>(sh.red64),
                           [&](float y, int idx) -> unsigned int { return (y == vy && row_in(s, y, idx)) ? 1u : 0u; },
                           [&](int idx, unsigned int) { sh.span[0].x = row_comp(v, idx); });
    __syncthreads();
    return sh.span[0].x;
}

// Whether some CTA's copy never came (checked after the first exchange).
__device__ __forceinline__ bool row_late(const RowCtx &x) {
    return __any_sync(0xFFFFFFFFu, x.lane < x.ncta && row_sh().late[x.lane] != 0u);
}

// Requests of a verification call: the last position to be finished scans all of them (ticket: zero between calls).
__device__ __forceinline__ void verify_combine(const KParams &P, int b);
__device__ __forceinline__ void row_ticket(const KParams &P, int b) {
    __threadfence();
    if (atomicAdd(&P.tickets[b], 1u) == (unsigned int)P.K) {
        __threadfence();
        P.tickets[b] = 0u;
        verify_combine(P, b);
    }
}

// Residual of a rejected draft: max(0, p - q) summed over the CTAs in fp64 with the support's mass W~ in fixed point,
// corrected by the exact W (resid_weight has the derivation), then the draw.
__device__ __noinline__ bool row_residual(const RowCtx &ctx, const KParams &P, const RowCfg &c, unsigned long long cutc, unsigned long long Wq, uint32_t a_draw,
                             int &token) {
    const RowCtx x = ctx;
    RowShared &sh = row_sh();
    const float Mf = x.Mf;
    const double Md = (double)Mf;
    const double inv_Wt = ROW_Q1 / (double)Wq;
    const float big = (float)((double)Wq * (1.0 / ROW_Q1) * (1.0 / 128.0));
    const float *q = P.draft_probs + ((size_t)c.b * P.K + c.l) * (size_t)P.V;
    double R = 0.0, Pp = 0.0, S = 0.0;
    auto weight = [&](float y, int idx) -> double {
        const uint32_t key = okey(y);
        return (y >= -CUDART_MAX_NORMAL_F && row_comp(key, idx) >= cutc) ? resid_weight(key, Mf, Md, big) : 0.0;
    };
    row_each(x, [&](float y, int idx) {
        const double w = weight(y, idx);
        const double r = w * inv_Wt - (double)__ldg(q + min(idx, P.V - 1));
        S += w;
        R += (r > 0.0) ? r : 0.0;
        Pp += (r > 0.0) ? w : 0.0;
    });
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        R += __shfl_xor_sync(0xFFFFFFFFu, R, off);
        Pp += __shfl_xor_sync(0xFFFFFFFFu, Pp, off);
        S += __shfl_xor_sync(0xFFFFFFFFu, S, off);
    }
    if (x.lane == 0) { sh.redd[0][x.warp] = R; sh.redd[1][x.warp] = Pp; sh.redd[2][x.warp] = S; }
    __syncthreads();
    if (x.tid < x.ncta) {
        R = Pp = S = 0.0;
        for (int w = 0; w < ROW_WARPS; ++w) { R += sh.redd[0][w]; Pp += sh.redd[1][w]; S += sh.redd[2][w]; }
        double *to = cl_map(&sh.resid[x.rank][0], x.tid);
        to[0] = R; to[1] = Pp; to[2] = S;
    }
    cl_sync();
    double W = 0.0;
    for (int r = 0; r < x.ncta; ++r) W += sh.resid[r][2];
    const double corr = inv_Wt - 1.0 / W;
    double tot = 0.0;
    for (int r = 0; r < x.ncta; ++r) tot += fmax(sh.resid[r][0] - corr * sh.resid[r][1], 0.0);
    if (!(tot > 0.0)) return false;                                 // p <= q on the whole support, by rounding: the draw is from p itself
    double rest = cell_to_u(a_draw) * tot;
    int owner = -1, last = 0;
    for (int r = 0; r < x.ncta; ++r) {
        const double t = fmax(sh.resid[r][0] - corr * sh.resid[r][1], 0.0);
        if (t > 0.0) last = r;
        if (owner < 0 && t > 0.0) { if (rest < t) owner = r; else rest -= t; }
    }
    if (owner < 0) owner = last;
    if (owner == x.rank) {
        const double inv_W = 1.0 / W;
        if (x.tid == 0) sh.land_n = 0u;                             // (not needed any more: set by the thread that finds the token)
        row_find<double>(x, rest, sh.redd[0], [&](float y, int idx) -> double {
            const double r = weight(y, idx) * inv_W - (double)__ldg(q + min(idx, P.V - 1));
            return r > 0.0 ? r : 0.0;
        }, [&](int idx, double) { token = idx; sh.land_n = 1u; });
        __syncthreads();
        // the part's residual was the correction's rounding alone: its first element of the support
        if (sh.land_n == 0u)
            row_find<unsigned long long>(x, 0ull, sh.red64, [&](float y, int idx) -> unsigned long long {
                return (y >= -CUDART_MAX_NORMAL_F && row_elem(y, idx) >= cutc) ? row_q(row_w(y, Mf)) : 0ull;
            }, [&](int idx, unsigned long long) { token = idx; });
    }
    return true;
}


// Grid: rows x CTAs of a cluster.  slice: elements per CTA (a multiple of ROW_UNIT, slice * cluster >= V).
template <int DT>
__global__ void __launch_bounds__(ROW_THREADS, 2)
sonic_row_kernel(const __grid_constant__ KParams P, const int slice) {
    constexpr int VEC = VecTraits<DT>::VEC, ELT = VecTraits<DT>::ELT;
    RowShared &sh = row_sh();
    RowCtx x;
    x.rank = (int)cgr::this_cluster().block_rank();
    x.ncta = (int)cgr::this_cluster().num_blocks();
    x.slice = slice;
    x.base = x.rank * slice;
    x.tid = threadIdx.x; x.lane = x.tid & 31; x.warp = x.tid >> 5;
    x.wn = slice / ROW_WARPS; x.wlo = x.warp * x.wn;
    uint32_t *mask = row_mask();
    unsigned char *raw = row_smem + (DT == 0 ? 0 : ROW_OFF_RX);
    const int row = (int)blockIdx.x / x.ncta;
    const int tid = x.tid, lane = x.lane;
    const bool lead = x.rank == 0 && tid == 0;

    const CfgRaw cfg_raw = fetch_cfg(P, row);
    const int req = (P.op == OP_VERIFY) ? row / (P.K + 1) : row;
    // Everything the row needs from global memory is asked for at once: its logits by one bulk copy, mask words,
    // parameters and the first entries of its lists (none of the addresses depends on a loaded value).
    if (tid == 0) {
        mbar_init(&sh.full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const int elems = min(slice, (P.V - x.base + VEC - 1) / VEC * VEC);
        if (elems > 0) {
            mbar_arrive_expect_tx(&sh.full, (unsigned int)elems * ELT);
#ifdef SONIC_TEST_WITHHOLD
            // test-only build: the bytes of one chosen part of a row are announced but its copy is never issued
            if (__ldcg(&P.error[WS_TEST_WITHHOLD]) != (unsigned int)(row * ROW_CMAX + x.rank) + 1u)
#endif
            bulk_load(raw, reinterpret_cast<const unsigned char *>(P.logits) + ((size_t)row * (size_t)P.row_stride + (size_t)x.base) * ELT,
                      (unsigned int)elems * ELT, &sh.full, l2_evict_first_policy());
        } else mbar_arrive(&sh.full);
        sh.land_n = 0u; sh.land_min = 0xFFFFFFFFu; sh.land_max = 0u;
    }
    if (tid < ROW_CMAX) sh.late[tid] = 0u;
    if (tid < ROW_GMAX) sh.gmax[tid] = 0u;
    if (P.bitmask) {
        const int w = (x.base >> 5) + tid;
        if (tid < slice / 32) mask[tid] = (w < ((P.V + 31) >> 5)) ? __ldg(P.bitmask + (size_t)row * P.bitmask_stride + w) : 0u;
    }
    const int *hid = P.hist_ids ? P.hist_ids + (size_t)req * P.hist_stride : nullptr;
    const int *hct = P.hist_counts ? P.hist_counts + (size_t)req * P.hist_stride : nullptr;
    const int *bid = P.bias_ids ? P.bias_ids + (size_t)req * P.bias_stride : nullptr;
    const float *bvl = P.bias_vals ? P.bias_vals + (size_t)req * P.bias_stride : nullptr;
    int h_id = -1, h_ct = 0, b_id = -1;
    float b_vl = 0.0f;
    if (hid && hct && tid < P.hist_stride) { h_id = __ldg(hid + tid); h_ct = __ldg(hct + tid); }
    if (bid && bvl && tid < P.bias_stride) { b_id = __ldg(bid + tid); b_vl = __ldg(bvl + tid); }
    const unsigned int err = P.fresh ? 0u : __ldcg(&P.error[WS_ERROR]);
    const unsigned long long seed = P.seed ? __ldg(P.seed + req) : 0ull, offset = P.offset ? __ldg(P.offset + req) : 0ull;
    int draft = -1;
    float q_draft = 0.0f;
    {
        const int l = row - req * (P.K + 1);
        if (P.op == OP_VERIFY && l < P.K) {
            draft = __ldg(P.draft_tokens + (size_t)req * P.K + l);
            if (draft < 0 || draft >= P.V) draft = -1;
            if (draft >= 0) q_draft = __ldg(P.draft_probs + ((size_t)req * P.K + l) * (size_t)P.V + draft);
        }
    }
    __syncthreads();
    cl_arrive();                                                    // (matched by the wait before the first remote write)
    const RowCfg c = resolve_cfg(P, row, cfg_raw);
    const bool finish_request = P.op == OP_VERIFY;
    // (sonic_topk comes here with k up to ROW_KMAX alone and is always finished from gathered elements, also where its class in
    // the streaming chain is the cluster kernel's: vocabularies just above MERGE_CAP with k beyond an eighth of them)
    const bool dense = c.cls == CLS_DENSE || (c.cls == CLS_EXACT && P.op != OP_TOPK), greedy = c.cls == CLS_GREEDY;
    auto emit = [&](int token, float prob, uint32_t flags, int support, float p_draft) {
        emit_row(P, c, row, token, prob, flags, support, p_draft);
        if (finish_request) row_ticket(P, c.b);
    };
    auto emit_late = [&]() {
                                            // (a wait for a copy ran out, in this call or an earlier one on this workspace)
        if (P.op == OP_TOPK) { for (int j = 0; j < P.ktop; ++j) { P.out_vals[(size_t)row * P.ktop + j] = -CUDART_INF_F; P.out_idx[(size_t)row * P.ktop + j] = -1; } }
        else emit(-1, 0.0f, F_TIMEOUT, 0, 0.0f);
    };
    // A copy that never comes, or the workspace's sticky error: every CTA of the cluster learns of it with the first
    // exchange, and all of them leave behind it (the values computed up to there are not used).  Every thread waits and reads
    // the error word for itself, and any of them may be the only one that is late: each tells all CTAs.
    bool late = (err & ERR_TIMEOUT) != 0u;
    if (!mbar_wait(&sh.full, 0)) {
        atomicOr(P.error, ERR_TIMEOUT);
        late = true;
        (void)mbar_wait(&sh.full, 0);                               // (once more: a copy under way must not land in the shared memory of what runs here next)
    }

    // ---------------------------------------------------------------- logit processing
    // Penalties and biases commute with the mask (a masked logit stays -inf); they are applied to the raw values.
    bool bad = c.bad;
    const bool lists = c.hist_len > 0 || c.bias_len > 0;
    auto raw4 = [&](int i) -> float4 {                              // elements i .. i + 3 of the CTA's part as they were loaded
        if (DT == 0) return *reinterpret_cast<const float4 *>(row_y() + i);
        const uint2 r = *reinterpret_cast<const uint2 *>(raw + i * 2);
        return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xFFFF0000u));
    };
    bool in_y = DT == 0;                                            // the values are in x.y already
    if (lists) {
        if (DT == 1) {
            for (int i = x.wlo + lane * 4; i < x.wlo + x.wn; i += 128) *reinterpret_cast<float4 *>(row_y() + i) = raw4(i);
            in_y = true;
            __syncthreads();
        }
        for (int t = tid; t < c.hist_len; t += ROW_THREADS) {
            const int id = (t == tid) ? h_id : __ldg(hid + t), ct = (t == tid) ? h_ct : __ldg(hct + t);
            if (id < 0 || id >= P.V) { bad = true; continue; }
            const int li = id - x.base;
            if (li >= 0 && li < slice) row_y()[li] = apply_penalties(row_y()[li], ct, c);
        }
        __syncthreads();
        for (int t = tid; t < c.bias_len; t += ROW_THREADS) {
            const int id = (t == tid) ? b_id : __ldg(bid + t);
            if (id < 0 || id >= P.V) { bad = true; continue; }
            const int li = id - x.base;
            if (li >= 0 && li < slice) row_y()[li] = __fadd_rn(row_y()[li], (t == tid) ? b_vl : __ldg(bvl + t));
        }
        bad = __syncthreads_or(bad ? 1 : 0) != 0;                   // (every CTA reads the whole lists: all take the exit below or none)
    }
    if (bad) {
        if (lead && late) emit_late();
        else if (lead) emit(-1, 0.0f, F_BADPARAM | (c.cls == CLS_DENSE ? F_DENSE : 0u), 0, 0.0f);
        return;
    }
    // Direct exchange of group maxima: the values stay undivided, only the candidates see the temperature.
    int gpw = 1;                                                    // groups per warp
    while (2 * gpw * x.ncta * ROW_WARPS <= ROW_GMAX && 2 * gpw * x.ncta * ROW_WARPS <= 8 * c.k) gpw *= 2;
    const int ngroups = gpw * x.ncta * ROW_WARPS;
    const bool direct = !dense && !greedy && 2 * c.k <= ngroups && c.k <= ROW_DIRECT;
    const bool masked = (c.z & M_GRAMMAR) != 0;
    float lmax = -CUDART_INF_F, lmin = CUDART_INF_F;                 // maximum, and smallest finite value
    auto process = [&](bool divide, bool first) {
        const float tau = c.tau;
#pragma unroll 2
        for (int i = x.wlo + lane * 4; i < x.wlo + x.wn; i += 128) {
            const float4 f = (first && !in_y) ? raw4(i) : *reinterpret_cast<const float4 *>(row_y() + i);
            float v[4] = {f.x, f.y, f.z, f.w};
            if (first && masked) {
                const uint32_t m = mask[i >> 5] >> (i & 31);
#pragma unroll
                for (int u = 0; u < 4; ++u) if (!((m >> u) & 1u)) v[u] = -CUDART_INF_F;
            }
            if (divide) {
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = div_tau(v[u], tau);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __fadd_rn(v[u], 0.0f);       // (-0 becomes +0)
            if (x.base + i + 3 >= P.V) {
#pragma unroll
                for (int u = 0; u < 4; ++u) if (x.base + i + u >= P.V) v[u] = CUDART_NAN_F;
            }
            lmax = fmaxf(lmax, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
            if (!direct) {
#pragma unroll
                for (int u = 0; u < 4; ++u) lmin = (v[u] > -CUDART_INF_F) ? fminf(lmin, v[u]) : lmin;
            }
            *reinterpret_cast<float4 *>(row_y() + i) = make_float4(v[0], v[1], v[2], v[3]);
        }
    };
    const bool divide = c.temp && c.tau != 1.0f;
    process(divide && !direct, true);
    cl_wait();                                                      // every CTA of the cluster is running
    if (late) for (int r = 0; r < (greedy ? 1 : x.ncta); ++r) *cl_map(&sh.late[x.rank], r) = 1u;        // (a greedy row's other CTAs wait for nobody)

    RowSel s;
    s.vmin = P.op == OP_TOPK ? -CUDART_INF_F : -CUDART_MAX_NORMAL_F;
    s.base = 0ull; s.lo = s.hi = 0ull; s.cut = false;
    auto draw = [&]() -> uint2 {                                    // the row's two uniforms (accept test, draw)
        const unsigned long long pos = offset + (unsigned long long)c.l;
        uint32_t r4[4];
        philox4x32_10((uint32_t)pos, (uint32_t)(pos >> 32), (uint32_t)c.b, 0u, (uint32_t)seed, (uint32_t)(seed >> 32), r4);
        return make_uint2(r4[0] >> 8, r4[1] >> 8);
    };

    if (direct) {
        // ------------------------------------------------------------ top-k, small k
        float g = lmax;
        for (int off = 16 / gpw; off > 0; off >>= 1) g = fmaxf(g, __shfl_xor_sync(0xFFFFFFFFu, g, off));
        {
            const uint32_t key = okey(g);
            for (int q = 0; q < gpw; ++q) {
                const uint32_t kq = __shfl_sync(0xFFFFFFFFu, key, q * (32 / gpw));
                if (lane < x.ncta) *cl_map(&sh.gmax[(x.rank * ROW_WARPS + x.warp) * gpw + q], lane) = kq;
            }
        }
        cl_sync();
        if (row_late(x)) { if (lead) emit_late(); return; }
        const uint32_t tk = kth_max<ROW_THREADS>(sh.gmax, sh.red32, ngroups, c.k, tid);
        // Everything that reaches the bound goes to CTA 0.  With a temperature a value a little below the bound may become
        // equal to it when divided, and then the index decides: the bound is what can divide to as much as it does.  (What
        // divides to -inf is masked by that.)
        float t = max(unkey(tk), s.vmin);
        if (divide) t = (fabsf(t) > c.tau * 0x1p-100f && fabsf(t) < c.tau * 0x1p100f) ? t - fabsf(t) * 0x1p-21f : row_bound_before_div(t, c.tau);
        if (__any_sync(0xFFFFFFFFu, lmax >= t)) {
            unsigned long long *land = cl_map(row_land(), 0);
            unsigned int mine = 0u;
            if (lmax >= t) {
                for (int i = x.wlo + lane * 4; i < x.wlo + x.wn; i += 128) {
                    const float4 f = *reinterpret_cast<const float4 *>(row_y() + i);
                    mine += (f.x >= t ? 1u : 0u) + (f.y >= t ? 1u : 0u) + (f.z >= t ? 1u : 0u) + (f.w >= t ? 1u : 0u);
                }
                unsigned int pos = atomicAdd(cl_map(&sh.land_n, 0), mine);
                for (int i = x.wlo + lane * 4; i < x.wlo + x.wn && mine; i += 128) {
                    const float4 f = *reinterpret_cast<const float4 *>(row_y() + i);
                    const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (v[u] >= t) { if (pos < (unsigned int)ROW_LAND) land[pos] = row_elem(v[u], x.base + i + u); ++pos; --mine; }
                }
            }
            __syncwarp();
        }
        cl_sync();
        RowBcast bc;
        bc.again = (x.rank == 0 && sh.land_n > (unsigned int)ROW_LAND) ? 1 : 0;
        const int n = (int)sh.land_n;                               // (CTA 0's)
        if (x.rank == 0) {
            __syncthreads();
            if (tid < x.ncta) cl_map(&sh.bc, tid)->again = bc.again;
        }
        if (x.rank == 0 && tid == 0 && bc.again) sh.land_n = 0u;
        cl_arrive();
        bool again = bc.again != 0;
        if (x.rank != 0) {
            cl_wait();
            again = sh.bc.again != 0;
        } else if (again) cl_wait();
        if (!again) {
            if (x.rank != 0) return;
            const uint2 cells = draw();
            if (n == 0) { if (tid == 0) emit_row(P, c, row, -1, 0.0f, F_NO_TOKEN, 0, 0.0f); }
            else if (n <= SMALL_MAX) finish_small(P, c, row, row_land(), divide, n, sh.list, tid, cells, draft, q_draft);
            else {
                unsigned long long *buf = reinterpret_cast<unsigned long long *>(row_smem);
                for (int i = tid; i < n; i += ROW_THREADS) {
                    unsigned long long v = row_land()[i];
                    if (divide) v = ((unsigned long long)okey(div_tau(unkey((uint32_t)(v >> 32)), c.tau)) << 32) | (uint32_t)v;
                    buf[i] = v;
                }
                __syncthreads();
                merge_finish<ROW_THREADS, BlockSync>(P, c, row, buf, reinterpret_cast<unsigned int *>(row_rx()), n, min(c.k, n), sh.merge, tid, cells);
            }
            if (finish_request && tid == 0) row_ticket(P, c.b);
            return;
        }
        // more than CTA 0 can hold (crowded ties, few finite values): by histogram over all elements, divided now
        lmax = -CUDART_INF_F;
        for (int i = x.wlo + lane * 4; i < x.wlo + x.wn; i += 128) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float v = divide ? __fadd_rn(div_tau(row_y()[i + u], c.tau), 0.0f) : row_y()[i + u];
                row_y()[i + u] = v;
                lmax = fmaxf(lmax, v);
                lmin = (v > -CUDART_INF_F) ? fminf(lmin, v) : lmin;
            }
        }
    }

    // ---------------------------------------------------------------- row maximum, smallest finite value; greedy rows
    {
        const uint32_t kmx = __reduce_max_sync(0xFFFFFFFFu, okey(lmax)), kmn = __reduce_min_sync(0xFFFFFFFFu, okey(lmin));
        if (lane == 0) { sh.red64[x.warp] = ((unsigned long long)kmx << 32) | kmn; sh.red32[x.warp] = 0xFFFFFFFFu; }
        __syncthreads();
        const unsigned long long kk = sh.red64[lane & (ROW_WARPS - 1)];
        const uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(kk >> 32)), mn = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)kk);
        if (greedy) {
            // lowest index of the CTA's maximum: only the warps that hold it look
            if (kmx == mx && mx > KEY_NEG_INF) {
                const float m = unkey(mx);
                uint32_t at = 0xFFFFFFFFu;
                for (int i = x.wlo + lane * 4; i < x.wlo + x.wn; i += 128) {
                    const float4 f = *reinterpret_cast<const float4 *>(row_y() + i);
                    const uint32_t a = f.x == m ? i : f.y == m ? i + 1 : f.z == m ? i + 2 : f.w == m ? i + 3 : 0xFFFFFFFFu;
                    at = min(at, a);
                }
                at = __reduce_min_sync(0xFFFFFFFFu, at);
                if (lane == 0) sh.red32[x.warp] = at;
            }
            __syncthreads();
            if (tid == 0) {
                uint32_t at = 0xFFFFFFFFu;
                for (int w = 0; w < ROW_WARPS; ++w) at = min(at, sh.red32[w]);
                *cl_map(&sh.ex1[x.rank], 0) = make_ulonglong2(0ull, mx > KEY_NEG_INF ? row_comp(mx, x.base + (int)at) : 0ull);
            }
            cl_arrive();
            if (x.rank != 0) return;
            cl_wait();
            if (row_late(x)) { if (lead) emit_late(); return; }
            if (tid < 32) {
                unsigned long long best = (tid < x.ncta) ? sh.ex1[tid].y : 0ull;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, off));
                const int token = best ? (int)(~(uint32_t)best) : -1;
                if (tid == 0) {
                    if (P.op == OP_TOPK) {                          // k = 1: a row of nothing but -inf still has a first element
                        P.out_vals[row] = best ? unkey((uint32_t)(best >> 32)) : -CUDART_INF_F;
                        P.out_idx[row] = best ? token : 0;
                    } else if (!best) emit(-1, 0.0f, F_NO_TOKEN, 0, 0.0f);
                    else {
                        const bool acc = P.op == OP_VERIFY && draft == token;
                        emit(token, 1.0f, acc ? F_ACCEPT : 0u, 1, acc ? 1.0f : 0.0f);
                    }
                }
            }
            return;
        }
        if (tid < x.ncta) {
            const unsigned long long kd = (draft >= x.base && draft < x.base + slice) ? okey(row_y()[draft - x.base]) : 0u;
            *cl_map(&sh.ex1[x.rank], tid) = make_ulonglong2(((unsigned long long)mx << 32) | mn, kd);
        }
    }
    cl_sync();
    if (row_late(x)) { if (lead) emit_late(); return; }
    uint32_t kmax, kmin;
    {
        const ulonglong2 e = sh.ex1[lane < x.ncta ? lane : 0];
        kmax = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(e.x >> 32));
        kmin = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)e.x);
    }
    x.Mf = unkey(kmax);
    if (kmax <= KEY_NEG_INF && P.op != OP_TOPK) {
        if (lead) emit(-1, 0.0f, F_NO_TOKEN | (c.cls == CLS_DENSE ? F_DENSE : 0u), 0, 0.0f);
        return;
    }

    if (!dense) {
        // ------------------------------------------------------------ top-k, larger k
        bool by_lanes = !direct && 4 * c.k <= x.ncta * ROW_THREADS;
        int n = 0;
        for (;;) {
            int bin;
            unsigned int above, inside;
            float scale;
            const bool enough = row_level_count(x, s, by_lanes, lmax, kmin, c.k, scale, bin, above, inside);
            if (by_lanes && !enough) { by_lanes = false; cl_sync(); continue; }          // fewer lanes with a finite value than k
            unsigned long long floorc = 0ull;
            if (!by_lanes && enough && above + inside > (unsigned int)ROW_LAND) {
                // a crowded bin: split what is at or above it until what is kept fits
                s.lo = 0ull; s.hi = ~0ull;
                unsigned long long need = (unsigned long long)c.k, in_part = 0ull;
                for (int i = 0; i < 12; ++i) {
                    row_split(x, s, false, need, in_part);
                    if ((unsigned long long)c.k - need + in_part <= (unsigned long long)ROW_LAND) break;
                }
                floorc = s.lo;
            }
            row_gather_count(x, s, scale, bin, floorc);
            cl_sync();
            n = (int)sh.land_n;                                     // (CTA 0's)
            if (!by_lanes) break;
            const bool over = n > ROW_LAND;
            if (x.rank == 0) {
                __syncthreads();
                if (tid < x.ncta) cl_map(&sh.bc, tid)->again = over ? 1 : 0;
                if (tid == 0 && over) sh.land_n = 0u;
            }
            cl_arrive();
            if (x.rank == 0 && !over) break;
            cl_wait();
            if (!sh.bc.again) break;
            by_lanes = false;
        }
        if (x.rank != 0) return;
        const uint2 cells = draw();
        n = min(n, ROW_LAND);
        unsigned long long *buf = reinterpret_cast<unsigned long long *>(row_smem);
        for (int i = tid; i < n; i += ROW_THREADS) buf[i] = row_land()[i];
        __syncthreads();
        merge_finish<ROW_THREADS, BlockSync>(P, c, row, buf, reinterpret_cast<unsigned int *>(row_rx()), n, min(c.k, n), sh.merge, tid, cells);
        if (finish_request && tid == 0) row_ticket(P, c.b);
        return;
    }

    // ---------------------------------------------------------------- top-k off, or a top-k beyond the gather
    const uint2 cells = draw();
    const uint32_t cls_flag = c.cls == CLS_DENSE ? F_DENSE : F_FALLBACK;
    // A finite logit over a small temperature can be +inf, whose weight relative to itself would be NaN: the largest finite value
    // stands for it (weight 1 for all such elements, 0 for the others: the limit), so that weights stay within [0, 1] and bins
    // and masses within their range.
    if (kmax > KEY_MAX_NORMAL) {
        for (int i = x.wlo + lane; i < x.wlo + x.wn; i += 32) if (row_y()[i] > CUDART_MAX_NORMAL_F) row_y()[i] = CUDART_MAX_NORMAL_F;
        __syncwarp();
        kmax = KEY_MAX_NORMAL; kmin = min(kmin, KEY_MAX_NORMAL);
        x.Mf = CUDART_MAX_NORMAL_F;
    }
    if (c.cls == CLS_EXACT) {
        // the k-th largest element by count: the row is split until that element is alone
        s.lo = 0ull; s.hi = ~0ull;
        unsigned long long need = (unsigned long long)c.k, in_part = 0ull;
        float scale;
        int bin;
        unsigned int above, inside;
        if (row_level_count(x, s, false, 0.0f, kmin, c.k, scale, bin, above, inside)) {
            for (int i = 0; i < 12 && s.lo != s.hi; ++i) row_split(x, s, false, need, in_part);
            s.base = s.lo;
            s.cut = true;
        }
        cl_sync();                                                  // (every CTA has read the received bins)
    }
    const bool top_p = (c.z & M_TOP_P) != 0;
    // what the support cannot go below, top-p aside
    unsigned long long floorc = s.cut ? s.base : (unsigned long long)(KEY_NEG_INF + 1u) << 32;
    if (c.z & M_MIN_P) floorc = max(floorc, (unsigned long long)minp_key(x.Mf, c.theta) << 32);
    unsigned long long Z = 0ull, goal = 0ull;
    if (top_p) {
        // Bins by the weight's bits: 2^m per octave, so that the row's finite range (41 octaves carry mass at all) takes 256.
        // (the smallest weight's octave is taken a hair lower: the approximate exponential is not promised to be monotone, and a
        // larger value's weight must not fall below the last bin)
        const uint32_t w_min = __float_as_uint(row_w(unkey(kmin), x.Mf));
        const int octaves = 128 - min(127, max(86, (int)((max(w_min, 16u) - 16u) >> 23)));
        const int m = octaves <= 4 ? 6 : octaves <= 8 ? 5 : octaves <= 16 ? 4 : octaves <= 32 ? 3 : 2, shift_a = 23 - m, shift_b = 15 - m;
        const float Mf = x.Mf;
        row_zero_bins(x);
        row_each(x, [&](float y, int idx) {
            const uint32_t bits = __float_as_uint(row_w(y, Mf));
            if (row_in(s, y, idx) && bits >= ROW_WMIN) row_add_weight(bits, (int)((0x3FFFFFFFu - bits) >> shift_a), lane);
        });
        __syncthreads();
        row_fold<true>(x, false, [=](int b) { return b >> m; });
        __syncthreads();
        unsigned long long t = row_sum_bins(x, ROW_BINS);
        if (tid < x.ncta) *cl_map(&sh.sum[0][x.rank], tid) = t;
        cl_sync();
        Z = dense_warp_sum(lane < x.ncta ? sh.sum[0][lane] : 0ull);
        goal = max(1ull, min((unsigned long long)ceil((double)c.p * (double)Z), Z));
        int bin_a, bin_b;
        double before, in_bin;
        row_cross(x, true, (double)goal, bin_a, before, in_bin);
        t = row_sum_bins(x, bin_a);                                 // exact mass above the bin, the CTA's own
        if (tid < x.ncta) *cl_map(&sh.sum[1][x.rank], tid) = t;
        row_zero_bins(x);
        row_each(x, [&](float y, int idx) {
            const uint32_t bits = __float_as_uint(row_w(y, Mf)), d = 0x3FFFFFFFu - bits;
            if ((int)(d >> shift_a) == bin_a && row_in(s, y, idx) && bits >= ROW_WMIN) row_add_weight(bits, (int)((d >> shift_b) & 255u), lane);
        });
        __syncthreads();
        row_fold<true>(x, true, [=](int) { return bin_a >> m; });
        cl_sync();
        const unsigned long long above_a = dense_warp_sum(lane < x.ncta ? sh.sum[1][lane] : 0ull);
        row_cross(x, false, (double)(goal > above_a ? goal - above_a : 1ull), bin_b, before, in_bin);
        const unsigned long long own_b = row_sum_bins(x, bin_b);
        row_gather_bin(x, s, shift_b, (bin_a << 8) | bin_b, t + own_b);
    } else row_mass_above(x, s.vmin, floorc);
    cl_sync();
    bool exact = !top_p;                                            // the gathered part is the right one by construction
    bool masses = !top_p;                                           // sh.above: the whole support, nothing gathered
    unsigned long long cutc = floorc;
    for (int guard = 0; guard < 40; ++guard) {
        RowBcast bc;
        bc.cutc = cutc; bc.W = 0ull; bc.rest = 0ull; bc.need = 0ull; bc.lo = 0ull; bc.hi = 0ull;
        bc.owner = 0u; bc.support = 0u; bc.flags = 0u; bc.again = RB_DONE; bc.p_draft = 0.0f; bc.tie_cta = -1; bc.tie_in = 0u; bc.pad = 0u;
        if (x.rank == 0) {
            const int nm = masses ? 0 : (int)sh.land_n;
            const uint32_t kmn = sh.land_min, kmx = sh.land_max;
            const ulonglong2 ab = (lane < x.ncta) ? sh.above[lane] : make_ulonglong2(0ull, 0ull);      // (lane r: CTA r)
            unsigned long long mass = ab.x;                         // CTA r's part of the support
            const unsigned int members = (unsigned int)(ab.y >> 32);
            bc.W = dense_warp_sum(ab.x);
            unsigned int n = __reduce_add_sync(0xFFFFFFFFu, (unsigned int)ab.y);
            if (tid < x.ncta) sh.cta_mass[tid] = ab.x;
            const uint32_t kd = (draft >= 0) ? min((uint32_t)sh.ex1[draft / slice].y, KEY_MAX_NORMAL) : 0u;
            bool draft_tie_in = false;
            __syncthreads();                                        // (land_n is reset by the broadcast)
            if (!masses) {
                // what is missing inside the part, exactly
                bc.need = goal > bc.W ? goal - bc.W : 0ull;
                bool lost = bc.need == 0ull || nm == 0;             // the float bins named a neighbour of the right bin
                if (!lost && kmn == kmx && !(kd == kmn && nm > ROW_MEMBERS)) {
                    // the ties of one value (low-precision logits: nearly always): as many as are missing, by index
                    const unsigned long long wv = max(1ull, row_q(row_w(unkey(kmn), x.Mf)));
                    unsigned long long m = (unsigned long long)((double)bc.need / (double)wv);
                    while (m * wv < bc.need) ++m;
                    while (m > 1ull && (m - 1ull) * wv >= bc.need) --m;
                    // (the sums of single weights and of bins round differently below 2^-44)
                    lost = m > (unsigned long long)nm && !exact && (m - (unsigned long long)nm) * wv > 65536ull;
                    m = min(m, (unsigned long long)nm);
                    if (lost) {
                    } else if ((uint32_t)(floorc >> 32) > kmn) { bc.again = RB_MASS; bc.cutc = floorc; }       // min-p decides
                    else {
                        const unsigned int pre = row_lane_scan<unsigned int>(members, lane) - members;
                        const unsigned int in = (unsigned int)min((unsigned long long)members, m > pre ? m - pre : 0ull);
                        const unsigned int at = __ballot_sync(0xFFFFFFFFu, members > 0u && pre < m && m <= (unsigned long long)pre + members);
                        mass += in * wv;
                        bc.W += m * wv;
                        n += (unsigned int)m;
                        bc.tie_cta = __ffs(at) - 1;
                        bc.tie_in = __shfl_sync(0xFFFFFFFFu, in, bc.tie_cta);
                        bc.cutc = (unsigned long long)kmn << 32;
                        if (kd == kmn) draft_tie_in = __syncthreads_count(tid < nm && row_land()[tid] > row_comp(kd, draft)) < (int)m;
                    }
                } else if (!lost && nm > ROW_MEMBERS) {
                    bc.again = RB_SPLIT; bc.lo = (unsigned long long)kmn << 32; bc.hi = ((unsigned long long)kmx << 32) | 0xFFFFFFFFull;
                } else if (!lost) {
                    // a short list: the mass ranked above every member, by counting (at most 64) or by sorting
                    unsigned long long mc = 0ull, mq = 0ull, pre = 0ull, tot;
                    if (tid == 0) sh.warp2[0] = 0ull;
                    if (nm <= 64) {
                        if (tid < 64) {
                            const unsigned long long c0 = (tid < nm) ? row_land()[tid] : 0ull;
                            sh.list[tid] = c0;
                            sh.list[64 + tid] = c0 ? row_q(row_w(unkey((uint32_t)(c0 >> 32)), x.Mf)) : 0ull;
                        }
                        __syncthreads();
                        const int j = tid >> 3;                     // eight threads per member
                        const unsigned long long c0 = sh.list[j], q0 = sh.list[64 + j];
                        for (int u = tid & 7; u < nm; u += 8) pre += (sh.list[u] > c0) ? sh.list[64 + u] : 0ull;
#pragma unroll
                        for (int off = 1; off < 8; off <<= 1) pre += __shfl_xor_sync(0xFFFFFFFFu, pre, off);
                        tot = dense_warp_sum(sh.list[64 + lane] + sh.list[96 + lane]);
                        if ((tid & 7) == 0) { mc = c0; mq = q0; }
                    } else {
                        row_rank(x, nm, mc, mq);
                        pre = dense_block_scan<unsigned long long>(mq, sh.red64, tid, tot);
                    }
                    // (the sums of single weights and of bins round differently below 2^-44)
                    if (bc.need > tot && (exact || bc.need - tot <= 65536ull)) bc.need = max(tot, 1ull);
                    lost = bc.need > tot && tot > 0ull;
                    // the element at which the running mass first reaches what is missing
                    if (mq > 0ull && pre < bc.need && bc.need <= pre + mq) { sh.warp2[0] = mc; sh.warp2[1] = pre + mq; }
                    __syncthreads();
                    const unsigned long long cut_p = sh.warp2[0];
                    bc.cutc = max(floorc, cut_p);
                    if (!lost) {
                        if (floorc > cut_p) bc.again = RB_MASS;     // min-p decides
                        else {
                            const bool in = mc != 0ull && mc >= cut_p;
                            if (in && mq) smem_add_u64(&sh.cta_mass[(int)(~(uint32_t)mc) / slice], mq);
                            n += (unsigned int)__syncthreads_count(in ? 1 : 0);
                            bc.W += cut_p ? sh.warp2[1] : 0ull;
                            mass = (lane < x.ncta) ? sh.cta_mass[lane] : 0ull;
                        }
                    }
                }
                if (lost) { bc.again = RB_SPLIT; bc.lo = 0ull; bc.hi = ~0ull; bc.need = goal; bc.cutc = cutc; }
            }
            if (bc.again == RB_DONE) {
                bc.support = n;
                if (P.op == OP_VERIFY && c.l < P.K) {
                    unsigned long long qd = 0ull;
                    if (draft >= 0) {
                        const bool in = (bc.tie_cta >= 0 && kd == (uint32_t)(bc.cutc >> 32)) ? draft_tie_in : row_comp(kd, draft) >= bc.cutc;
                        if (in) qd = row_q(row_w(unkey(kd), x.Mf));
                    }
                    const double Pd = (double)qd / (double)bc.W;
                    bc.flags = ((Pd > 0.0) && (cell_to_u(cells.x) * (double)q_draft <= Pd)) ? RB_ACCEPT : RB_REJECT;
                    bc.p_draft = (float)Pd;
                }
                bc.rest = draw_target(bc.W, cells.y);
                const unsigned long long incl = row_lane_scan<unsigned long long>(mass, lane);
                const unsigned int hit = __ballot_sync(0xFFFFFFFFu, incl > bc.rest);
                const int owner = hit ? __ffs(hit) - 1 : 0;
                bc.rest -= __shfl_sync(0xFFFFFFFFu, incl - mass, owner);
                bc.owner = (unsigned int)owner;
            }
        }
        row_broadcast(x, bc);
        const int again = sh.bc.again;
        if (again == RB_DONE) break;
        if (again == RB_SPLIT) {
            s.lo = sh.bc.lo; s.hi = sh.bc.hi;
            unsigned long long need = sh.bc.need, in_part;
            row_split(x, s, true, need, in_part);
            row_gather_part(x, s);
            exact = true;
        } else {
            cutc = sh.bc.cutc;
            row_mass_above(x, s.vmin, cutc);
            masses = true;
        }
        cl_sync();
    }
    RowBcast bc = sh.bc;
    if (bc.flags & RB_ACCEPT) {                                     // the request moves on with the draft token
        if (lead) emit(P.draft_tokens[(size_t)c.b * P.K + c.l], 0.0f, cls_flag | F_ACCEPT, (int)bc.support, bc.p_draft);
        return;
    }
    if (bc.tie_cta >= 0 && ((bc.flags & RB_REJECT) || x.rank == (int)bc.owner))
        bc.cutc = max(floorc, row_tie_cut(x, s, (uint32_t)(bc.cutc >> 32), bc.tie_cta, bc.tie_in));
    if (bc.flags & RB_REJECT) {
        int token = -1;
        if (row_residual(x, P, c, bc.cutc, bc.W, cells.y, token)) {
            if (token >= 0) emit(token, 0.0f, cls_flag, (int)bc.support, bc.p_draft);
            return;
        }
    }
    if (x.rank == (int)bc.owner) {
        const float Mf = x.Mf;
        const unsigned long long cutw = bc.cutc;
        row_find<unsigned long long>(x, bc.rest, sh.red64, [=](float y, int idx) -> unsigned long long {
            const unsigned long long q = row_q(row_w(y, Mf));
            return (y >= -CUDART_MAX_NORMAL_F && row_elem(y, idx) >= cutw) ? q : 0ull;
        }, [&](int idx, unsigned long long q) {
            emit(idx, (bc.flags & RB_REJECT) ? 0.0f : (float)((double)q / (double)bc.W), cls_flag, (int)bc.support, bc.p_draft);
        });
    }
}

}  // namespace sonic
