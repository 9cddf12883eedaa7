// Streaming kernel of calls that carry a grammar bitmask (rows without the mode bit among them).
//
// The same work as the kernel of that name in sonic_stream.cuh (tiles through a bulk-copy ring, one record per tile), built the other way round:
// nothing of a tile stays in registers.  Under a sparse mask (a grammar allows a few per cent of the ids) a lane walks its
// mask word's few set bits instead of its 32 elements, and list entries that the mask forbids are not patched.  The CTA
// takes a top-k row's cutoff from its first tile of the row and keeps it, so that a tile needs no block barrier; the
// producer requests the next tile before it writes the last one's record.  128 fp32 rows of 2^18, 2 % allowed, 512 entries
// of history each: 58.9 -> 53.2 us a call.  Without a mask this form is the slower one (what it reads twice costs more than
// registers: 256 bf16 rows of 2^18 63 against 61 us), and one kernel with both forms spills, which with 225 KB of shared
// memory and hardly any L1 left beside it costs a fifth: hence two kernels, chosen by whether the call has a bitmask.
#pragma once
#include "sonic_stream.cuh"

namespace sonic {
namespace masked_stream {

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
    int wgroups;                               // top-k rows: groups by which a warp bounds its part alone (0: none serves the row's k)
    int bad;                                   // a list id outside [0, V)
    int off[MAX_TILES + 1];                    // the history entries of tile t: list[off[t], off[t + 1])
    uint32_t list[FILTER_HIST];                // id | count << 18
    Hit bias[FILTER_BIAS];
};

// A kept cutoff is taken for stale where more lanes of a warp than this hold a candidate.  The fullest steps it is kept for bring
// one to 22 of 32 lanes (8 groups per warp tile, the smallest of 64 maxima as the cutoff: 38 of 1024 elements), the usual ones to 4.
constexpr int CROWDED = 28;

template <int DT>
struct StreamShared {
    static constexpr int NSTAGE = VecTraits<DT>::NSTAGE;
    unsigned long long full[NSTAGE];           // producer -> consumers: stage described and copy issued (one arrival + the copy's bytes)
    unsigned long long empty[NSTAGE];          // consumers -> producer: stage free (one arrival per consumer warp)
    StageMeta meta[NSTAGE];
    // per-stage results of the consumer warps, which the producer turns into the tile's record once all of them are done
    alignas(16) float tw[NSTAGE][STREAM_WARPS];
    unsigned int ncand[NSTAGE], badid[NSTAGE];
    unsigned long long best[NSTAGE][STREAM_WARPS];       // greedy rows: argmax; top-k rows: cutoff key << 32; dense rows: largest key << 32
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
            if (lane == 0) { q.cfg = c; q.patch = patch; q.bad = bad ? 1 : 0; q.wgroups = (c.cls == CLS_TOPK) ? pick_warp_groups(P.groups, c.k) : 0; }
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
        // lane 0: the tile's bulk copy, with its bytes announced on full[s] (the arrival follows once the stage's description is
        // written)
        auto issue_copy = [&](int row, int tile, int s) {
            const int first = tile * CTA_TILE;
            const int elems = min(CTA_TILE, ((P.V - first) + VEC - 1) / VEC * VEC);
            const unsigned int bytes = (unsigned int)elems * ELT;
            const unsigned char *src = reinterpret_cast<const unsigned char *>(P.logits) +
                                       ((size_t)row * (size_t)P.row_stride + (size_t)first) * ELT;
            mbar_expect_tx(&sh.full[s], bytes);
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
        if (item >= 0 && lane == 0) issue_copy(item / tiles, item % tiles, 0);
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
                        for (int i = n - NSTAGE; i < n; ++i) (void)mbar_wait(&sh.full[i % NSTAGE], (i / NSTAGE) & 1);       // copies under way
                        return;
                    }
                    // (the first tiles' copies are under way; nothing is copied for rows of the cluster kernel's class)
                    if (item >= 0 && !skip && lane == 0) issue_copy(row, tile, s);
                    retire(s);
                }
                if (item < 0) {                            // out of work: tell the consumers
                    if (lane == 0) { sh.meta[s].stop = 1; mbar_arrive(&sh.full[s]); }
                    break;
                }
                advance();
                const int hint = current_item();           // the tile that follows
                if (lane == 0) {
                    if (n > 0 && n < NSTAGE && !skip) issue_copy(row, tile, s);
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
                for (; i < n; ++i) (void)mbar_wait(&sh.full[i % NSTAGE], (i / NSTAGE) & 1);
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
        const uint32_t mword = (row == pre_row && tile == pre_tile) ? mword_pre : load_mask_words(row, tile);
        pre_row = meta.next_row; pre_tile = meta.next_tile;
        if (pre_row >= 0) mword_pre = load_mask_words(pre_row, pre_tile);
        if (!meta.skip) {
            const unsigned char *stage = stages + (size_t)s * STAGE_BYTES;
            const RowSlot &slot = sh.slot[meta.slot];
            const bool masked = (slot.cfg.z & M_GRAMMAR) != 0;
            const bool tail = tile_base + CTA_TILE > P.V;
            const int patch = slot.patch;
            // word: which of the 32 consecutive elements from lane * 32 count.  Under a sparse mask (a grammar allows a few per
            // cent of the ids) a lane walks its word's few set bits instead of 32 elements, where no lane of the warp has more than 8.
            // 256 bf16 rows of 131072, k = 64: with 4 as the limit 50.3 us instead of 46.3 when 5 % are allowed, with 16 as the limit
            // 68.2 instead of 52.9 when 30 % are (the warp waits for its longest word).
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
                        dr->nmembers = 0u;
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
            float mv[NV];
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
                        const uint4 raw = *reinterpret_cast<const uint4 *>(stage + (size_t)li * ELT);
                        const __nv_bfloat162 m = __hmax2(__hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x), *reinterpret_cast<const __nv_bfloat162 *>(&raw.y)),
                                                         __hmax2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.z), *reinterpret_cast<const __nv_bfloat162 *>(&raw.w)));
                        const uint32_t u = *reinterpret_cast<const uint32_t *>(&m);
                        mv[j] = fmaxf(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
                    } else {
                        const float4 a = *reinterpret_cast<const float4 *>(ptile + li);
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
                // matter, this tile's included (with a temperature: above what can divide to as much): a dense tile's lanes look
                // at a vector or two instead of all of theirs.
                if (row != g_row) { g_row = row; g_thr = -CUDART_MAX_NORMAL_F; }
                unsigned long long best = 0ull;
                if (__any_sync(0xFFFFFFFFu, lm >= g_thr)) {
                    const bool temp = slot.cfg.temp;
                    const float tau = slot.cfg.tau, z = unkey(__reduce_max_sync(0xFFFFFFFFu, okey(lm)));
                    g_thr = fmaxf(g_thr, temp ? bound_before_div(z, tau) : z);
                    if (lm >= g_thr) visit(g_thr, [&](float z, int li) {
                        const uint32_t key = okey(temp ? div_tau(z, tau) : z);
                        if (key > KEY_NEG_INF) best = max(best, ((unsigned long long)key << 32) | (uint32_t)(~(uint32_t)(tile_base + li)));
                    });
                    __syncwarp();
                    const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(best >> 32));
                    const uint32_t lo = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(best >> 32) == hi ? (uint32_t)best : 0u);
                    best = ((unsigned long long)hi << 32) | lo;
                }
                if (lane == 0) sh.best[s][warp] = best;
            } else {
                const int G = slot.cfg.G;
                const bool tmin = slot.cfg.tile_min;
                // warp cutoff: minimum over g groups of the group maximum.  Tile cutoff: the largest of the eight warp cutoffs
                // (warp mode) or the smallest (tile mode: a minimum over all 8 g groups of the tile).  In tile mode a group
                // without a finite element (masked, or past the row's end) does not take part: it would drag the cutoff
                // to -inf and the tile would emit everything it has.
                auto group_cutoff = [&](int g, bool tile_mode) -> float {
                    switch (g) {                               // (one straight-line butterfly per group count)
                    case 0: return -CUDART_INF_F;
                    case 1: return warp_cutoff<32>(lm, tile_mode);
                    case 2: return warp_cutoff<16>(lm, tile_mode);
                    case 4: return warp_cutoff<8>(lm, tile_mode);
                    case 8: return warp_cutoff<4>(lm, tile_mode);
                    case 16: return warp_cutoff<2>(lm, tile_mode);
                    case 32: return warp_cutoff<1>(lm, tile_mode);
                    default: {                                 // 64: half-lane groups
                        const float a0 = (tile_mode && h0 == -CUDART_INF_F) ? CUDART_INF_F : h0;
                        const float a1 = (tile_mode && h1 == -CUDART_INF_F) ? CUDART_INF_F : h1;
                        return warp_cutoff<1>(fminf(a0, a1), false);
                    }
                    }
                };
                // (Many groups, many candidates: a cutoff per tile keeps them down.  Where the line lies makes no difference: beyond 4, 8 or
                // 16 groups all within 1 us at k = 64 and 1000.)
                float t = cut;
                if (row != cut_row || G > 8) {
                    const float g = group_cutoff(G, tmin);
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
                } else if (__popc(__ballot_sync(0xFFFFFFFFu, lm >= t)) > CROWDED) {
                    // Far more candidates than the cutoff was meant for (values that depend on the position): the warp bounds its
                    // own part, by the warp-mode step for the row's k.  (Not by the row's own step: a warp's share of a tile-mode
                    // cutoff lies so high that the row could no longer be proven, and the cluster kernel would have to finish it.)
                    t = fmaxf(t, group_cutoff(slot.wgroups, false));
                }
                if (lane == 0) sh.best[s][warp] = (unsigned long long)okey(t) << 32;
                // every finite element >= t goes to the tile's candidate slot
                const float t2 = fmaxf(t, -CUDART_MAX_NORMAL_F);           // e >= t2  <=>  e >= t and e is not -inf
                const unsigned int cand = __ballot_sync(0xFFFFFFFFu, lm >= t2);
                if (cand) {
                    unsigned long long *dst = P.cand + (size_t)row * P.cand_stride + (size_t)tile * cap_t;
                    auto put = [&](unsigned int pos, float z, int li) {
                        if ((int)pos < cap_t) dst[pos] = ((unsigned long long)okey(z) << 32) | (uint32_t)(~(uint32_t)(tile_base + li));
                    };
                    if (sparse || __popc(cand) <= 8) {
                        // few lanes hold candidates: those look for themselves (up to 4 lanes instead of 8: bf16 rows under masks that allow
                        // a fifth or more 2 us slower; up to 16: the same)
                        if (lm >= t2) visit(t2, [&](float z, int li) { put(atomicAdd(&sh.ncand[s], 1u), z, li); });
                    } else {
                        // many: every lane marks its own, one reservation for the warp
                        unsigned int cm = 0u;
#pragma unroll
                        for (int j = 0; j < NV; ++j) {
                            if (__any_sync(0xFFFFFFFFu, mv[j] >= t2)) {
#pragma unroll
                                for (int q = 0; q < VEC; ++q) cm |= (value(lane0 + j * 32 * VEC + q) >= t2) ? (1u << (j * VEC + q)) : 0u;
                            }
                        }
                        cm &= ebits;
                        const int cnt = __popc(cm);
                        int incl = cnt;
#pragma unroll
                        for (int off = 1; off < 32; off <<= 1) { const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off); if (lane >= off) incl += o; }
                        unsigned int base = 0u;
                        if (lane == 31) base = atomicAdd(&sh.ncand[s], (unsigned int)incl);
                        base = __shfl_sync(0xFFFFFFFFu, base, 31) + (unsigned int)(incl - cnt);
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

}  // namespace masked_stream
}  // namespace sonic
