// Kernels of the dispatch / combine hot path for sm_100a.
//
//   count_kernel / scan_kernel        TokenCnt and CalCumSum as separate launches (the
//                                     bulk-synchronous pipeline; kernel boundaries = barriers)
//   dispatch_kernel<mode, fp8>        persistent CTA per work slice: layout warps plus a mover
//                                     warp that streams rows with TMA bulk copies.  FUSED: the
//                                     layout steps of different CTAs are ordered by
//                                     release/acquire flags instead of launches (kernel
//                                     decomposition).  LOCAL: every CTA derives its offsets
//                                     from the whole routing table (small T*k, no flags), rank-level
//                                     rows.  Clusters (ubep_cluster.cuh): the CTAs of a cluster
//                                     count the table between them; a cluster of one for small
//                                     tables with one row per (token, expert).
//                                     (Small batches: ubep_few.cu.)
//   combine_kernel<K>                 gather + fp32 weighted sum + one bf16 rounding
//   layout_kernel<K>                  counts only (ubep_get_dispatch_layout)
#include <type_traits>

#include "ubep_cluster.cuh"
#include "ubep_kernels.h"
#include "ubep_launch.cuh"
#include "ubep_layout.cuh"
#include "ubep_quant.cuh"

namespace ubep {

// --------------------------------------------------------------- phased: count / scan

// TokenCnt of one token chunk per CTA: bin bitmaps -> chunk histogram and boundary snapshots.
__global__ void __launch_bounds__(256) count_kernel(const Params p, const SmemPlan pl) {
    extern __shared__ __align__(16) uint8_t sm_c[];
    const int c = blockIdx.x, tid = threadIdx.x;
    const int t0 = (int)chunk_begin(c, p.T, p.nchunks), t1 = (int)chunk_begin(c + 1, p.T, p.nchunks);
    int* ids = reinterpret_cast<int*>(sm_c);
    BinMaps bmaps{reinterpret_cast<unsigned*>(sm_c + (pl.off_mask - pl.off_ids)),
                  reinterpret_cast<unsigned*>(sm_c + (pl.off_bm - pl.off_ids)), pl.map_wb, pl.map_bp,
                  pl.map_groups};
    stage_ids(p, t0, t1, ids, tid, 256);
    __syncthreads();
    build_bin_maps(p, ids, t1 - t0, bmaps, tid / 32, 8, tid % 32);
    __syncthreads();
    publish_chunk_counts(p, c, t0, t1, bmaps, tid, 256);
}

__global__ void __launch_bounds__(256) scan_kernel(const Params p) {
    extern __shared__ int sm_i[];
    scan_rank_publish(p, blockIdx.x, sm_i, threadIdx.x / 32, 8, threadIdx.x % 32, 1);
    scan_rank_sources(p, blockIdx.x, sm_i, threadIdx.x, 256);
}

// What a kernel instance moves: bf16 rows, or FP8 rows in one of the two arrangements of the comment above Fp8Ring.  An instance
// holds the code of one of them: what a CTA runs once arrives cold, and with both in one instance a layer of 1 to 128 tokens
// took 0.3 to 0.5 us more.  Token stealing goes with long rows.
enum RowKind { kBf16Rows = 0, kShortFp8Rows = 1, kLongFp8Rows = 2 };

constexpr int kRowWarps = 4;   // flag-free kernel, rank-level rows: warps 1 .. 4 assign the rows of the CTA's tokens

// Everything the roles of one dispatch CTA share.
struct Cta {
    const Params& p;
    const SmemPlan& pl;
    uint8_t* smem;
    uint64_t *full_bar, *empty_bar, *out_full, *out_empty, *ready_bar, *epoch_bar, *staged_bar;
    int* abort_flag;
    int tid, lane, warp, c, part, ch, t0, t1, ntok, stages;
    int gn, nw;        // layout (count) group: warps 1 .. nw, gn = 32 * nw threads
    bool beside;       // FP8: the quantising warps are not layout warps and run beside the layout
    int *ids_sm, *pos, *pos_raw, *key;
    float* w_sm;
    BinMaps bmaps;
    int *hist, *arr, *order_sm;
    unsigned epoch, in_bytes, out_bytes;   // (epoch: 0 until the role that needs it has learnt it from *epoch_late)
    unsigned* epoch_late;
    size_t in_off, out_off;
    bool early0;  // flag-free kernel: the copies of the CTA's first row are issued by the warp that assigns the rows
    int issued;   // rows whose load the mover has started (thread 0's copy is used when leaving early)
    bool early_arrival;   // the mover warp publishes the arrival counters
    int landed_warps;     // ... once these warps (itself among them) have met: they issue copies or write row metadata
    // Every one of those warps calls this once, whatever happened to it; only the mover (wait = 1) stays.
    __device__ __forceinline__ void rows_landed(int wait) const {
        if (wait) asm volatile("bar.sync 14, %0;" ::"r"(landed_warps * 32) : "memory");
        else asm volatile("bar.arrive 14, %0;" ::"r"(landed_warps * 32) : "memory");
    }
};

// The role functions below keep the names the kernel uses for these.
#define UBEP_CTA_LOCALS(x, all15)                                                                              \
    [[maybe_unused]] const Params& p = (x).p;                                                                \
    [[maybe_unused]] const SmemPlan& pl = (x).pl;                                                            \
    [[maybe_unused]] uint8_t* const smem = (x).smem;                                                         \
    [[maybe_unused]] uint64_t* const full_bar = (x).full_bar;                                                \
    [[maybe_unused]] uint64_t* const empty_bar = (x).empty_bar;                                              \
    [[maybe_unused]] uint64_t* const out_full = (x).out_full;                                                \
    [[maybe_unused]] uint64_t* const out_empty = (x).out_empty;                                              \
    [[maybe_unused]] uint64_t& ready_bar = *(x).ready_bar;                                                   \
    [[maybe_unused]] int& abort_flag = *(x).abort_flag;                                                      \
    [[maybe_unused]] volatile int* const abortp = (x).abort_flag;                                            \
    [[maybe_unused]] const int tid = (x).tid, lane = (x).lane, warp = (x).warp, c = (x).c;                   \
    [[maybe_unused]] const int part = (x).part, ch = (x).ch, t0 = (x).t0, t1 = (x).t1, ntok = (x).ntok;     \
    [[maybe_unused]] const int stages = (x).stages, nq = (x).pl.q_warps;                                       \
    [[maybe_unused]] int* const ids_sm = (x).ids_sm;                                                         \
    [[maybe_unused]] int* const pos = (x).pos;                                                               \
    [[maybe_unused]] int* const pos_raw = (x).pos_raw;                                                       \
    [[maybe_unused]] int* const key = (x).key;                                                               \
    [[maybe_unused]] float* const w_sm = (x).w_sm;                                                           \
    [[maybe_unused]] const BinMaps& bmaps = (x).bmaps;                                                       \
    [[maybe_unused]] int* const hist = (x).hist;                                                             \
    [[maybe_unused]] int* const arr = (x).arr;                                                               \
    [[maybe_unused]] int* const order_sm = (x).order_sm;                                                     \
    [[maybe_unused]] const unsigned epoch = (x).epoch, in_bytes = (x).in_bytes, out_bytes = (x).out_bytes;   \
    [[maybe_unused]] const size_t in_off = (x).in_off, out_off = (x).out_off;                                \
    [[maybe_unused]] int& issued = (x).issued;                                                               \
    /* layout group: warps 1 .. nw; a compile-time constant where it is always all 15 */                    \
    [[maybe_unused]] const int nw = (all15) ? kWarps - 1 : (x).nw;                                           \
    [[maybe_unused]] const int gn = nw * 32;                                                                 \
    [[maybe_unused]] const int out_stages = (x).pl.out_stages;                                               \
    [[maybe_unused]] const int gtid = (x).tid - 32, gw = (x).warp - 1

// Pieces of this CTA's rows have landed: add them to the per-region arrival counters (unit: eighths of a row, so that
// the total does not depend on the column split); thread i of n.
__device__ __forceinline__ void publish_arrivals(const Params& p, const int* arr, unsigned half, int i, int n) {
    fence_proxy_async();   // rows written through the async proxy, counters through the generic one
    for (int r = i; r < p.R; r += n)
        if (arr[r]) red_release_add(p.arrival + half * p.R + r, (unsigned)(arr[r] * (8 / p.parts)));
}

// Short rows (row n in ring stage n % stages; the first `head` of them are on their way): `rows` of them at once, a lane
// per copy.  (A trip costs 0.4 us however few bytes it sends; rows with 32 KB of copies take longer than that by
// themselves.  Dispatch of 1536 tokens, 1024 channels, top-4: 11.4 us, one row at a time 14.3.)  Out of line: the code
// of long rows stays short.  Returns how many loads were issued, negative if a wait gave up.
static __device__ __noinline__ int send_short_rows(int n0, int ntok, int head, int rows, int stages, int k, uint64_t* full_bar,
                                                   const int* pos, uint8_t* smem, int stage_bytes, uint8_t* dst, int rowB,
                                                   unsigned bytes, const uint8_t* src, size_t src_stride, unsigned in_bytes,
                                                   volatile int* abort) {
    const int lane = threadIdx.x & 31, sub = lane / k, j = lane - sub * k;
    for (int n = n0; n < ntok; n += rows) {
        const int row = n + sub;
        const bool mine = sub < rows && row < ntok;
        const int s = mine ? row % stages : 0;
        if (!__all_sync(0xffffffffu, !mine || mbar_wait(&full_bar[s], (row / stages) & 1, abort))) return -1 - head;
        const int where = mine ? pos[row * k + j] : -1;
        if (where >= 0) bulk_store(dst + (size_t)where * rowB, smem + (size_t)s * stage_bytes, bytes);
        bulk_commit();
        if (head < ntok) {
            bulk_wait_read<1>();   // every lane: its copies of the trips before this one have read their stages
            __syncwarp();
            const int more = min(min(ntok, n + stages) - head, 32);   // rows that go where rows before n were
            if (lane < more) {
                const int r = head + lane, rs = r % stages;
                mbar_arrive_expect_tx(&full_bar[rs], in_bytes);
                bulk_load(smem + (size_t)rs * stage_bytes, src + (size_t)r * src_stride, in_bytes, &full_bar[rs]);
            }
            head += max(more, 0);
        }
    }
    return head;
}

// ------------------------------------------------------------------------ mover warp
// Warp 0.  Lane 0 issues the TMA loads; for bf16 rows lane j issues the TMA store of slot j,
// so the k copies of a row are issued side by side; for FP8 rows the warp only loads.
template <int kMode, int kRows, bool kSteal>
__device__ __forceinline__ void mover_warp(Cta& x) {
    constexpr bool kFp8 = kRows != kBf16Rows;
    if (kMode == kModeCluster) cluster_arrive();   // (this warp counts nothing)
    if (kMode != kModeLocal) {
        // The epoch: one acquire load and one ticket, two round trips to L2.  This warp has nothing
        // urgent to do yet, so it fetches it while the layout group already stages the routing table.
        unsigned ep = 0;
        if (x.lane == 0) {
            // (before anybody can claim from this chunk: pos_flag is released behind a wait for epoch_bar)
            if (kSteal) x.p.cursor[x.ch] = 0;
            ep = read_epoch_and_check_in(x.p);
            *x.epoch_late = ep;
            mbar_arrive(x.epoch_bar);
        }
        x.epoch = __shfl_sync(0xffffffffu, ep, 0);
    }
    UBEP_CTA_LOCALS(x, !kFp8);
    // Lane 0 issues the TMA loads; for bf16 rows lane j issues the TMA store of slot j,
    // so the k copies of a row are issued side by side.  Tokens come from a feeder: the
    // CTA's own chunk first and, when stealing is on, blocks of other chunks afterwards.
    bool ok = true;
    int v = ch, v_t0 = t0, v_ntok = ntok;   // chunk the feeder currently draws from
    int blk_lo = 0, blk_hi = 0;             // tokens of that chunk this CTA may take now
    unsigned pend = 0;                      // lane 0: answer of a claim made ahead of time
    bool pend_valid = false, feeder_done = false;
    int scanned = 0;                        // victims looked at so far
    blk_hi = kSteal ? ntok - steal_tail(ntok) : ntok;   // the chunk (without stealing), or what is handed out to nobody else: no claims
    // (With a claim per two tokens from the first one on, a round trip to L2 each, the ring was not full when the movers were
    // released: the first copy of 8192 tokens of 4096 channels left 4 us later.)
    if (kSteal && ntok > 0) {
        if (lane == 0) pend = atomicAdd(p.cursor + ch, (unsigned)kStealBlock);   // the first block of the tail, ahead of time
        pend_valid = true;
    }
    const int q_tok = p.T / p.nchunks, q_more = p.T - q_tok * p.nchunks;   // (chunks have q_tok tokens, q_more of them one more)
    const int tails = kSteal ? q_more * steal_tail(q_tok + 1) + (p.nchunks - q_more) * steal_tail(q_tok) : 0;
    auto pick_victim = [&]() -> int {
        while (scanned < p.nchunks - 1) {
            unsigned done = 0;
            if (lane == 0) done = __ldcg(p.claimed + (epoch & 1));
            if ((int)__shfl_sync(0xffffffffu, done, 0) >= tails) return -1;   // every tail is handed out
            const int idx = scanned + lane;
            int cand = ch + 1 + idx;
            if (cand >= p.nchunks) cand -= p.nchunks;
            int rem = 0;
            if (idx < p.nchunks - 1 && ld_acquire(p.pos_flag + cand) == epoch) {
                const int nt = (int)chunk_begin(cand + 1, p.T, p.nchunks) - (int)chunk_begin(cand, p.T, p.nchunks);
                rem = steal_tail(nt) - (int)__ldcg(p.cursor + cand);
            }
            int best = rem > 0 ? (rem << 9) | cand : 0;   // most remaining tokens first (cand < 512)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (best > 0) return best & 511;
            scanned += 32;
        }
        return -1;
    };
    // Next token of the feeder: its index inside chunk v (warp-uniform).  Returns 1 = token,
    // 0 = nothing left anywhere, 2 = only other chunks have work and the caller does not
    // want to take it yet (it still has rows of its own queued).
    bool v_empty = false;   // chunk v has handed out all its tokens
    auto next_token = [&](int& tl, bool allow_steal) -> int {
        while (blk_lo >= blk_hi) {
            if (feeder_done || !kSteal) { feeder_done = true; return 0; }
            if (v_empty) {
                if (!allow_steal) return 2;
                v = pick_victim();
                if (v < 0) { feeder_done = true; return 0; }
                v_t0 = (int)chunk_begin(v, p.T, p.nchunks);
                v_ntok = (int)chunk_begin(v + 1, p.T, p.nchunks) - v_t0;
                v_empty = false;
                pend_valid = false;
            }
            if (v != ch && !allow_steal) return 2;
            if (!pend_valid && lane == 0) pend = atomicAdd(p.cursor + v, (unsigned)kStealBlock);
            const int old = (int)__shfl_sync(0xffffffffu, pend, 0);
            pend_valid = false;
            const int v_tail = steal_tail(v_ntok);
            if (old < v_tail) {
                blk_lo = v_ntok - v_tail + old;
                blk_hi = min(blk_lo + kStealBlock, v_ntok);
                if (lane == 0) {
                    atomicAdd(p.claimed + (epoch & 1), (unsigned)(blk_hi - blk_lo));
                    pend = atomicAdd(p.cursor + v, (unsigned)kStealBlock);   // answer needed a block later
                }
                pend_valid = true;
            } else {
                v_empty = true;
            }
        }
        tl = blk_lo++;
        return 1;
    };
    int* item_src = reinterpret_cast<int*>(smem + pl.off_item);           // [stages] (chunk << 16 | index), -1 = end
    int* item_pos = item_src + kStealStages;                              // [stages, k] destinations of stolen tokens
    int head = 0, tail = 0;   // rows whose load was issued / whose copies were issued
    unsigned ticket = 0u, epoch_mine = 0u;   // (flag-free kernel, FP8 rows)
    // load of the feeder's next token into ring stage head % stages
    auto issue_item = [&](int tl) {
        const int s = head % stages;
        // What travels with the row is written before the load is started: the consumers read it
        // as soon as the row has landed.
        if (kSteal && v != ch) {   // a stolen token: its destinations come from the owner's published list
            for (int j = lane; j < p.k; j += 32)
                item_pos[s * p.k + j] = __ldcg(p.copy_pos + (size_t)(v_t0 + tl) * p.k + j);
            __syncwarp();
        }
        if (lane == 0) {
            if (kSteal) item_src[s] = (v << 16) | tl;
            mbar_arrive_expect_tx(&full_bar[s], in_bytes);
            bulk_load(smem + (size_t)s * pl.stage_bytes,
                      reinterpret_cast<const uint8_t*>(p.x) + (size_t)(v_t0 + tl) * p.H * 2 + in_off, in_bytes,
                      &full_bar[s]);
        }
        if (kSteal) __syncwarp();
        ++head;
    };
    // The first rows of the CTA's own chunk, one load per lane, issued side by side: one lane issuing
    // them one after the other was measured at 0.15 - 0.2 us per load, on the way to the first copy.
    auto issue_first = [&](int n) {   // n <= 32 rows from row `head` on; without stealing
        if (lane < n) {
            const int tl = head + lane, s = tl % stages;
            mbar_arrive_expect_tx(&full_bar[s], in_bytes);
            bulk_load(smem + (size_t)s * pl.stage_bytes,
                      reinterpret_cast<const uint8_t*>(p.x) + (size_t)(t0 + tl) * p.H * 2 + in_off, in_bytes, &full_bar[s]);
        }
        head += n;
    };
    // The same with stealing, for tokens that are handed out to nobody else.
    auto issue_own = [&](int n) {
        if (lane < n) {
            const int tl = blk_lo + lane, s = (head + lane) % stages;
            item_src[s] = (ch << 16) | tl;
            mbar_arrive_expect_tx(&full_bar[s], in_bytes);
            bulk_load(smem + (size_t)s * pl.stage_bytes,
                      reinterpret_cast<const uint8_t*>(p.x) + (size_t)(t0 + tl) * p.H * 2 + in_off, in_bytes, &full_bar[s]);
        }
        __syncwarp();
        head += n;
        blk_lo += n;
    };
    // Rows fetched before the layout is done.  With flags the layout takes many microseconds in which a
    // few small loads and stores of every CTA wait on one another; a ring-full of rows per CTA fetched
    // meanwhile fills the memory system's queues in front of them.  Three rows start the copies, the
    // rest follows once the movers are released.  (With stealing the whole ring: so it was settled when every block of
    // rows cost a claim, a round trip each, best paid while the layout ran.  The head of a slice costs none now; FUSED and PHASED,
    // which AUTO takes only where the plan of the layout by clusters does not fit, have not been timed again since.)
    const int early = (kMode == kModeLocal || kMode == kModeCluster || kSteal) ? kMaxStages : 3;
    if (!kFp8) {
        // loads run (stages - 3) rows ahead; up to 3 rows' stores stay in flight (all rows at once where they fit)
        const int ahead = !kSteal && ntok <= stages ? ntok : pl.trip_rows > 1 ? stages : stages - 3;
        int tl = 0;
        // Flag-free kernel: the routing table first, the rows after it.  The table is the one load the
        // whole layout waits for; the rows of 148 CTAs queued in front of it cost about a microsecond.
        const RankMaps rm{bmaps.bm, bmaps.mask_t, (p.R + 31) / 32, ((p.R + 31) / 32) * 32, (p.T + 31) / 32};
        if (kMode == kModeLocal) {
            // Two rows are asked for at once, so that the first copies find their row in shared memory when
            // the movers are released; then this warp lends a hand with the routing table and asks for the
            // rest of the ring.  (More than two rows in front of the table delay it, 148 CTAs' worth of them
            // queue in front of the one load the layout waits for: measured per layer 25.6 us with one or two
            // rows first, 25.9 with four or with none, 26.5 with the whole ring.)
            if (!kSteal) {
                issue_first(max(min(2, min(ahead, ntok)), 0));
                issued = head;
            }
            local_stage_and_rank_maps(p, ids_sm, rm, rm.groups, 0, kWarps, lane);
            group_sync(2, kThreads);
        } else if (kMode == kModeCluster) {
            // Two rows at once, the rest of the ring when the counts have been exchanged: a ring-full of rows per
            // CTA in flight slows the reads of the other CTAs' shared memory down (by 2 us at 1537 tokens).
            if (kSteal) {
                issue_own(min(2, blk_hi));
            } else {
                issue_first(max(min(2, min(ahead, ntok)), 0));
            }
            issued = head;
            cluster_wait();
            cluster_arrive();    // (this warp reads nothing of the others)
            ok = mbar_wait(x.staged_bar, 0, abortp);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (kSteal) {
            issue_own(max(min(min(ahead, early) - head, min(blk_hi - blk_lo, 32)), 0));
            while (head < min(ahead, early) && next_token(tl, false) == 1) issue_item(tl);
        } else {
            issue_first(max(min(min(min(ahead, early), ntok), 32) - head, 0));
            while (head < min(min(ahead, early), ntok)) issue_item(head);
        }
        issued = head;
        ok = mbar_wait(&ready_bar, 0, abortp) && !*abortp;  // no rows without a layout
        ok = __all_sync(0xffffffffu, ok);
        if (kMode != kModeLocal && kMode != kModeCluster && ok) {   // the rest of the ring
            if (kSteal) {
                while (head < ahead && next_token(tl, false) == 1) issue_item(tl);
            } else {
                while (head < min(ahead, ntok)) issue_item(head);
            }
            issued = head;
        }
        if (!kSteal) {
            // the CTA's own rows, in order: row n sits in stage n % stages
            const int n0 = x.early0 ? 1 : 0;   // (the first row's copies may have been issued by the row group)
            if (pl.trip_rows > 1) {
                if (lane == 0) trace(p, c, kTrFirstRow);
                if (ok) {
                    const int sent = send_short_rows(n0, ntok, head, pl.trip_rows, stages, p.k, full_bar, pos, smem, pl.stage_bytes,
                                                     p.recv_x + out_off, p.rowB, out_bytes,
                                                     reinterpret_cast<const uint8_t*>(p.x) + (size_t)t0 * p.H * 2 + in_off,
                                                     (size_t)p.H * 2, in_bytes, x.abort_flag);
                    ok = sent >= 0;
                    issued = head = ok ? sent : -1 - sent;
                }
            } else
            for (int n = n0; ok && n < ntok; ++n) {
                const int s = n % stages;
                ok = mbar_wait(&full_bar[s], (n / stages) & 1, abortp);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (n == n0 && lane == 0) trace(p, c, kTrFirstRow);
                const uint8_t* src = smem + (size_t)s * pl.stage_bytes;
                for (int j = lane; j < p.k; j += 32) {
                    const int where = pos[n * p.k + j];
                    if (where >= 0) bulk_store(p.recv_x + (size_t)where * p.rowB + out_off, src, out_bytes);
                }
                bulk_commit();
                if (head < ntok) {
                    bulk_wait_read<3>();     // every lane: its copies of the row 3 back have read the stage
                    __syncwarp();
                    issue_item(head);        // without stealing a row's index in the chunk is its sequence number
                    issued = head;
                }
            }
        }
        while (kSteal && ok) {
            if (tail == head) {
                // nothing queued: take over rows of another chunk, or finish
                if (feeder_done || next_token(tl, true) != 1) break;
                issue_item(tl);
                issued = head;
            }
            const int s = tail % stages;
            ok = mbar_wait(&full_bar[s], (tail / stages) & 1, abortp);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (tail == 0 && lane == 0) trace(p, c, kTrFirstRow);
            const uint8_t* src = smem + (size_t)s * pl.stage_bytes;
            const int from = kSteal ? item_src[s] : ((ch << 16) | tail);   // without stealing: own rows in order
            const bool own = (from >> 16) == ch;
            for (int j = lane; j < p.k; j += 32) {
                const int where = own ? pos[(from & 0xffff) * p.k + j] : item_pos[s * p.k + j];
                if (where >= 0) {
                    bulk_store(p.recv_x + (size_t)where * p.rowB + out_off, src, out_bytes);
                    if (kSteal) atomicAdd(&arr[where / p.cap], 1);   // rows per rank: counted by whoever copies
                }
            }
            bulk_commit();
            ++tail;
            if (!feeder_done && head - tail < stages - 3) {
                bulk_wait_read<3>();     // every lane: its copies of the row 3 back have read the stage
                __syncwarp();
                // own rows first, then rows of other chunks, all loaded as far ahead as the ring allows
                if (next_token(tl, true) == 1) issue_item(tl);
                issued = head;
            }
        }
    } else {
        unsigned epoch_ctr = 0u;
        if (kMode == kModeLocal) {
            const RankMaps rm{bmaps.bm, bmaps.mask_t, (p.R + 31) / 32, ((p.R + 31) / 32) * 32, (p.T + 31) / 32};
            local_stage_and_rank_maps(p, ids_sm, rm, rm.groups, 0, kWarps, lane);   // the table first, the rows after it
            group_sync(2, kThreads);
            if (lane == 0) epoch_ctr = ld_relaxed(p.epoch_ctr);
        } else if (kMode == kModeCluster) {
            if (kSteal) issue_own(min(min(2, p.prefetch_rows), min(stages, blk_hi)));   // (see above)
            else issue_first(min(min(2, p.prefetch_rows), min(stages, ntok)));
            issued = head;
            cluster_wait();
            cluster_arrive();
            ok = mbar_wait(x.staged_bar, 0, abortp);
            ok = __all_sync(0xffffffffu, ok);
        } else if (x.beside) {
            // the routing table first: it is the one load the layout waits for
            ok = mbar_wait(x.staged_bar, 0, abortp);
            ok = __all_sync(0xffffffffu, ok);
        }
        // loader only; the quantising warps free the stages.  A closing item with no row
        // tells them that nothing follows.  Rows are fetched as
        // far ahead as the rings allow, at most prefetch_rows of them before the layout is done.
        int tl = 0;
        bool ready_seen = kMode == kModeLocal;   // (the flag-free kernel: its quantisers start after the layout)
        auto wait_ready_at = [&](int n) -> bool {   // warp-uniform
            if (ready_seen || n < p.prefetch_rows) return true;
            bool r = true;
            if (lane == 0) r = mbar_wait(&ready_bar, 0, abortp);
            ready_seen = true;
            return __shfl_sync(0xffffffffu, (int)r, 0) != 0;
        };
        if (!kSteal) {
            // the CTA's own rows only, as far ahead as the ring allows
            while (ok && head < ntok) {
                ok = wait_ready_at(head);
                if (!ok) break;
                if (head >= stages) {
                    if (lane == 0) ok = mbar_wait(&empty_bar[head % stages], ((head / stages) - 1) & 1, abortp);
                    ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                    if (!ok) break;
                }
                tl = head;
                issue_item(tl);
                issued = head;
            }
        }
        while (kSteal && ok) {
            // rows of other chunks are taken only once all but two queued rows are consumed
            bool drained = head < 3;
            if (!drained) {
                const int hs = head - 3;
                drained = mbar_test_wait(&empty_bar[hs % stages], (hs / stages) & 1);
                drained = __all_sync(0xffffffffu, drained);
            }
            ok = wait_ready_at(head);
            if (!ok) break;
            const int got = feeder_done ? 0 : next_token(tl, drained);
            if (got == 2) {
                const int hs = head - 3;   // wait for the queue to drain, then ask again
                ok = mbar_wait(&empty_bar[hs % stages], (hs / stages) & 1, abortp);
                ok = __all_sync(0xffffffffu, ok);
                continue;
            }
            const int s = head % stages;
            if (head >= stages) {
                ok = mbar_wait(&empty_bar[s], ((head / stages) - 1) & 1, abortp);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
            }
            if (got == 1) {
                issue_item(tl);
                issued = head;
            } else {
                if (lane == 0) {   // the closing item
                    item_src[s] = -1;
                    mbar_arrive(&full_bar[s]);
                }
                break;
            }
        }
        if (kMode == kModeLocal && lane == 0) {
            // The epoch (see the row group): asked for in front of the rows, and the ticket taken here, whatever became of
            // the loads; its answer is looked at further down.  (By the first warp of the row group, which quantises, the two
            // round trips to L2 held the first row up: 0.2 us of a layer of 1 to 128 tokens.)
            epoch_mine = epoch_from_counter(epoch_ctr);
            *x.epoch_late = epoch_mine;
            ticket = atomicAdd(p.done_ticket, 1u);
        }
    }
    if (kFp8 && kMode == kModeLocal && ok) {
        // metadata of the CTA's own tokens (see the row group): one warp, no barrier but its own
        ok = mbar_wait(&ready_bar, 0, abortp);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            float* w_own = reinterpret_cast<float*>(key);   // the ordering keys are no longer needed
            if (part == 0)
                for (int i = lane; i < ntok * p.k; i += 32) w_own[i] = ld_plain(p.topk_w + (size_t)t0 * p.k + i);
            local_clean_own_duplicates(p, t0, t1, ids_sm, lane, 32);
            __syncwarp();
            if (part == 0) local_meta_dedup(p, t0, t1, ids_sm, pos_raw, reinterpret_cast<int*>(w_sm), w_own, lane, 32);
        }
    }
    if (kFp8 && kMode == kModeLocal && lane == 0) epoch_finish_check_in(p, ticket, epoch_mine);
    if (!ok && lane == 0) {
        report(p.status, kErrTimeout);  // a wait gave up: record it and let everybody leave
        abort_flag = 1;
    }
    if (lane == 0) trace(p, c, kTrIssued);
    bulk_wait_all<0>();
    if (lane == 0) trace(p, c, kTrStored);
    if (x.early_arrival) {
        // The arrival counters, as soon as the rows have landed and their metadata is written, while other warps still
        // write what belongs to no row.  (At the kernel's end the release waited for those stores as well: 1.6 us of
        // a dispatch of 128 tokens.)
        x.rows_landed(1);
        if (!*abortp) publish_arrivals(p, arr, *reinterpret_cast<volatile unsigned*>(x.epoch_late) & 1u, lane, 32);
    }
}

// ------------------------------------------------------------- layout by clusters
// (see ubep_cluster.cuh)  Every CTA counts its slice of the routing table and its own tokens; after a barrier of
// the cluster it reads, per bin, what the others counted and has all totals and the rows before its own tokens.
// Ends with the movers released.  FP8 rows: once the counting is done the warps behind the first five quantise.
constexpr int kClusterCountWarps = 5;
template <bool kFp8, bool kSteal>
__device__ __forceinline__ void cluster_layout(Cta& x) {
    UBEP_CTA_LOCALS(x, !kFp8);
    int* tot = hist;
    int* base = hist + p.B;    // rows before the CTA's tokens in the bin's segment
    int* eo = hist + 2 * p.B;
    int* row_sm = reinterpret_cast<int*>(w_sm);
    unsigned* cnt = reinterpret_cast<unsigned*>(smem + pl.off_cnt);   // per bin: counts of the slice,
    unsigned* own = cnt + p.B + 1;                                    // counts of the own tokens
    const int cs = p.cluster, me = (int)cluster_ctarank(), c0 = c - me;
    const int first = (int)chunk_begin(c0 / p.parts, p.T, p.nchunks);   // first token of the cluster
    // tokens per rank are an output of their own with one row per (token, expert); the first cluster counts them
    const bool ranks = p.dedup || c0 == 0;
    const int nb = p.E + (ranks ? p.R : 0);
    const int per = (p.T + cs - 1) / cs;
    const int lo = min(p.T, me * per), hi = min(p.T, lo + per);
    constexpr int an = kThreads - 32;   // all warps but the mover count
    // (the own tokens from the last thread on: the first ones may have a token more to count)
    const bool twice = stage_own(p, t0, t1, ids_sm, bmaps.bm, bmaps.bp, own, an - 1 - gtid, an);
    count_tokens(count_args(p), lo, hi, first, ranks, cnt, gtid, an);
    if (p.ordered)
        for (int r = gtid; r < p.R; r += an) order_sm[r] = ld_plain(p.order_pos + r);
    if (group_or(1, an, twice)) {
        local_clean_own_duplicates(p, 0, ntok, ids_sm, gtid, an);
        group_sync(1, an);
    }
    if (gtid == 0) trace(p, c, kTrCounted);
    cluster_arrive();          // this CTA's counts are there
    cluster_wait();            // ... and so are the others'
    if (kFp8 && gw >= nw) {    // FP8 rows: the warps behind the count group go on to quantise
        cluster_arrive();
        return;
    }
    if (gtid == 0) trace(p, c, kTrHistSeen);
    constexpr int bid = kFp8 ? 4 : 1;   // barrier of the count group
#pragma unroll 1
    for (int b = gtid; b < nb; b += gn) {
        unsigned below = 0u, all = 0u;
#pragma unroll 2
        for (int q = 0; q < cs; ++q) {
            const unsigned v = ld_cluster(cnt + b, (unsigned)q);
            below += v & 0xffffu;
            all += v >> 16;
            // its own tokens come earlier than this CTA's (the column parts of a chunk count them once)
            if (c0 + q < c - part && ((c0 + q) & (p.parts - 1)) == 0) below += ld_cluster(own + b, (unsigned)q);
        }
        tot[b] = (int)all;
        base[b] = (int)below;
    }
    cluster_arrive();   // the others' counts have been read: they may leave
    group_sync(bid, gn);
    if (gtid == 0) mbar_arrive(x.staged_bar);   // the mover may fetch the rest of the ring's rows now
#pragma unroll 1
    for (int e = gtid; e < p.E; e += gn) {
        int o = 0;
        for (int q = (e / p.L) * p.L; q < e; ++q) o += tot[q];
        eo[e] = o;
        base[e] += o;
    }
    group_sync(bid, gn);
    if (gtid == 0) trace(p, c, kTrScanSeen);
    bool full = false;
#pragma unroll 1
    for (int li = gtid; li < ntok * p.k; li += gn) {
        const int tl = li / p.k, packed = ids_sm[li];
        const bool have = packed >= 0;
        const int r = have ? slot_rank(packed) : 0;
        bool first_of_rank = have;
        int bin = have ? slot_expert(packed) : 0;
        if (p.dedup) {
            for (int i = tl * p.k; i < li; ++i) first_of_rank = first_of_rank && slot_rank(ids_sm[i]) != r;   // (-1 >> 16 is no rank)
            bin = p.E + r;
        }
        const int row = base[bin] + own_below(bmaps, bin, tl);
        const bool fits = row < p.cap, send = first_of_rank && fits;
        full = full || (have && !fits);
        if (send && !kSteal) atomicAdd(&arr[r], 1);   // rows this CTA will copy to rank r (stealing: counted at copy time)
        pos_raw[li] = send ? r * p.cap + row : -1;
        row_sm[li] = have ? row : -1;
        if (p.ordered) key[li] = send ? rotated_key(order_sm, r, c, p.R) : p.R;
    }
    if (full) report(p.status, kErrCapacity);
    group_sync(bid, gn);
    if (gtid == 0) trace(p, c, kTrFinalized);
    if (p.ordered) {   // a destination table is set: the copies of a token in its order (else pos_raw is pos)
        order_destinations(p, pos_raw, key, pos, ntok * p.k, gtid, gn);
        group_sync(bid, gn);
    }
    if (gtid == 0) {
        mbar_arrive(&ready_bar);
        trace(p, c, kTrReady);
    }
    if (kSteal) {
        // this chunk's destinations, for CTAs that run out of work and take over some of its tokens (FP8 rows: not by the warp
        // that issues the copies, whose first one left 2 us later)
        constexpr int s0 = kFp8 ? 1 : 0, sbar = kFp8 ? 3 : 1;
        if (gw < s0) return;
        const int st = gtid - s0 * 32, sn = gn - s0 * 32;
        for (int i = st; i < ntok * p.k; i += sn) p.copy_pos[(size_t)t0 * p.k + i] = pos[i];
        if (st == 0) (void)mbar_wait(x.epoch_bar, 0, abortp);
        group_sync(sbar, sn);
        if (st == 0) st_release(p.pos_flag + ch, *reinterpret_cast<volatile unsigned*>(x.epoch_late));
    }
}

// What nobody inside the kernel waits for: the metadata of the own tokens, the totals (one CTA) and the counts and
// offsets of the source ranks whose tokens begin among the CTA's own.  Tokens of such a rank beyond the CTA's own
// are counted from the table.
constexpr int kEarlyDutyTokens = 256;   // flag-free kernel, rank-level rows: the expert-level outputs do not wait for the movers
template <bool kFp8>
__device__ __forceinline__ void cluster_duty(Cta& x, int dtid, int dn, int bar) {
    UBEP_CTA_LOCALS(x, !kFp8);
    const int* tot = hist;
    const int* base = hist + p.B;
    const int* eo = hist + 2 * p.B;
    const int* row_sm = reinterpret_cast<const int*>(w_sm);
    unsigned* cnt = reinterpret_cast<unsigned*>(smem + pl.off_cnt) + 2 * (p.B + 1);   // (those in front are read by the cluster)
#pragma unroll 1
    for (int li = dtid; part == 0 && li < ntok * p.k; li += dn) {
        const int tl = li / p.k, packed = ids_sm[li], row = row_sm[li], where = pos_raw[li];
        const size_t i = (size_t)t0 * p.k + li;
        const bool have = packed >= 0;
        const int r = have ? slot_rank(packed) : 0;
        p.slot_row[i] = row;
        p.slot_pos[i] = have && row < p.cap ? r * p.cap + row : -1;
        if (p.dedup && have) {
            const int e = slot_expert(packed), at = base[e] + own_below(bmaps, e, tl);
            if (at < p.er_cap) p.expert_rows[(size_t)r * p.er_cap + at] = row;
            else report(p.status, kErrCapacity);
        }
        if (where < 0) continue;
        p.recv_src_idx[where] = t0 + tl;
        if (!p.dedup) {
            p.recv_weight[where] = ld_plain(p.topk_w + i);
        } else if ((p.k & 3) == 0) {   // rows of the two arrays start on 16-byte boundaries: four slots per store
#pragma unroll 1
            for (int j = 0; j < p.k; j += 4) {
                const float4 w = ld_plain(reinterpret_cast<const float4*>(p.topk_w + (size_t)(t0 + tl) * p.k + j));
                const float wv[4] = {w.x, w.y, w.z, w.w};
                int e4[4];
                float w4[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int v = ids_sm[tl * p.k + j + u];
                    const bool here = v >= 0 && slot_rank(v) == r;
                    e4[u] = here ? slot_expert(v) - r * p.L : -1;
                    w4[u] = here ? wv[u] : 0.0f;
                }
                *reinterpret_cast<int4*>(p.recv_topk_idx + (size_t)where * p.k + j) = make_int4(e4[0], e4[1], e4[2], e4[3]);
                *reinterpret_cast<float4*>(p.recv_topk_w + (size_t)where * p.k + j) = make_float4(w4[0], w4[1], w4[2], w4[3]);
            }
        } else {
#pragma unroll 1
            for (int j = 0; j < p.k; ++j) {
                const int v = ids_sm[tl * p.k + j];
                const bool here = v >= 0 && slot_rank(v) == r;
                p.recv_topk_idx[(size_t)where * p.k + j] = here ? slot_expert(v) - r * p.L : -1;
                p.recv_topk_w[(size_t)where * p.k + j] = here ? ld_plain(p.topk_w + (size_t)(t0 + tl) * p.k + j) : 0.0f;
            }
        }
    }
    x.rows_landed(0);
    if (c == 0) write_totals(p, tot, eo, dtid, dn);
    if (ntok != 0) write_own_sources<false>(p, t0, t1, part, p.parts, bmaps, base, cnt, dtid, dn, bar);
}

// ---------------------------------------------------------------------- layout group
// Warps 1..15: TokenCnt, CalCumSum (by exchange or alone), slot -> row assignment; releases
// the movers and then writes what nobody inside the kernel waits for.  Returns 1, 0 if a wait ran
// out, or 2 for a warp that has done its share of the counting and now leaves to quantise.
template <int kMode, int kRows, bool kSteal>
__device__ __forceinline__ int layout_group(Cta& x) {
    constexpr bool kFp8 = kRows != kBf16Rows;
    UBEP_CTA_LOCALS(x, !kFp8);
    bool ok = true;
    const int* ids = ids_sm;  // staged slots of this CTA's tokens
    // Small global reads whose values are needed only after the first barriers: issue the
    // loads now (first trip of each loop), store to shared memory after the ids are staged.
    const int order_r = kMode != kModeCluster && gtid < p.R ? ld_plain(p.order_pos + gtid) : 0;
    const bool stage_w = kMode != kModeCluster && kMode != kModeLocal;
    const float w_first = (stage_w && gtid < ntok * p.k) ? ld_plain(p.topk_w + (size_t)t0 * p.k + gtid) : 0.0f;
    auto stage_small = [&](int n) {   // by n threads
        if (gtid < p.R) order_sm[gtid] = order_r;
        for (int r = gtid + n; r < p.R; r += n) order_sm[r] = ld_plain(p.order_pos + r);
        if (stage_w) {
            if (gtid < ntok * p.k) w_sm[gtid] = w_first;
            for (int i = gtid + n; i < ntok * p.k; i += n) w_sm[i] = ld_plain(p.topk_w + (size_t)t0 * p.k + i);
        }
    };
    if (kMode == kModeLocal) {
        // rank-level rows first, movers released, expert-level outputs afterwards
        const RankMaps rm{bmaps.bm, bmaps.mask_t, (p.R + 31) / 32, ((p.R + 31) / 32) * 32, (p.T + 31) / 32};
        int* row_sm = reinterpret_cast<int*>(w_sm);
        // (the own tokens' gate weights, asked for while the table is on its way; needed for the metadata)
        const float w_row = !kFp8 && part == 0 && gw < kRowWarps && gtid < ntok * p.k ? ld_plain(p.topk_w + (size_t)t0 * p.k + gtid) : 0.0f;
        local_stage_and_rank_maps(p, ids_sm, rm, rm.groups, warp, kWarps, lane);   // with the mover warp
        stage_small(gn);
        group_sync(2, kThreads);
        if (gtid == 0) trace(p, c, kTrCounted);
        // From here the group splits.  Assigning rows to the CTA's own few tokens keeps a handful of
        // threads busy, and nothing expert-level depends on it: warps 1..4 (the row group) assign the
        // rows, release the movers and write the metadata of the own tokens, while the other warps
        // (the duty group) already derive the expert-level outputs from the staged table.  (One after
        // the other, the expert-level outputs ended after the last copy and set the kernel's duration.)
        constexpr int kRowThreads = kRowWarps * 32;
        if (gw < kRowWarps) {
            const int rn = kRowThreads;
            local_rows_dedup(p, t0, t1, ids_sm, rm, c, order_sm, pos_raw, key, row_sm, arr, gtid, rn);
            if (x.early0 && gw == 0) {
                // The copies of the CTA's first row leave from here: lane j has just worked out where slot j of
                // the first token goes (its own write to pos_raw), and the row was asked for before the routing
                // table was (and prefetched into L2 before that), so it sits in the ring's first stage or is
                // about to.  The mover warp, which needs another 0.5 us to notice the release and get going,
                // starts with the second row.  (Measured per layer, 512 tokens: 25.2 us against 25.6; neither
                // this nor the prefetch of the rows changes anything without the other.)
                const int where = lane < p.k ? pos_raw[lane] : -1;
                const bool got = mbar_wait(&full_bar[0], 0, abortp);
                if (got && where >= 0) bulk_store(p.recv_x + (size_t)where * p.rowB + out_off, smem, out_bytes);
                bulk_commit();
                if (!got && lane == 0) {
                    report(p.status, kErrTimeout);
                    *abortp = 1;
                }
            }
            group_sync(1, rn);
            if (gtid == 0) trace(p, c, kTrFinalized);
            if (p.ordered) {   // a destination table is set: the copies of a token in its order (else pos_raw is pos)
                order_destinations(p, pos_raw, key, pos, ntok * p.k, gtid, rn);
                group_sync(1, rn);
            }
            if (gtid == 0) {
                mbar_arrive(&ready_bar);
                trace(p, c, kTrReady);
            }
            // FP8 rows: every copy waits for a quantised row, so this group goes straight on to quantise
            // (its first warp to issue the copies of long rows; the warps of the duty group take no part, a CTA of
            // this kernel has few rows).  The epoch, and the metadata of the own tokens, are left to the loader warp,
            // which is idle once the CTA's few rows are asked for.
            if (kFp8) return 1;
            unsigned ticket = 0u, ep_mine = 0u;
            if (gtid == 0) {
                // The epoch: nothing needs it before the kernel's last lines.  A relaxed load (nothing
                // is ordered against it); its value is in hand before the ticket is taken -- the store
                // to shared memory needs it -- and the ticket's answer is looked at at the end.
                ep_mine = epoch_from_counter(ld_relaxed(p.epoch_ctr));
                *x.epoch_late = ep_mine;
                ticket = atomicAdd(p.done_ticket, 1u);
            }
            if (part == 0) {
                float* w_own = reinterpret_cast<float*>(key);   // the ordering keys are no longer needed
                if (gtid < ntok * p.k) w_own[gtid] = w_row;
                for (int i = gtid + rn; i < ntok * p.k; i += rn) w_own[i] = ld_plain(p.topk_w + (size_t)t0 * p.k + i);
            }
            local_clean_own_duplicates(p, t0, t1, ids_sm, gtid, rn);   // (rank-level rows do not depend on them)
            group_sync(1, rn);
            if (p.trace && gtid == 0) p.trace[(size_t)c * kTraceSlots + 11] = trace_ns(p);
            if (part == 0) local_meta_dedup(p, t0, t1, ids_sm, pos_raw, row_sm, reinterpret_cast<float*>(key), gtid, rn);
            if (gtid == 0) {
                epoch_finish_check_in(p, ticket, ep_mine);
                if (p.trace) p.trace[(size_t)c * kTraceSlots + 12] = trace_ns(p);
            }
            if (x.early0 && gw == 0) bulk_wait_all<0>();   // the first row's copies (issued by this warp)
            x.rows_landed(0);
        } else if (kFp8 && warp - pl.q_warp0 < nq) {
            return 1;   // FP8 rows: the first warps behind the row group quantise as well
        } else {
            // expert-level outputs of rank r: shared by Q CTAs so that no CTA trails the others
            const int dgw0 = kFp8 ? max(kRowWarps, pl.q_warp0 + nq - 1) : kRowWarps;   // first warp of the duty group
            const int dn = gn - dgw0 * 32, dw = nw - dgw0;
            const int Q = p.grid / p.R > 1 ? p.grid / p.R : 1;
            // ... once the movers are released: started earlier, these warps take issue slots and
            // shared-memory bandwidth from the few threads every copy of this CTA is waiting for.  (Small tables: the
            // copies end long before these outputs, which start at once; not with FP8 rows, which have to be quantised.)
            const bool go = (!kFp8 && p.T <= kEarlyDutyTokens) || mbar_wait_idle(&ready_bar, 0, abortp);
            for (int u = c; go && u < p.R * Q; u += p.grid)
                local_rank_duty(p, u / Q, u % Q, Q, ids_sm, rm, hist, gw - dgw0, dw, lane, gtid - dgw0 * 32, dn, 3);
            if (gtid == dgw0 * 32) trace(p, c, kTrScanned);   // deferred outputs written
            if (kFp8) return go ? 3 : 0;   // (these warps do not quantise: the row group's warps do)
        }
    } else if (kMode == kModeCluster) {
        cluster_layout<kFp8, kSteal>(x);
        if (kFp8 && gw >= nw) return 2;   // off to quantise
        constexpr int d0 = kRows == kLongFp8Rows ? 1 : 0;
        if (gw < d0) return 1;            // off to issue the copies
        // the others write what nobody waits for
        cluster_duty<kFp8>(x, gtid - d0 * 32, gn - d0 * 32, kFp8 ? 3 : 1);
        if (gtid == d0 * 32) trace(p, c, kTrScanned);   // deferred outputs written
        return kFp8 ? 3 : 1;
    } else {
        // FP8 rows with a count group: TokenCnt itself -- staging the ids, the bitmaps, publishing the
        // chunk's counts -- is pure computation and is done by all 15 warps; then the warps behind the
        // count group leave to quantise, and the count group alone goes through the steps that mostly
        // wait for other CTAs (flag exchange, CalCumSum duty) and assigns the rows.
        const bool split = kFp8 && x.beside;
        const int an = split ? kThreads - 32 : gn, aw = split ? kWarps - 1 : nw;
        const int bid = split ? 4 : 1;   // barrier of the count group once the others have left
        stage_ids(p, t0, t1, ids_sm, gtid, an);
        stage_small(an);
        group_sync(1, an);
        if (kFp8 && gtid == 0) mbar_arrive(x.staged_bar);   // the loader may fetch rows now
        build_bin_maps(p, ids_sm, ntok, bmaps, gw, aw, lane);
        group_sync(1, an);
        if (kMode == kModeFused) publish_chunk_counts(p, ch, t0, t1, bmaps, gtid, an);
        if (split) {
            group_sync(1, an);          // the counts are stored (the flag is released further down)
            if (gw >= nw) return 2;     // off to quantise
        }
        int deferred = -1;
        // The mover warp fetched the epoch while the table was staged; one thread makes sure it has
        // arrived, the barrier that follows hands it to the others.
        unsigned ep = 0;
        auto learn_epoch = [&]() {
            if (gtid == 0) (void)mbar_wait(x.epoch_bar, 0, abortp);
            group_sync(bid, gn);
            ep = *reinterpret_cast<volatile unsigned*>(x.epoch_late);
        };
        if (kMode == kModeFused) {
            learn_epoch();
            if (gtid == 0) {
                if (ch != p.withhold) {
                    st_release(p.hist_flag + ch, ep);   // release: cumulative over what the barrier above ordered
                }
                trace(p, c, kTrCounted);
            }
            // CalCumSum duty: this CTA serves rank ch (and ch + nchunks, ...)
            bool lost = false;  // a wait of this thread ran out
            for (int r = ch; r < p.R; r += p.nchunks) {
                for (int cc = gtid; cc < p.nchunks; cc += gn)
                    if (!wait_flag(p.hist_flag + cc, ep, abortp)) lost = true;
                if (group_or(bid, gn, lost || *abortp)) { lost = true; break; }  // same answer for all
                if (gtid == 0) trace(p, c, kTrHistSeen);
                scan_rank_publish(p, r, hist, gw, nw, lane, bid);
                if (gtid == 0) {
                    st_release(p.scan_flag + r, ep);
                    trace(p, c, kTrScanned);
                }
                if (r + p.nchunks < p.R) {
                    scan_rank_sources(p, r, hist, gtid, gn);
                    group_sync(bid, gn);
                } else {
                    deferred = r;   // cnt / src_offset: after our own movers are released
                }
            }
            // every slot of this chunk may need any rank's bases
            if (!lost)
                for (int r = gtid; r < p.R; r += gn)
                    if (!wait_flag(p.scan_flag + r, ep, abortp)) lost = true;
            ok = !group_or(bid, gn, lost || *abortp);
            if (gtid == 0) trace(p, c, kTrScanSeen);
            if (!ok && gtid == 0) {
                report(p.status, kErrTimeout);
                abort_flag = 1;
            }
        }
        if (ok) {
            // rows before a token = rows of earlier chunks (+ the expert's offset in its
            // region), published by the prefix-sum step, + earlier tokens of this chunk.
            // The published part is fetched once per bin into shared memory (one round
            // trip to L2), the rest is bit counting.
            const int32_t* cb = p.chunk_base + ch;   // [bin][chunk]
            int* base_sm = hist + p.B;   // second half of the scratch (the first may hold scan totals)
            for (int b = gtid; b < p.B; b += gn)
                base_sm[b] = __ldcg(cb + (size_t)b * p.nchunks) + (b < p.E ? __ldcg(p.expert_offset + b) : 0);
            group_sync(bid, gn);
            finalize_chunk(p, t0, t1, ids, w_sm,
                           [&](int e, int tl) { return base_sm[e] + bits_in_range(bmaps, e, 0, tl); },
                           [&](int r, int tl) { return base_sm[p.E + r] + bits_in_range(bmaps, p.E + r, 0, tl); },
                           true, c, order_sm, pos_raw, key, kSteal ? nullptr : arr, gtid, gn);
            group_sync(bid, gn);
            if (gtid == 0) trace(p, c, kTrFinalized);
            if (p.ordered) {   // a destination table is set: the copies of a token in its order (else pos_raw is pos)
                order_destinations(p, pos_raw, key, pos, ntok * p.k, gtid, gn);
                group_sync(bid, gn);
            }
        }
        if (gtid == 0) {
            mbar_arrive(&ready_bar);
            trace(p, c, kTrReady);
        }
        if (ok && kSteal) {
            // this chunk's destinations, for CTAs that run out of work and take over some of its tokens
            for (int i = gtid; i < ntok * p.k; i += gn) p.copy_pos[(size_t)t0 * p.k + i] = pos[i];
            if (kMode == kModeFused) group_sync(bid, gn);
            else learn_epoch();   // (with kernel boundaries instead of flags nothing has asked for it yet)
            if (gtid == 0) {
                st_release(p.pos_flag + ch, ep);
            }
        }
        if (ok && deferred >= 0) scan_rank_sources(p, deferred, hist, gtid, gn);
    }
    return ok ? 1 : 0;
}

// ------------------------------------------------------------ FP8: quantise and store
// Long rows (40 KB of copies and more).  Two roles around a ring of quantised rows (payload + scales): the quantising
// warps turn one row after the other into FP8 and know nothing about destinations (own rows) -- so they can run
// beside the layout; the store issuer sends every quantised row to its destinations with bulk copies once the
// layout is done, at most three rows at a time.
//
// Short rows.  The quantising warps work in teams (fp8_worker).  A team takes every teams-th row the loader has fetched,
// quantises it into one of its two slots and sends it itself once the layout is done; the next row is quantised
// meanwhile.  A team is one warp, so that a row costs no barrier and as many rows are on their way as there are
// warps; only where a CTA has fewer rows than warps do several of them share one.  (In the arrangement for long rows
// each row costs a CTA 1.1 us, however short.  Dispatch of 1536 tokens, 1024 channels, top-4: 24.0 us that way, 11.6 this
// way; 2048 channels: 21.6 and 13.5; 4096 channels, top-8: 21.8 and 18.9.  So many long rows on their way at once run at
// less bandwidth: 7168 channels, top-8, 1024 / 4096 tokens 18.0 / 62 and 20.3 / 67 us.)
//
// Shared-memory bookkeeping behind the input ring's items: out_src[os] = where the row of
// output stage os comes from (chunk << 16 | index, -1 = nothing follows), out_pos[os] = the
// destinations of a row taken over from another chunk.
struct Fp8Ring {
    uint8_t* out_ring;
    const int* item_src;   // [kStealStages]
    const int* item_pos;   // [kStealStages, k]
    int* out_src;          // [out_stages]
    int* out_pos;          // [out_stages, k]
    int g0;                // first scale group of this CTA's piece
    unsigned scale_bytes;  // its scales travel with the payload
    bool scale_bulk;       // ... by a bulk copy when their size allows it
};
__device__ __forceinline__ Fp8Ring fp8_ring(const Cta& x) {
    const Params& p = x.p;
    int* item = reinterpret_cast<int*>(x.smem + x.pl.off_item);
    Fp8Ring q;
    q.out_ring = x.smem + x.pl.off_out;
    q.item_src = item;
    q.item_pos = item + kStealStages;
    q.out_src = item + kStealStages * (p.k + 1);
    q.out_pos = q.out_src + x.pl.out_stages;
    q.g0 = x.part * (p.G / p.parts);
    q.scale_bytes = (unsigned)(p.G / p.parts) * 4u;
    q.scale_bulk = (q.scale_bytes & 15u) == 0;
    return q;
}

// The copies of the quantised row in stage `os`; lanes 0 .. k - 1 the payload, k .. 2k - 1 the scales.
template <bool kSteal>
__device__ __forceinline__ void fp8_issue(Cta& x, const Fp8Ring& q, const uint8_t* src, int from, int os) {
    UBEP_CTA_LOCALS(x, false);
    const int* wpos = (from >> 16) == ch ? pos + (from & 0xffff) * p.k : q.out_pos + os * p.k;
    for (int j = lane; j < (q.scale_bulk ? 2 * p.k : p.k); j += 32) {
        const bool payload = j < p.k;
        const int where = wpos[payload ? j : j - p.k];
        if (where < 0) continue;
        if (payload) {   // (two instructions, not one with the operands selected per lane: that was 10 - 15 % slower)
            bulk_store(p.recv_x + (size_t)where * p.rowB + out_off, src, out_bytes);
            if (kSteal) atomicAdd(&arr[where / p.cap], 1);
        } else {
            bulk_store(p.recv_scale + (size_t)where * p.G + q.g0, src + out_bytes, q.scale_bytes);
        }
    }
    if (!q.scale_bulk) {   // a piece of scales that no bulk copy can carry: plain stores
        const int Gp = p.G / p.parts;   // scale groups of this CTA's piece
        const float* sc = reinterpret_cast<const float*>(src + out_bytes);
        for (int i = lane; i < p.k * Gp; i += 32) {
            const int jj = i / Gp, g = i - jj * Gp;
            const int where = wpos[jj];
            if (where >= 0) p.recv_scale[(size_t)where * p.G + q.g0 + g] = sc[g];
        }
    }
    bulk_commit();
}

// Long rows: quantising warp qw of nq.
template <bool kSteal>
__device__ __forceinline__ void fp8_quantiser(Cta& x, int qw) {
    UBEP_CTA_LOCALS(x, false);
    const Fp8Ring q = fp8_ring(x);
    const int nvec = (int)in_bytes / 16;          // 8-channel vectors in this CTA's piece
    unsigned long long w_in = 0, w_out = 0, t_cmp = 0, tq = 0;
    for (int n = 0; kSteal || n < ntok; ++n) {
        const int s = n % stages, os = n % out_stages;
        if (p.trace) tq = trace_ns(p);
        if (!mbar_wait_idle(&full_bar[s], (n / stages) & 1, abortp)) break;
        if (p.trace) { unsigned long long t2 = trace_ns(p); w_in += t2 - tq; tq = t2; }
        if (n >= out_stages && !mbar_wait_idle(&out_empty[os], ((n / out_stages) - 1) & 1, abortp)) break;
        if (p.trace) { unsigned long long t2 = trace_ns(p); w_out += t2 - tq; tq = t2; }
        const int from = kSteal ? q.item_src[s] : ((ch << 16) | n);
        if (from < 0) {
            // the loader's closing item: pass it on to the store issuer and leave
            if (qw == 0 && lane == 0) q.out_src[os] = -1;
            __syncwarp();
            if (lane == 0) mbar_arrive(&out_full[os]);
            break;
        }
        if (kSteal && qw == 0) {
            if ((from >> 16) != ch)   // a row of another chunk: its destinations travel with it
                for (int j = lane; j < p.k; j += 32) q.out_pos[os * p.k + j] = q.item_pos[s * p.k + j];
            if (lane == 0) q.out_src[os] = from;
        }
        const uint8_t* src = smem + (size_t)s * pl.stage_bytes;
        uint8_t* dst = q.out_ring + (size_t)os * pl.out_stage_bytes;
        float* dst_scale = reinterpret_cast<float*>(dst + out_bytes);
        // two vectors per thread and trip, independent of each other
        for (int vb = qw * 32; vb < nvec; vb += 2 * nq * 32) {
            const int v0 = vb + lane, v1 = v0 + nq * 32;
            const bool ok0 = v0 < nvec, ok1 = v1 < nvec;
            uint4 in0 = make_uint4(0, 0, 0, 0), in1 = make_uint4(0, 0, 0, 0);
            if (ok0) in0 = *reinterpret_cast<const uint4*>(src + (size_t)v0 * 16);
            if (ok1) in1 = *reinterpret_cast<const uint4*>(src + (size_t)v1 * 16);
            uint2 q0, q1;
            float sc0, sc1;
            quantize8(in0, ok0, q0, sc0);
            quantize8(in1, ok1, q1, sc1);
            if (ok0) *reinterpret_cast<uint2*>(dst + (size_t)v0 * 8) = q0;
            if (ok1) *reinterpret_cast<uint2*>(dst + (size_t)v1 * 8) = q1;
            if ((lane & 15) == 0) {
                if (ok0) dst_scale[v0 >> 4] = sc0;
                if (ok1) dst_scale[v1 >> 4] = sc1;
            }
        }
        fence_proxy_async_smem();   // the bulk stores read what we just wrote
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&out_full[os]);
            mbar_arrive(&empty_bar[s]);
        }
        if (p.trace) t_cmp += trace_ns(p) - tq;
    }
    if (p.trace && qw == 0 && lane == 0) {
        p.trace[(size_t)c * kTraceSlots + 11] = w_in;
        p.trace[(size_t)c * kTraceSlots + 12] = w_out;
        p.trace[(size_t)c * kTraceSlots + 13] = t_cmp;
    }
}

// Long rows: the store issuer (one warp, after the layout).
template <bool kSteal>
__device__ __forceinline__ void fp8_store_issuer(Cta& x) {
    UBEP_CTA_LOCALS(x, false);
    const Fp8Ring q = fp8_ring(x);
    bool sok = true;
    unsigned long long w_full = 0, w_read = 0, tq = 0;
    for (int n = 0; kSteal || n < ntok; ++n) {
        const int os = n % out_stages;
        if (p.trace) tq = trace_ns(p);
        sok = mbar_wait(&out_full[os], (n / out_stages) & 1, abortp);
        if (p.trace) w_full += trace_ns(p) - tq;
        sok = __all_sync(0xffffffffu, sok);
        const int from = kSteal ? q.out_src[os] : ((ch << 16) | n);
        if (!sok || from < 0) break;
        if (n == 0 && lane == 0) trace(p, c, kTrFirstRow);
        fp8_issue<kSteal>(x, q, q.out_ring + (size_t)os * pl.out_stage_bytes, from, os);
        if (n + 1 >= kStorePending) {
            if (p.trace) tq = trace_ns(p);
            bulk_wait_read<kStorePending - 1>();   // every lane: the copies of the row kStorePending - 1 back have read it
            if (p.trace) w_read += trace_ns(p) - tq;
            __syncwarp();
            if (lane == 0) mbar_arrive(&out_empty[(n + 1 - kStorePending) % out_stages]);
        }
    }
    if (!sok && lane == 0) {
        report(p.status, kErrTimeout);
        abort_flag = 1;
    }
    bulk_wait_all<0>();
    if (p.trace && lane == 0) {
        p.trace[(size_t)c * kTraceSlots + 14] = w_full;
        p.trace[(size_t)c * kTraceSlots + 15] = w_read;
    }
}

// Short rows (see Fp8Ring): quantising warp qw, in teams that send what they have quantised themselves.
__device__ __forceinline__ void fp8_worker(Cta& x, int qw) {
    UBEP_CTA_LOCALS(x, false);
    const Fp8Ring q = fp8_ring(x);
    const int teams = pl.q_teams, tw = pl.q_team_warps, team = qw / tw, m = qw - team * tw;
    if (team >= teams) return;
    auto team_sync = [&]() {
        if (tw > 1) group_sync(5 + team, tw * 32);
        else __syncwarp();
    };
    const int nvec = (int)in_bytes / 16;   // 8-channel vectors in this CTA's piece
    bool ready = false, good = true;
    int sent = 0;   // rows of this team on their way
    auto layout_done = [&]() {
        if (!ready) {
            good = __all_sync(0xffffffffu, mbar_wait_idle(&ready_bar, 0, abortp) && !*abortp);   // no rows without a layout
            ready = true;
        }
    };
    auto send = [&]() {
        const int os = team * 2 + (sent & 1);
        fp8_issue<false>(x, q, q.out_ring + (size_t)os * pl.out_stage_bytes, (ch << 16) | (team + sent * teams), os);
        ++sent;
    };
    int i = 0;
    for (;; ++i) {
        const int n = team + i * teams;
        if (n >= ntok) break;
        const int s = n % stages;
        const unsigned par = (n / stages) & 1;
        if (tw == 1 && sent < i) {   // the first row still waits for the layout: whichever comes first
            const unsigned long long t_end = global_ns() + kWaitLimitNs;
            for (;;) {
                if (__any_sync(0xffffffffu, mbar_test_wait(&ready_bar, 0))) {
                    layout_done();
                    if (good) send();
                    break;
                }
                if (__any_sync(0xffffffffu, mbar_try_wait(&full_bar[s], par, 200u))) break;
                if (__any_sync(0xffffffffu, *abortp || global_ns() > t_end)) break;   // (the wait below gives up)
            }
        }
        good = good && __all_sync(0xffffffffu, mbar_wait_idle(&full_bar[s], par, abortp));
        if (tw == 1 && !good) break;
        if (i >= 2) {          // the copies of the row before the last one have read its slot
            if (m == 0) bulk_wait_read<1>();
            team_sync();
        }
        const int os = team * 2 + (i & 1);
        const uint8_t* src = smem + (size_t)s * pl.stage_bytes;
        uint8_t* dst = q.out_ring + (size_t)os * pl.out_stage_bytes;
        float* dst_scale = reinterpret_cast<float*>(dst + out_bytes);
        // four vectors per thread and trip, independent of each other
        for (int vb = m * 32; good && vb < nvec; vb += 4 * tw * 32) {
            uint4 in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int v = vb + u * tw * 32 + lane;
                in[u] = v < nvec ? *reinterpret_cast<const uint4*>(src + (size_t)v * 16) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int v = vb + u * tw * 32 + lane;
                uint2 o;
                float sc;
                quantize8(in[u], v < nvec, o, sc);
                if (v < nvec) {
                    *reinterpret_cast<uint2*>(dst + (size_t)v * 8) = o;
                    if ((lane & 15) == 0) dst_scale[v >> 4] = sc;
                }
            }
        }
        fence_proxy_async_smem();   // the bulk stores read what we just wrote
        // (each warp of a team begins as soon as the row is there, some of them before the rows are assigned; they leave together)
        if (tw > 1) good = !group_or(5 + team, tw * 32, !good);
        else __syncwarp();
        if (!good) break;
        if (lane == 0) mbar_arrive(&empty_bar[s]);
        if (m != 0) continue;
        if (tw == 1 && i == 0 && !ready && !__any_sync(0xffffffffu, mbar_test_wait(&ready_bar, 0))) continue;
        layout_done();
        while (good && sent <= i) send();
    }
    if (m == 0) {
        if (good && sent < i) layout_done();
        if (good && sent < i) send();
        if (!good && lane == 0) {
            report(p.status, kErrTimeout);
            *abortp = 1;
        }
        bulk_wait_all<0>();
    }
}

// --------------------------------------------------------------------- dispatch kernel
// Warp roles: warp 0 = mover; warps 1..15 = layout group (count, prefix sums, row assignment).  FP8 rows: warp 0 only loads,
// and some of the others quantise (plan_dispatch: q_warp0, q_warps):
//   clusters    all 15 warps count, then warps 6..15 quantise beside the rest of the layout, which warps 1..5 do;
//   FUSED, PHASED with a count group   the same with warps 1..count_warps; without one all 15 compute the layout and
//               warps 2..15 (short rows: 1..15, at most 14) quantise afterwards;
//   LOCAL       warps 1..4 assign the rows and then quantise with the next warps, five or six in all (warp 1 not with long
//               rows); the others write the expert-level outputs.
// Warp 1 issues the copies of long rows once the layout is done; short rows are sent by who quantised them.
//
// The flag-free instance for bf16 rows needs so few registers that two combine CTAs of top-8 (64 registers) would fit beside it.
// Then every combine CTA of a small batch is placed during the dispatch, the dispatch after it is let in as soon as this one
// leaves, and the combine runs with the registers that are left (sixteen layers of 128 tokens, top-8: 208 us; with one combine CTA
// beside it 179).  A warp that leaves at once holds the registers in question.  (The combines of top-4 and top-2 take 40 and 32
// registers, of which two and three CTAs still fit: no harm was seen there, 1 to 512 tokens of 256 to 2048 channels.)
template <int kMode, int kRows>
constexpr int kDispatchThreads = kThreads + (kMode == kModeLocal && kRows == kBf16Rows ? 32 : 0);
template <int kMode, int kRows, bool kSteal>
__global__ void __launch_bounds__((kDispatchThreads<kMode, kRows>), 1) dispatch_kernel(const Params p, const SmemPlan pl) {
    constexpr bool kFp8 = kRows != kBf16Rows, kLong = kRows == kLongFp8Rows;
    if ((kDispatchThreads<kMode, kRows>) > kThreads && threadIdx.x >= kThreads) return;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages];    // input row landed
    __shared__ __align__(8) uint64_t empty_bar[kMaxStages];   // FP8: input row consumed
    __shared__ __align__(8) uint64_t out_full[kMaxOutStages];    // FP8: quantised row written
    __shared__ __align__(8) uint64_t out_empty[kMaxOutStages];   // FP8: its stores have read it
    __shared__ __align__(8) uint64_t ready_bar;               // rows assigned, movers may go
    __shared__ __align__(8) uint64_t epoch_bar;               // epoch_sm holds this launch's epoch
    __shared__ __align__(8) uint64_t staged_bar;              // flag-free kernel: the routing table is in shared memory
    __shared__ int abort_flag;
    __shared__ unsigned epoch_sm;

    const int tid = threadIdx.x;
    const int c = blockIdx.x;
    const int part = c % p.parts, ch = c / p.parts;
    const int t0 = (int)chunk_begin(ch, p.T, p.nchunks), t1 = (int)chunk_begin(ch + 1, p.T, p.nchunks);
    const int stages = pl.stages;
    const bool beside = kFp8 && (kMode == kModeCluster || (kMode != kModeLocal && p.count_warps > 0));
    const int nw = kFp8 && kMode == kModeCluster ? kClusterCountWarps : beside ? p.count_warps : kWarps - 1;      // layout group: warps 1 .. nw
    int* arr = reinterpret_cast<int*>(smem + pl.off_arr);
    griddep_launch();   // the next kernel in the stream may be placed as soon as SMs have room

    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], !kFp8 ? 1 : kLong ? pl.q_warps : pl.q_team_warps);
        }
        for (int s = 0; kLong && s < pl.out_stages; ++s) {
            mbar_init(&out_full[s], pl.q_warps);
            mbar_init(&out_empty[s], 1);
        }
        mbar_init(&ready_bar, 1);
        mbar_init(&epoch_bar, 1);
        mbar_init(&staged_bar, 1);
        abort_flag = 0;
        epoch_sm = 0u;
        mbar_fence_init();
    }
    for (int r = tid; r < p.R; r += kThreads) arr[r] = 0;
    if (kMode == kModeCluster) {
        unsigned* cnt = reinterpret_cast<unsigned*>(smem + pl.off_cnt);
        unsigned* bm = reinterpret_cast<unsigned*>(smem + pl.off_bm);
        for (int b = tid; b < 2 * (p.B + 1); b += kThreads) cnt[b] = 0u;
        for (int b = tid; b < pl.map_groups * pl.map_bp; b += kThreads) bm[b] = 0u;
    }
    if (kMode == kModeLocal || kMode == kModeCluster) {
        // The routing table is the first thing every CTA of the flag-free kernel needs, and it comes cold
        // from HBM.  A prefetch into L2 reads no value, so it may run ahead of the wait below: L2 is where
        // an earlier kernel's stores to the table land too, so the line cannot go stale.
        const char* tab = reinterpret_cast<const char*>(p.topk_idx);
        const size_t bytes = (size_t)p.T * p.k * 4;
        for (size_t off = ((size_t)c * kThreads + tid) * 128; off < bytes; off += (size_t)p.grid * kThreads * 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(tab + off));
        // The same for the CTA's own pieces of its rows: inside a layer they come from HBM while it is still
        // writing back what the kernels before left in L2, and the first of them is what the first copy waits for.
        const unsigned piece = (unsigned)(p.H * 2 / p.parts);
        const int lines = (int)((piece + 127u) / 128u);
        const char* xs = reinterpret_cast<const char*>(p.x) + (size_t)t0 * p.H * 2 + (size_t)part * piece;
        for (int i = tid; kMode == kModeLocal && i < (t1 - t0) * lines; i += kThreads) {
            const int tl = i / lines, l = i - tl * lines;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(xs + (size_t)tl * p.H * 2 + (size_t)l * 128));
        }
    }
    griddep_wait();     // shared-memory set-up done; everything below reads what earlier kernels wrote
    // The epoch is not read here, in front of everything: the flag-free kernel needs it only for the
    // arrival counters at its very end and reads it once the movers are released; in the other
    // kernels the mover warp fetches it while the layout group stages the routing table.
    if (tid == 0) trace_begin(p, c);
    __syncthreads();
    const unsigned epoch = 0u;

    const unsigned in_bytes = (unsigned)(p.H * 2 / p.parts);   // this CTA's piece of a bf16 row
    const unsigned out_bytes = (unsigned)(p.rowB / p.parts);   // and of a payload row
    Cta x{p, pl, smem, full_bar, empty_bar, out_full, out_empty, &ready_bar, &epoch_bar, &staged_bar, &abort_flag,
          tid, tid & 31, tid >> 5, c, part, ch, t0, t1, t1 - t0, stages,
          nw * 32, nw, beside,
          reinterpret_cast<int*>(smem + pl.off_ids),
          reinterpret_cast<int*>(smem + pl.off_ord),    // destinations in issue order
          reinterpret_cast<int*>(smem + (p.ordered ? pl.off_pos : pl.off_ord)),   // in slot order (the same array
                                                                                  // when no table reorders them)
          reinterpret_cast<int*>(smem + pl.off_key),
          reinterpret_cast<float*>(smem + pl.off_w),
          BinMaps{reinterpret_cast<unsigned*>(smem + pl.off_mask), reinterpret_cast<unsigned*>(smem + pl.off_bm),
                  pl.map_wb, pl.map_bp, pl.map_groups},
          reinterpret_cast<int*>(smem + pl.off_hist), arr, reinterpret_cast<int*>(smem + pl.off_order),
          epoch, in_bytes, out_bytes, &epoch_sm, (size_t)part * in_bytes, (size_t)part * out_bytes,
          // (its stage is never loaded a second time, no order of destinations is asked for, a lane per copy)
          kMode == kModeLocal && !kFp8 && !kSteal && !p.ordered && p.k <= 32 && t1 > t0 &&
              t1 - t0 <= stages,
          0, kMode == kModeCluster || (kMode == kModeLocal && !kFp8),
          // the mover; the row group (rank-level rows, bf16) or the duty group (clusters); who issues FP8 copies
          1 + (kMode == kModeCluster ? nw - (kLong ? 1 : 0) : kFp8 ? 0 : kRowWarps) +
              (kLong ? 1 : kFp8 ? pl.q_warps : 0)};

    if (x.warp == 0) {
        mover_warp<kMode, kRows, kSteal>(x);
    } else {
        const int lg = layout_group<kMode, kRows, kSteal>(x);   // 0 = a wait ran out, 1 = done, 2 = left to quantise
        // (2: beside the rest of the layout; 1: after it, unless the quantising warps are others)
        const int qw = x.warp - pl.q_warp0;
        if (kLong && lg == 1 && x.warp == 1) {
            if constexpr (kLong) fp8_store_issuer<kSteal>(x);
            if (x.early_arrival) x.rows_landed(0);
        } else if (kFp8 && (lg == 2 || (lg == 1 && !beside)) && qw >= 0 && qw < pl.q_warps) {
            if constexpr (kLong) {
                fp8_quantiser<kSteal>(x, qw);
            } else if constexpr (kFp8) {
                fp8_worker(x, qw);
                if (x.early_arrival) x.rows_landed(0);
            }
        }
    }
    if (kMode == kModeCluster) cluster_wait();   // the others have read what this CTA counted
    __syncthreads();
    const unsigned half = epoch_sm & 1u;
    if (abort_flag) {
        // leaving early.  The arrival counters of the next call live in the other half; they are
        // cleared here too, otherwise the call after the next one would add to stale totals.
        // (epoch_sm == 0: the call gave up before it learnt its epoch and has used neither half.)
        if (c == 0 && epoch_sm != 0u) {
            for (int r = tid; r < p.R; r += kThreads) p.arrival[(half ^ 1u) * p.R + r] = 0;
            if (tid == 0) p.claimed[half ^ 1u] = 0;
        }
        // the newest load of every ring stage may still be landing
        if (tid == 0) {
            for (int n = max(0, x.issued - stages); n < x.issued; ++n)
                (void)mbar_wait(&full_bar[n % stages], (n / stages) & 1, nullptr);
        }
        return;
    }
    if (!x.early_arrival) publish_arrivals(p, arr, half, tid, kThreads);
    // the arrival counters of the next call live in the other half; clear them now
    if (c == 0) {
        for (int r = tid; r < p.R; r += kThreads) p.arrival[(half ^ 1u) * p.R + r] = 0;
        if (tid == 0) p.claimed[half ^ 1u] = 0;   // same for the count of tokens handed out
    }
    if (tid == 0) trace(p, c, kTrEnd);
}

// ---------------------------------------------------------------------------- combine
// One thread per 16-byte vector of the output row: K independent 128-bit gathers, fp32
// fused multiply-adds in slot order, one round-to-nearest-even pack to bf16.
// kStream: rows are read past L1 (nothing is read twice).  Measured for the combine alone: 512 tokens of 7168 channels, top-8, one row
// per (token, rank) 11.7 -> 10.2 us, 1537 tokens of 4096 channels 21.7 -> 18.7, but 4096 tokens of 7168 channels 82 -> 88 and
// 16384 tokens 307 -> 338: the line lies at 384 MB of gathered rows (3000 tokens, 344 MB: dispatch + combine 139.2 -> 138.2).
constexpr int64_t kStreamMaxBytes = 384ll << 20;
template <bool kStream>
__device__ __forceinline__ uint4 load_row16(const uint4* a) {
    uint4 v;   // (plain loads: see ld_plain)
    if (!kStream) {
        asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
        return v;
    }
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
    return v;
}
template <int K, bool kStream>
__global__ void __launch_bounds__(256) combine_kernel(const uint16_t* y, const int32_t* slot_pos, const float* topk_w,
                                                     int T, int H, int k, uint16_t* __restrict__ out) {
    const int nvec = H / 8;
    const int64_t total = (int64_t)T * nvec;
    const int kk = K > 0 ? K : k;
    griddep_launch();   // lets a dispatch that follows in the stream be placed while this kernel drains
    griddep_wait();
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total;
         u += (int64_t)gridDim.x * blockDim.x) {
        // (small calls: no 64-bit division and no scalar loads in front of the first row; in large ones, 16384 tokens, the
        // same changes cost half a percent)
        const int t = kStream && total <= 0x7fffffff ? (int)((unsigned)u / (unsigned)nvec) : (int)(u / nvec);
        const int v = (int)(u - (int64_t)t * nvec);
        float acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
        if (K > 0) {
            constexpr int KK = K > 0 ? K : 1;
            uint4 q[KK];
            float w[KK];
            int wh[KK];
            if (kStream && KK % 4 == 0) {   // (both arrays start on 16-byte boundaries)
#pragma unroll
                for (int j = 0; j + 3 < KK; j += 4) {
                    const int4 a = ld_plain(reinterpret_cast<const int4*>(slot_pos + (size_t)t * KK + j));
                    wh[j] = a.x; wh[j + 1] = a.y; wh[j + 2] = a.z; wh[j + 3] = a.w;
                }
#pragma unroll
                for (int j = 0; j + 3 < KK; j += 4) {
                    const float4 b = ld_plain(reinterpret_cast<const float4*>(topk_w + (size_t)t * KK + j));
                    w[j] = b.x; w[j + 1] = b.y; w[j + 2] = b.z; w[j + 3] = b.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < KK; ++j) {
                    wh[j] = ld_plain(slot_pos + (size_t)t * KK + j);
                    w[j] = ld_plain(topk_w + (size_t)t * KK + j);
                }
            }
#pragma unroll
            for (int j = 0; j < KK; ++j) {
                q[j] = make_uint4(0, 0, 0, 0);
                if (wh[j] >= 0) q[j] = load_row16<kStream>(reinterpret_cast<const uint4*>(y + (size_t)wh[j] * H) + v);
            }
#pragma unroll
            for (int j = 0; j < KK; ++j) {
                if (wh[j] < 0) continue;  // an empty slot contributes nothing
                const uint32_t ww[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[2 * i] = __fmaf_rn(w[j], __uint_as_float(ww[i] << 16), acc[2 * i]);
                    acc[2 * i + 1] = __fmaf_rn(w[j], __uint_as_float(ww[i] & 0xffff0000u), acc[2 * i + 1]);
                }
            }
        } else {
            for (int j = 0; j < kk; ++j) {
                const int where = ld_plain(slot_pos + (size_t)t * kk + j);
                if (where < 0) continue;
                const float w = ld_plain(topk_w + (size_t)t * kk + j);
                const uint4 q = load_row16<kStream>(reinterpret_cast<const uint4*>(y + (size_t)where * H) + v);
                const uint32_t ww[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[2 * i] = __fmaf_rn(w, __uint_as_float(ww[i] << 16), acc[2 * i]);
                    acc[2 * i + 1] = __fmaf_rn(w, __uint_as_float(ww[i] & 0xffff0000u), acc[2 * i + 1]);
                }
            }
        }
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
            o[i] = *reinterpret_cast<uint32_t*>(&h);
        }
        reinterpret_cast<uint4*>(out + (size_t)t * H)[v] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// ---------------------------------------------------------------- counts-only layout
// ubep_get_dispatch_layout.  A lane per token: its slots are fetched side by side (16 bytes each where the table allows it), the
// experts and the ranks it visits are counted in shared memory, and which ranks those are becomes a tile of 32 tokens' bytes in
// shared memory that leaves in 16-byte stores.
//
// Bound by latency: table (cold, 1.2 us) -> counts -> sums over the CTAs.  kCluster: the CTAs are one cluster and read one
// another's counts; nothing outside shared memory is needed, and one CTA needs not even that.  Otherwise a CTA adds its
// counts to the totals in `acc`, and the last one to finish (ticket) hands them out and leaves `acc` and the ticket zero for
// the next call: a fence and two round trips to L2 more, but as many SMs as there are tokens for.
// Captured calls, top-8 of 256 experts on 32 ranks, one cluster / totals in global memory: 1 token 2.6 / 4.6 us, 512 tokens 3.2 / 4.9, 4096
// tokens 4.4 / 5.3, 8192 tokens 6.2 / 5.4; top-4 of 32 experts on 8 ranks 1 token 2.0 / 3.3, 4096 tokens 3.1 / 4.0, 8192 tokens 4.4 / 4.1.  (Rank
// masks per lane, transposed by the warp, and no cluster: 4.8, 5.2, 5.7 and 5.8 us on 32 ranks; with four words of masks, 72 ranks,
// 4096 tokens 7.0, now 4.8.)
constexpr int kLayoutThreads = 128;
constexpr int kLayoutClusterTokens = 8 * kThreads;   // eight CTAs, a token per thread
constexpr int kLayoutTileRanks = 128;   // most ranks whose bytes go through shared memory

// kK: slots per token if fixed (0: p.k, at most kMaxTopk); kTile: no more ranks than kLayoutTileRanks
template <int kK, bool kTile, bool kCluster>
__global__ void __launch_bounds__(kCluster ? kThreads : kLayoutThreads) layout_kernel(const Params p, int32_t* num_tokens_per_rank,
                                                               int32_t* num_tokens_per_expert,
                                                               uint8_t* is_token_in_rank, int32_t* acc,
                                                               int acc_words, unsigned* ticket) {
    extern __shared__ __align__(16) int hist[];   // [B], then a tile per warp
    __shared__ bool last;
    constexpr int kN = kCluster ? kThreads : kLayoutThreads, kSlots = kK ? kK : kMaxTopk, kUnroll = kK ? kK : 1;
    const int B = p.B, R = p.R, T = p.T, k = kK ? kK : p.k, lane = threadIdx.x & 31;
    uint8_t* tile = reinterpret_cast<uint8_t*>(hist + (B + 3) / 4 * 4) + (threadIdx.x >> 5) * 32 * R;   // [32, R]
    for (int b = threadIdx.x; b < B; b += kN) hist[b] = 0;
    griddep_launch();
    griddep_wait();
    __syncthreads();
    const int warps = gridDim.x * (kN / 32);
    bool bad = false;
    for (int g = blockIdx.x * (kN / 32) + (threadIdx.x >> 5); g * 32 < T; g += warps) {
        const int t = g * 32 + lane;
        const bool flags = is_token_in_rank != nullptr;
        uint8_t* out = flags ? is_token_in_rank + (size_t)g * 32 * R : nullptr;
        if (kTile && flags) {
            for (int i = lane; i < 2 * R; i += 32) reinterpret_cast<uint4*>(tile)[i] = make_uint4(0, 0, 0, 0);
            __syncwarp();
        }
        if (t < T) {
            const int32_t* src = p.topk_idx + (size_t)t * k;
            int e[kSlots];
            if (kK % 4 == 0 && kK > 0) {
#pragma unroll
                for (int j = 0; j < kSlots; j += 4) {
                    const int4 v = ld_plain(reinterpret_cast<const int4*>(src + j));
                    e[j] = v.x; e[j + 1] = v.y; e[j + 2] = v.z; e[j + 3] = v.w;
                }
            } else {
#pragma unroll kUnroll
                for (int j = 0; j < k; ++j) e[j] = ld_plain(src + j);
            }
            uint8_t* mine = !flags ? nullptr : kTile ? tile + lane * R : out + (size_t)lane * R;
            if (!kTile && flags)
                for (int r = 0; r < R; ++r) mine[r] = 0;
            if (kK) {
                resolve_slots(p, t, e, bad);
                bool twice = false;
#pragma unroll
                for (int j = 0; j < kSlots; ++j) {
                    e[j] = e[j] >= 0 ? e[j] : -1 - j;   // (no two empty slots are equal)
#pragma unroll
                    for (int i = 0; i < j; ++i) twice = twice || e[i] == e[j];
                }
                if (twice) {   // an expert named twice: reported, the later slot counts as empty
                    bad = true;
#pragma unroll
                    for (int j = 1; j < kSlots; ++j)
#pragma unroll
                        for (int i = 0; i < j; ++i)
                            if (e[i] == e[j]) e[j] = -1 - j;
                }
#pragma unroll
                for (int j = 0; j < kSlots; ++j) {
                    if (e[j] >= 0) atomicAdd(&hist[e[j]], 1);
                    e[j] = e[j] < 0 ? e[j] : p.L == 1 ? e[j] : fast_div(e[j], p.L_magic);
                    bool first = e[j] >= 0;   // a rank counts a token once: with the first of the slots that name it
#pragma unroll
                    for (int i = 0; i < j; ++i) first = first && e[i] != e[j];
                    if (first) {
                        atomicAdd(&hist[p.E + e[j]], 1);
                        if (flags) mine[e[j]] = 1;
                    }
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < k; ++j) {
                    e[j] = resolve_expert(p, t, e[j], bad);
#pragma unroll 1
                    for (int i = 0; i < j; ++i)
                        if (e[j] >= 0 && e[i] == e[j]) {
                            bad = true;
                            e[j] = -1;
                        }
                    if (e[j] < 0) continue;
                    atomicAdd(&hist[e[j]], 1);
                    const int r = p.L == 1 ? e[j] : fast_div(e[j], p.L_magic);
                    bool first = true;
#pragma unroll 1
                    for (int i = 0; i < j; ++i) first = first && !(e[i] >= r * p.L && e[i] < (r + 1) * p.L);
                    if (first) {
                        atomicAdd(&hist[p.E + r], 1);
                        if (flags) mine[r] = 1;
                    }
                }
            }
        }
        if (kTile && flags) {
            __syncwarp();
            const int bytes = min(32, T - g * 32) * R;
            if ((reinterpret_cast<uintptr_t>(is_token_in_rank) & 15) == 0) {   // (32 tokens' bytes start on a 32-byte boundary)
                for (int i = lane; i < bytes / 16; i += 32) reinterpret_cast<uint4*>(out)[i] = reinterpret_cast<const uint4*>(tile)[i];
                for (int i = bytes / 16 * 16 + lane; i < bytes; i += 32) out[i] = tile[i];
            } else {
                for (int i = lane; i < bytes; i += 32) out[i] = tile[i];
            }
            __syncwarp();   // (the tile is used again)
        }
    }
    if (bad) report(p.status, kErrBadIndex);
    if (kCluster) {
        const int cs = gridDim.x;
        cluster_arrive();
        cluster_wait();
        for (int b = (int)threadIdx.x * cs + (int)blockIdx.x; b < B; b += kN * cs) {
            unsigned sum = 0u;
#pragma unroll 8
            for (int q = 0; q < cs; ++q) sum += ld_cluster(reinterpret_cast<const unsigned*>(hist) + b, (unsigned)q);
            if (b < p.E) {
                if (num_tokens_per_expert) num_tokens_per_expert[b] = (int)sum;
            } else if (num_tokens_per_rank) {
                num_tokens_per_rank[b - p.E] = (int)sum;
            }
        }
        cluster_arrive();   // (a CTA's counts stay until all have read them)
        cluster_wait();
        return;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < B; b += kN)
        if (hist[b]) atomicAdd(acc + b, hist[b]);
    __threadfence();
    __syncthreads();
    // The shares of a grid's CTAs add up to 2^32, so the ticket is zero again when all have come, whatever else is under
    // way: calls that overlap on the GPU (which share the totals, so that their answers are undefined) leave nothing behind.
    const unsigned share = 0xffffffffu / gridDim.x;
    const unsigned mine = blockIdx.x == 0 ? 0u - share * (gridDim.x - 1u) : share;
    if (threadIdx.x == 0) last = atomicAdd(ticket, mine) + mine == 0u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int b = threadIdx.x; b < B; b += kN) {
        const int sum = atomicExch(acc + b, 0);   // (zero for the next call)
        if (b < p.E) {
            if (num_tokens_per_expert) num_tokens_per_expert[b] = sum;
        } else if (num_tokens_per_rank) {
            num_tokens_per_rank[b - p.E] = sum;
        }
    }
    for (int b = B + threadIdx.x; b < acc_words; b += kN) acc[b] = 0;   // (an overlapping call may have had more bins)
}

// ------------------------------------------------------------------------- launchers

static int round_up_i(int v, int m) { return (v + m - 1) / m * m; }

// Rows (pieces of rows) that the kernel sends several at a time: see send_short_rows and the comment above Fp8Ring.
bool short_rows(const Params& p) {
    const int64_t copies = (int64_t)p.k * (p.rowB / p.parts);
    return p.payload ? copies < 40 * 1024 : p.k <= 16 && copies <= 16384;
}

// Shared-memory plan of the dispatch kernel for one call; -1 if it cannot fit.
int plan_dispatch(const Params& p, int mode, int max_smem, SmemPlan* out) {
    SmemPlan pl{};
    const int chunk_tokens = (p.T + p.nchunks - 1) / p.nchunks;
    const int chunk_slots = chunk_tokens * p.k;
    const int map_tokens = mode == kModeLocal ? p.T : chunk_tokens;   // tokens the bitmaps cover
    const int64_t ids_ints = (int64_t)map_tokens * p.k;
    int hist_ints = mode == kModeLocal || mode == kModeCluster ? 2 * p.B + p.E : 2 * p.B;
    if (hist_ints < 64) hist_ints = 64;   // the per-rank duty of the flag-free kernel keeps 2 x 32 ints here
    pl.map_groups = map_tokens / 32 + (mode == kModeCluster || map_tokens % 32 != 0 ? 1 : 0);   // (own_below may look at one more)
    pl.map_wb = (p.B + 31) / 32;
    pl.map_bp = pl.map_wb * 32;
    pl.stage_bytes = round_up_i(p.H * 2 / p.parts, 128);
    pl.out_stage_bytes = p.payload ? round_up_i(p.rowB / p.parts + (p.G / p.parts) * 4, 128) : 0;
    const bool fast = mode == kModeLocal && p.local_fast;
    const int64_t mask_ints = (int64_t)(fast ? 2 * pl.map_groups + 1 : pl.map_groups) * 32;   // (fast: local_rank_duty)
    const int64_t bm_ints = (int64_t)pl.map_groups * pl.map_bp;
    const bool beside = p.payload && (mode == kModeCluster || (mode != kModeLocal && p.count_warps > 0));
    if (p.payload) {   // who quantises, and how (see Fp8Ring)
        pl.q_long = short_rows(p) ? 0 : 1;
        pl.q_warp0 = beside ? (mode == kModeCluster ? kClusterCountWarps : p.count_warps) + 1 : pl.q_long ? 2 : 1;
        const int most = fast ? kFastQuantWarps + (pl.q_long ? 0 : 1) : kWarps - pl.q_warp0;
        pl.q_warps = p.quant_warps < most ? p.quant_warps : most;
        pl.q_teams = pl.q_warps;
        if (pl.q_teams > chunk_tokens) pl.q_teams = chunk_tokens < 1 ? 1 : chunk_tokens;
        pl.out_stages = !pl.q_long ? 2 * pl.q_teams : beside ? kMaxOutStages : kOutStages;   // at most
    }
    const int item_ints = p.steal ? (kStealStages + pl.out_stages) * (p.k + 1) : 0;
    const int max_stages = p.steal ? kStealStages : kMaxStages;
    const int64_t cnt_ints = mode == kModeCluster ? 3 * ((int64_t)p.B + 1) : 0;
    const int64_t ints = ids_ints + mask_ints + bm_ints + 4 * (int64_t)chunk_slots + hist_ints + 2 * p.R + item_ints +
                         cnt_ints;
    const int64_t fixed = ints * 4 + 128 + 1536;  // 1.5 KB: static shared memory
    // no more stages than rows this CTA will ever hold at once
    const int want = chunk_tokens + 3 < 4 ? 4 : chunk_tokens + 3;
    int64_t room = max_smem - fixed;
    const int64_t in = pl.stage_bytes, out_b = pl.out_stage_bytes;
    if (p.payload && !pl.q_long) {
        // Two quantised rows per team, the rest for rows that have been fetched: as many as there are teams at least.
        while (pl.q_teams > 1 && room < pl.q_teams * (in + 2 * out_b)) --pl.q_teams;
        pl.q_team_warps = pl.q_warps / pl.q_teams;
        pl.out_stages = 2 * pl.q_teams;
    } else if (beside) {
        // the quantising warps run beside the layout: a short input ring (enough loads in flight to keep them busy) and
        // as many quantised rows as fit, which wait for the layout.  (Otherwise they start after the layout: a deep
        // input ring that the loader fills meanwhile, a short ring of quantised rows.)
        int st = 4;
        while (st > 2 && room < st * in + 4 * out_b) --st;
        if (room < st * in + 4 * out_b) return -1;
        const int64_t fit = (room - st * in) / out_b;
        if (pl.out_stages > fit) pl.out_stages = (int)fit;
        if (pl.out_stages > want) pl.out_stages = want;
    }
    room -= pl.out_stages * out_b;
    const int least = p.payload && !p.steal ? 2 : 4;   // (stealing looks at the row three back)
    if (room < least * in) return -1;
    pl.stages = room / in > max_stages ? max_stages : (int)(room / in);
    if (pl.stages > want) pl.stages = want;
    // Teams: where the ring is used more than once, every stage belongs to one team (row n is in stage n % stages and
    // goes to team n % teams).  A team waits by the parity of the stage's barrier, which only tells the row it waits for
    // from the row that had the stage before: that one must have landed, and loads land in any order, so it must have been
    // this team's own.  (A team needs one stage: rows leave an SM at 0.9 us each at 32 KB of copies, a load takes about as long.)
    if (p.payload && !pl.q_long && pl.stages < chunk_tokens) pl.stages -= pl.stages % pl.q_teams;
    int at = pl.stages * pl.stage_bytes;
    const int copies = p.k * (p.rowB / p.parts);
    pl.trip_rows = 1;
    if (!p.payload && !p.steal && chunk_tokens > 2 && short_rows(p)) {
        pl.trip_rows = 32 / p.k < 32768 / copies ? 32 / p.k : 32768 / copies;
        if (chunk_tokens > pl.stages && pl.trip_rows > pl.stages / 3) pl.trip_rows = pl.stages / 3 > 1 ? pl.stages / 3 : 1;
    }
    pl.off_out = at; at += pl.out_stages * pl.out_stage_bytes;
    pl.off_ids = at; at += (int)ids_ints * 4;
    pl.off_mask = at; at += (int)mask_ints * 4;
    pl.off_bm = at; at += (int)bm_ints * 4;
    pl.off_pos = at; at += chunk_slots * 4;
    pl.off_key = at; at += chunk_slots * 4;
    pl.off_ord = at; at += chunk_slots * 4;
    pl.off_w = at; at += chunk_slots * 4;
    pl.off_hist = at; at += hist_ints * 4;
    pl.off_arr = at; at += p.R * 4;
    pl.off_order = at; at += p.R * 4;
    pl.off_item = at; at += item_ints * 4;
    pl.off_cnt = at; at += (int)cnt_ints * 4;
    pl.total = round_up_i(at, 128);
    *out = pl;
    return 0;
}

template <int kMode, int kRows, bool kSteal>
static cudaError_t allow_dispatch_smem(int bytes) {
    static std::atomic<int> granted[kAttrDevices];
    return allow_dynamic_smem(reinterpret_cast<const void*>(dispatch_kernel<kMode, kRows, kSteal>), bytes, granted);
}

// An SM's shared memory comes in a few sizes, and a kernel gets the smallest that holds its CTA (its dynamic and static
// memory and the 1 KB every CTA takes).  Where that leaves less than 1 KB, no combine CTA can be placed beside the dispatch:
// layers of 74 tokens of 1024 channels, FP8, in one graph, 15.4 of 16 KB, 10.6 us, with the next size 9.9; 128 tokens of 256
// channels, 7.5 of 8 KB, 10.2 and 9.5; 74 tokens of 2048 channels, bf16, 9.1 and 8.5.  So such a call asks for a little more.
// (The largest size for every call: 512 tokens of 7168 channels 24.3 -> 25.6, more combine CTAs beside the dispatch.)
int with_room_beside(int dynamic, int least_static) {
    const int kLeast = least_static + 1024, kMost = 1280 + 1024;   // static memory of the dispatch kernels, reserved
    for (int kb : {8, 16, 32, 64, 100, 132, 164, 196}) {
        const int size = kb * 1024;
        if (dynamic + kLeast <= size && dynamic + kMost + 1024 > size) return size - kLeast + 128;
    }
    return dynamic;
}

template <int kMode, int kRows, bool kSteal>
static cudaError_t launch_dispatch_s(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    auto kern = dispatch_kernel<kMode, kRows, kSteal>;
    const int smem = with_room_beside(pl.total, kLeastStatic);
    cudaError_t e = allow_dispatch_smem<kMode, kRows, kSteal>(smem);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, p.grid, kDispatchThreads<kMode, kRows>, (size_t)smem, st, kMode == kModeFused,
                             kMode == kModeCluster ? p.cluster : 1, p, pl);
}

template <int kMode>
static cudaError_t launch_dispatch_t(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    if constexpr (kMode != kModeLocal) {
        if (p.steal) return p.payload ? launch_dispatch_s<kMode, kLongFp8Rows, true>(p, pl, st)
                                      : launch_dispatch_s<kMode, kBf16Rows, true>(p, pl, st);
    }
    if (!p.payload) return launch_dispatch_s<kMode, kBf16Rows, false>(p, pl, st);
    return pl.q_long ? launch_dispatch_s<kMode, kLongFp8Rows, false>(p, pl, st)
                     : launch_dispatch_s<kMode, kShortFp8Rows, false>(p, pl, st);
}

// TokenCnt and CalCumSum as two launches over the whole routing table (chunk histograms, then per rank
// the prefix over chunks, expert offsets, totals and the per-source tables).
cudaError_t launch_count_scan(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    cudaError_t e;
    const int count_smem = pl.off_pos - pl.off_ids;   // ids + both bitmap arrays
    static std::atomic<int> granted[kAttrDevices];
    if ((e = allow_dynamic_smem(reinterpret_cast<const void*>(count_kernel), count_smem, granted)) != cudaSuccess)
        return e;
    count_kernel<<<p.nchunks, 256, count_smem, st>>>(p, pl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int scan_smem = (int)sizeof(int) * (p.L + 1);
    static std::atomic<int> scan_granted[kAttrDevices];
    if (scan_smem > 48 * 1024 &&
        (e = allow_dynamic_smem(reinterpret_cast<const void*>(scan_kernel), scan_smem, scan_granted)) != cudaSuccess)
        return e;
    scan_kernel<<<p.R, 256, scan_smem, st>>>(p);
    return cudaGetLastError();
}

// CTAs of the dispatch kernel, one per SM, that can run at once in clusters of `cluster` on the current device (SMs are
// grouped, and a group's size need not be a multiple of the cluster's: on a B200 148, 132, 120 for 2, 4, 8).
int cluster_ctas(int cluster, int max_smem) {
    static std::atomic<int> known[kAttrDevices][4];
    const int slot = cluster == 2 ? 1 : cluster == 4 ? 2 : cluster == 8 ? 3 : 0;
    int dev = 0;
    if (slot == 0 || cudaGetDevice(&dev) != cudaSuccess) return 0;
    const bool cached = dev >= 0 && dev < kAttrDevices;
    if (cached) {
        const int v = known[dev][slot].load(std::memory_order_relaxed);
        if (v) return v - 1;
    }
    const int smem = max_smem - 2048;   // (more than half of an SM's: one CTA per SM)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cluster);
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (allow_dispatch_smem<kModeCluster, kBf16Rows, false>(smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(dispatch_kernel<kModeCluster, kBf16Rows, false>), &cfg) != cudaSuccess)
        n = 0;
    (void)cudaGetLastError();
    if (cached) known[dev][slot].store(n * cluster + 1, std::memory_order_relaxed);
    return n * cluster;
}

cudaError_t launch_dispatch(const Params& p, int mode, const SmemPlan& pl, cudaStream_t st, int* launches) {
    cudaError_t e;
    *launches = 1;
    if (mode == kModePhased) {
        if ((e = launch_count_scan(p, pl, st)) != cudaSuccess) return e;
        *launches = 3;
        return launch_dispatch_t<kModePhased>(p, pl, st);
    }
    if (mode == kModeFew) return launch_few(p, pl, st);
    if (mode == kModeCluster) return launch_dispatch_t<kModeCluster>(p, pl, st);
    if (mode == kModeLocal) return launch_dispatch_t<kModeLocal>(p, pl, st);
    return launch_dispatch_t<kModeFused>(p, pl, st);
}

// Both kinds of calls are placed while their predecessor still runs (and wait for its end before they read anything).  A large
// one asks for as much L1 as there is: its gathers land there, and beside a dispatch or behind one whose division of the SM it
// inherits, with most of it shared memory, it takes a quarter longer (prefill 80 -> 102 us).  So it is placed only where that
// division can be changed, SM by SM as the dispatch's CTAs leave, not behind the last of them: dispatch + combine of 1537 tokens of 4096
// channels, top-8 43.9 -> 43.3 us against an ordinary launch, 2500 tokens of 2048 channels, top-4 26.2 -> 25.7, 4096 of 7168, FP8, 148.8 ->
// 147.9; placed ahead without asking 46.0, 26.6 and 169.6.  Small calls don't wait for it: 128 tokens of 256 channels 4.6 us, 5.4 with it.
template <int K, bool kStream>
static cudaError_t launch_combine_s(bool small, int g, cudaStream_t st, const uint16_t* y, const int32_t* slot_pos,
                                    const float* topk_w, int T, int H, int k, uint16_t* out) {
    if (small) return launch_overlapped(combine_kernel<K, kStream>, g, 256, 0, st, false, 1, y, slot_pos, topk_w, T, H, k, out);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxL1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, combine_kernel<K, kStream>, y, slot_pos, topk_w, T, H, k, out);
}
template <int K>
static cudaError_t launch_combine_k(bool small, int g, cudaStream_t st, const uint16_t* y, const int32_t* slot_pos,
                                    const float* topk_w, int T, int H, int k, uint16_t* out) {
    if ((int64_t)T * k * H * 2 <= kStreamMaxBytes) return launch_combine_s<K, true>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
    return launch_combine_s<K, false>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
}

cudaError_t launch_combine(const uint16_t* y, const int32_t* slot_pos, const float* topk_w, int T, int H, int k,
                           uint16_t* out, int num_sms, bool small, cudaStream_t st) {
    const int64_t total = (int64_t)T * (H / 8);
    int64_t blocks = (total + 255) / 256;
    const int64_t cap = (int64_t)num_sms * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const int g = (int)blocks;
    switch (k) {
        case 1: return launch_combine_k<1>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
        case 2: return launch_combine_k<2>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
        case 4: return launch_combine_k<4>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
        case 6: return launch_combine_k<6>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
        case 8: return launch_combine_k<8>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
        default: return launch_combine_k<0>(small, g, st, y, slot_pos, topk_w, T, H, k, out);
    }
}

// A kernel that does nothing, one CTA per SM: what a launch costs by itself.
__global__ void __launch_bounds__(32) empty_kernel(int) {
    griddep_launch();
    griddep_wait();
}

cudaError_t launch_empty(int num_sms, bool ahead, cudaStream_t st) {
    if (ahead) return launch_overlapped(empty_kernel, num_sms, 32, 0, st, false, 1, 0);
    empty_kernel<<<num_sms, 32, 0, st>>>(0);
    return cudaGetLastError();
}

template <int kK, bool kTile, bool kCluster>
static cudaError_t launch_layout_t(const Params& p, int blocks, int smem, int32_t* per_rank, int32_t* per_expert, uint8_t* in_rank,
                                   int32_t* acc, int acc_words, unsigned* ticket, cudaStream_t st) {
    auto kern = layout_kernel<kK, kTile, kCluster>;
    if (smem > 48 * 1024) {
        static std::atomic<int> granted[kAttrDevices];
        const cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void*>(kern), smem, granted);
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(kern, blocks, kCluster ? kThreads : kLayoutThreads, (size_t)smem, st, false, kCluster ? blocks : 1, p,
                             per_rank, per_expert, in_rank, acc, acc_words, ticket);
}

cudaError_t launch_layout(const Params& p, int32_t* num_tokens_per_rank, int32_t* num_tokens_per_expert,
                          uint8_t* is_token_in_rank, int32_t* acc, int acc_words, unsigned* ticket, cudaStream_t st) {
    const bool tile = p.R <= kLayoutTileRanks;
    const int counts = (p.B + 3) / 4 * 16;
    if (p.B * 4 > 48 * 1024) return cudaErrorInvalidValue;   // (the counts of some twelve thousand bins at most)
    const bool cluster = p.T <= kLayoutClusterTokens;
    const int threads = cluster ? kThreads : kLayoutThreads;
    // a token per thread; beyond one cluster (two CTAs per SM) a thread takes several
    int64_t blocks = ((int64_t)p.T + threads - 1) / threads;
    const int64_t most = cluster ? kLayoutClusterTokens / kThreads : 296;
    if (blocks > most) blocks = most;
    if (blocks < 1) blocks = 1;
    while (cluster && (blocks & (blocks - 1)) != 0) ++blocks;   // a power of two
    const int smem = counts + (tile ? threads * p.R : 0);
    auto go = [&](auto kk, auto tl) {
        if (cluster) return launch_layout_t<kk(), tl(), true>(p, (int)blocks, smem, num_tokens_per_rank, num_tokens_per_expert, is_token_in_rank, acc, acc_words, ticket, st);
        return launch_layout_t<kk(), tl(), false>(p, (int)blocks, smem, num_tokens_per_rank, num_tokens_per_expert, is_token_in_rank, acc, acc_words, ticket, st);
    };
    auto by_k = [&](auto tl) {
        switch (p.k) {
            case 2: return go(std::integral_constant<int, 2>{}, tl);
            case 4: return go(std::integral_constant<int, 4>{}, tl);
            case 6: return go(std::integral_constant<int, 6>{}, tl);
            case 8: return go(std::integral_constant<int, 8>{}, tl);
            default: return go(std::integral_constant<int, 0>{}, tl);
        }
    };
    return tile ? by_k(std::true_type{}) : by_k(std::false_type{});
}

}  // namespace ubep
