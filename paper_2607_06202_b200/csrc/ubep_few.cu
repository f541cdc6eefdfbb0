// Dispatch of small batches: a CTA has no more slots of the routing table than warps (plan_few below).
//
// What bounds it is latency, not bytes: 13 tokens are 1.4 MB.  The kernels for larger batches spend most of such a call on
// control flow that is worth its while only with many rows -- rings, roles that release one another through barriers, counting
// and prefix sums through shared memory, and every jump to a piece of code that has not run yet costs 0.15 us (64 functions 2 KB
// apart, called once: 300 cycles each, 190 the second time; code that runs straight on: 3.5 cycles per instruction).  Here the
// table is staged once; then every slot of the CTA's own tokens is a warp's, which counts the table for its own expert and rank
// alone, sends its copy, writes its metadata and adds to the arrival counter by itself.  There is no barrier after the
// one behind the staging (FP8 rows: one more, between quantising and sending).
#include "ubep_few.cuh"
#include "ubep_kernels.h"
#include "ubep_launch.cuh"
#include "ubep_quant.cuh"

namespace ubep {

namespace {

constexpr int kFewSmem = 120 * 1024;   // more than half of an SM's shared memory

// kTraced: with time stamps, an instance of its own: behind run-time branches they were 0.2 us of code in every call (sixteen layers of
// 128 tokens of 7168 channels in one graph 154.4 us, without it 151.4).
template <int K, bool kFp8, bool kDedup, bool kTraced>
__global__ void __launch_bounds__(kThreads, 1) few_kernel(const Params p, const SmemPlan pl) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t row_bar[kWarps];   // per own token: its row has landed
    __shared__ unsigned epoch_sm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = blockIdx.x;
    const int part = c % p.parts, ch = c / p.parts;
    const int t0 = (int)chunk_begin(ch, p.T, p.nchunks), ntok = (int)chunk_begin(ch + 1, p.T, p.nchunks) - t0;
    const unsigned in_bytes = (unsigned)(p.H * 2 / p.parts), out_bytes = (unsigned)(p.rowB / p.parts);
    const size_t out_off = (size_t)part * out_bytes;
    const uint8_t* xs = reinterpret_cast<const uint8_t*>(p.x) + (size_t)t0 * p.H * 2 + (size_t)part * in_bytes;
    uint16_t* ids = reinterpret_cast<uint16_t*>(smem + pl.off_ids);
    auto mark = [&](int phase) {   // the whole CTA has come this far (every warp sends rows of its own: a stamp by one of them says little)
        if (!kTraced) return;
        __syncthreads();
        if (tid == 0) trace(p, c, phase);
    };
    griddep_launch();
    if (warp == 0) {
        if (lane < ntok) mbar_init(&row_bar[lane], 1);
        mbar_fence_init();
    }
    {   // (prefetches into L2 read no value, so they may run ahead of the wait: see dispatch_kernel)
        const char* tab = reinterpret_cast<const char*>(p.topk_idx);
        if (tid * 128 < p.T * K * 4) asm volatile("prefetch.global.L2 [%0];" ::"l"(tab + tid * 128));
        if (p.phys != nullptr) {
            if (tid * 32 < p.E_log) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.ncopies + tid * 32));
            if (tid * 32 < (int64_t)p.E_log * p.C) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.phys + tid * 32));
        }
        const int lines = (int)((in_bytes + 127u) / 128u);
        for (int tl = 0; tl < ntok; ++tl)
            for (int i = tid; i < lines; i += kThreads) asm volatile("prefetch.global.L2 [%0];" ::"l"(xs + (size_t)tl * p.H * 2 + (size_t)i * 128));
    }
    griddep_wait();
    if (kTraced && tid == 0) trace_begin(p, c);

    // ---- the routing table, by warps 1 .. 15; warp 0 asks for the own rows and for the epoch
    bool bad = false;
    if (warp == 0) {
        const unsigned ctr = lane == 0 ? ld_relaxed(p.epoch_ctr) : 0u;
        if (lane < ntok) {
            mbar_arrive_expect_tx(&row_bar[lane], in_bytes);
            bulk_load(smem + (size_t)lane * pl.stage_bytes, xs + (size_t)lane * p.H * 2, in_bytes, &row_bar[lane]);
        }
        if (lane == 0) epoch_sm = epoch_from_counter(ctr);
    } else {
        bad = stage_table<K>(p, ids, tid - 32, kThreads - 32);
    }
    // this warp's slot, if it has one: slot j of own token tl
    const int tl = warp / K, j = warp % K, t = t0 + tl;
    const bool slot = tl < ntok;
    const float w_i = slot && lane < K ? ld_plain(p.topk_w + (size_t)t * K + lane) : 0.0f;   // the token's gate weights, a lane each
    __syncthreads();
    mark(kTrCounted);
    unsigned ticket = 0u;
    if (tid == 0) ticket = atomicAdd(p.done_ticket, 1u);   // (every CTA has read the epoch when the last ticket is taken)
    const unsigned half = epoch_sm & 1u;

    // ---- the slot's row, its copy if the row has landed, its metadata
    bool send = false, sent = false;
    int r = 0, gpos = -1;
    auto copy = [&]() {   // bf16
        if (lane == 0) bulk_store(p.recv_x + (size_t)gpos * p.rowB + out_off, smem + (size_t)tl * pl.stage_bytes, out_bytes);
        bulk_commit();
        sent = true;
    };
    if (slot) {
        const SlotRow s = slot_row<K>(p, ids, t, j, kDedup, lane);
        bad = bad || s.twice;
        r = s.r;
        gpos = s.valid && s.row < p.cap ? r * p.cap + s.row : -1;
        send = s.first && gpos >= 0;
        if (!kFp8 && send && __all_sync(kAll, mbar_test_wait(&row_bar[tl], 0))) copy();   // (the metadata while it is on its way)
        if (part == 0) slot_meta<K>(p, s, t, j, gpos, w_i, kDedup, lane);
        else if (s.valid && gpos < 0) report(p.status, kErrCapacity);
    }
    if (bad) report(p.status, kErrBadIndex);
    mark(kTrFinalized);
    mark(kTrReady);   // (nobody waits to be released)
    if (kTraced && ntok > 0) {
        (void)mbar_wait(&row_bar[0], 0, nullptr);
        mark(kTrFirstRow);
    }

    // ---- the copy
    if (kFp8) {
        // every warp quantises: eight channels per lane
        const int nvec = (int)in_bytes / 16;
        const int gp = p.G / p.parts;   // scale groups of this CTA's piece
        const int strips = (nvec + 31) / 32;   // of a row, a warp's vectors at a time
        bool got = true;
#pragma unroll 1
        for (int u = warp; u < ntok * strips; u += 2 * kWarps) {   // two strips side by side
            uint4 d[2];
            int i[2], v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int uh = u + h * kWarps;
                i[h] = uh / strips;
                v[h] = (uh - i[h] * strips) * 32 + lane;
                if (uh >= ntok * strips) v[h] = nvec;   // nothing
                d[h] = make_uint4(0, 0, 0, 0);
                if (v[h] < nvec) {
                    got = mbar_wait(&row_bar[i[h]], 0, nullptr) && got;
                    d[h] = *reinterpret_cast<const uint4*>(smem + (size_t)i[h] * pl.stage_bytes + (size_t)v[h] * 16);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && u + kWarps >= ntok * strips) break;   // (the whole warp)
                uint8_t* out = smem + pl.off_out + (size_t)i[h] * pl.out_stage_bytes;
                uint2 q;
                float sc;
                quantize8(d[h], v[h] < nvec, q, sc);
                if (v[h] < nvec) {
                    *reinterpret_cast<uint2*>(out + (size_t)v[h] * 8) = q;
                    if ((lane & 15) == 0) reinterpret_cast<float*>(out + out_bytes)[v[h] >> 4] = sc;
                }
            }
        }
        if (!got) report(p.status, kErrTimeout);
        fence_proxy_async_smem();   // the bulk stores read what has just been written
        if (__syncthreads_or(!got)) send = false;
        if (send) {
            const uint8_t* src = smem + pl.off_out + (size_t)tl * pl.out_stage_bytes;
            float* scales = p.recv_scale + (size_t)gpos * p.G + part * gp;
            if ((gp & 3) == 0) {
                if (lane == 1) bulk_store(scales, src + out_bytes, (unsigned)gp * 4u);
            } else {   // (a piece of scales that no bulk copy can carry)
                for (int i = lane; i < gp; i += 32) scales[i] = reinterpret_cast<const float*>(src + out_bytes)[i];
            }
            if (lane == 0) bulk_store(p.recv_x + (size_t)gpos * p.rowB + out_off, src, out_bytes);
            bulk_commit();
        }
    } else if (send && !sent) {
        send = __all_sync(kAll, mbar_wait(&row_bar[tl], 0, nullptr));
        if (send) copy();
        else report(p.status, kErrTimeout);
    }
    mark(kTrIssued);

    // ---- what no row waits for; the warps without a slot, the last ones of every CTA, come first
#pragma unroll 1
    for (int u = (kWarps - 1 - warp) * p.grid + c; u < p.R * pl.duty_units; u += kWarps * p.grid)
        write_table_unit<K>(p, ids, u, pl.duty_units, kDedup, lane);
    mark(kTrScanned);

    // ---- the arrival counters (eighths of a row: see publish_arrivals): every warp for its own row
    if (send) {
        bulk_wait_all<0>();
        __syncwarp();
        if (lane == 0) red_release_add(p.arrival + half * p.R + r, (unsigned)(8 / p.parts));
    }
    mark(kTrStored);
    if (c == p.grid - 1 && warp == kWarps - 1) {   // those of the next call live in the other half
        for (int i = lane; i < p.R; i += 32) p.arrival[(half ^ 1u) * p.R + i] = 0;
        if (lane == 0) p.claimed[half ^ 1u] = 0;
    }
    if (warp == 0) {
        if (lane == 0) epoch_finish_check_in(p, ticket, epoch_sm);
        if (lane < ntok) (void)mbar_wait(&row_bar[lane], 0, nullptr);   // (a row that no slot sends may still be landing)
    }
    mark(kTrEnd);
}

template <int K, bool kFp8, bool kDedup, bool kTraced>
cudaError_t launch_few_s(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    auto kern = few_kernel<K, kFp8, kDedup, kTraced>;
    const int smem = with_room_beside(pl.total, 0);
    static std::atomic<int> granted[kAttrDevices];
    cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void*>(kern), smem, granted);
    if (e != cudaSuccess) return e;
    return launch_overlapped(kern, p.grid, kThreads, (size_t)smem, st, false, 1, p, pl);
}
template <int K, bool kFp8, bool kDedup>
cudaError_t launch_few_t(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    return p.trace != nullptr ? launch_few_s<K, kFp8, kDedup, true>(p, pl, st) : launch_few_s<K, kFp8, kDedup, false>(p, pl, st);
}
template <int K>
cudaError_t launch_few_k(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    if (p.payload) return p.dedup ? launch_few_t<K, true, true>(p, pl, st) : launch_few_t<K, true, false>(p, pl, st);
    return p.dedup ? launch_few_t<K, false, true>(p, pl, st) : launch_few_t<K, false, false>(p, pl, st);
}

}  // namespace

bool plan_few(const Params& p, int max_smem, SmemPlan* out) {
    const int most = (p.T + p.nchunks - 1) / p.nchunks;   // tokens of a CTA
    if (most * p.k > kWarps || (int64_t)most * p.k * p.T * (p.k + 8) > kFewWork || p.L > 32 || p.ordered) return false;
    if (p.k != 1 && p.k != 2 && p.k != 4 && p.k != 6 && p.k != 8) return false;
    if (p.payload && p.quant_warps < kWarps - 2) return false;   // (fewer quantising warps were asked for)
    if (p.payload && p.prefetch_rows < most) return false;       // (rows to be fetched behind the layout; here all are at once)
    SmemPlan pl{};
    auto round_up = [](int64_t v, int m) { return (v + m - 1) / m * m; };
    const int64_t stage = round_up((int64_t)p.H * 2 / p.parts, 128);
    const int64_t out_stage = p.payload ? round_up((int64_t)p.rowB / p.parts + (p.G / p.parts) * 4, 128) : 0;
    const int64_t total = most * (stage + out_stage) + round_up((int64_t)p.T * p.k * 2, 128);
    if (total + 1536 > max_smem) return false;   // (1.5 KB: static shared memory)
    pl.stages = most;
    pl.stage_bytes = (int)stage;
    pl.trip_rows = 1;
    pl.out_stages = p.payload ? most : 0;
    pl.out_stage_bytes = (int)out_stage;
    pl.q_warps = p.payload ? kWarps : 0;   // one team of all of them
    pl.q_teams = p.payload ? 1 : 0;
    pl.q_team_warps = pl.q_warps;
    pl.off_out = (int)(most * stage);
    pl.off_ids = pl.off_out + (int)(most * out_stage);
    // One CTA per SM.  Two of them fit in an SM's registers, and where a call may be placed while the combine before it runs
    // (programmatic launches), SMs without combine CTAs took two and others none: sixteen layers of 128 tokens of 7168 channels,
    // top-8, in one graph 12.6 us per layer, this way 10.4 (both at the time; 9.5 now).  (Warps that leave at once do not hold their registers: no change.)
    pl.total = (int)(total < kFewSmem ? kFewSmem : total);
    pl.duty_units = table_units(p);
    *out = pl;
    return true;
}

cudaError_t launch_few(const Params& p, const SmemPlan& pl, cudaStream_t st) {
    switch (p.k) {
        case 1: return launch_few_k<1>(p, pl, st);
        case 2: return launch_few_k<2>(p, pl, st);
        case 4: return launch_few_k<4>(p, pl, st);
        case 6: return launch_few_k<6>(p, pl, st);
        default: return launch_few_k<8>(p, pl, st);
    }
}

}  // namespace ubep
