// Dispatch with a selectable readiness protocol (Sec. 3.4 of the paper, "Data-as-Flag
// Synchronization"): stop-and-wait counters, Token-Flag Fusion, Data-for-Checksum and
// Sentinel Polling.  One persistent kernel; every CTA is first a sender (the rows of its
// token chunk) and then a receiver (a slice of one receive region), so the waits of the
// receivers are satisfied by CTAs that never wait themselves.  All CTAs must be resident
// (grid <= number of SMs, one CTA per SM).
//
// The layout (TokenCnt, CalCumSum, slot -> row) is derived by every CTA alone from the
// whole routing table, by the counting functions of the layout by clusters (a cluster of one), so the two
// paths leave identical metadata in the arena.  (From bitmaps of every bin over the whole table it took 7.4 us at
// 128 tokens and 21.7 us at 900; this way 4.1 - 5.1 and 5.7 us.)
//
// A DataBlock is the 16 bytes one thread stores with a single 128-bit access.
#include "ubep_cluster.cuh"
#include "ubep_few.cuh"
#include "ubep_quant.cuh"
#include "ubep_sync.h"

namespace ubep {

namespace {

constexpr int kSW = 0, kTFF = 1, kDC = 2, kSP = 3;
constexpr int kDcBlockVecs = 32;    // 512-byte checksum block = 32 vectors of 16 bytes
constexpr int kDcMarkerVecs = 2;    // its leading 32 bytes are the marker
constexpr int kStrip = 256;         // DataBlocks a warp of a receiver looks at together: eight loads in flight per lane
constexpr int kStripWords = kStrip * 3;   // payload words of a Token-Flag strip

__device__ __forceinline__ uint4 ld_relaxed_v4(const void* ptr) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_v4(void* ptr, const uint4 v) {
    asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(ptr), "r"(v.x), "r"(v.y), "r"(v.z),
                 "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* ptr) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ bool is_sentinel(const uint4 v) { return (v.x & v.y & v.z & v.w) == 0xffffffffu; }
__device__ __forceinline__ unsigned long long marker_words(const uint4 v) {
    return ((unsigned long long)v.x | ((unsigned long long)v.y << 32)) +
           ((unsigned long long)v.z | ((unsigned long long)v.w << 32));
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sequence number of the running call, kept on the device like the dispatch epoch: every
// CTA reads the counter and takes a ticket, the last ticket advances the counter.
__device__ __forceinline__ unsigned read_seq_and_check_in(const SyncParams& sp, int grid) {
    unsigned s = ld_acquire(sp.seq_ctr) + 1u;
    if (s == 0u) s = 1u;   // 0 is what a never-written flag holds
    if (atomicAdd(sp.seq_ticket, 1u) == (unsigned)grid - 1u) {
        *sp.seq_ticket = 0u;
        *sp.seq_ctr = s;
    }
    return s;
}

// Bounded polling: give up after kWaitLimitNs or when another thread of the CTA has.
struct Waiter {
    volatile int* abort;
    unsigned long long t_end;
    int32_t* status;
    unsigned* dirty;   // Sentinel Polling: word that tells the next call that this one gave up (else null)
    __device__ __forceinline__ bool keep_waiting(unsigned& spins) {
        __nanosleep(32);
        if ((++spins & 127u) != 0) return true;
        if (*abort) return false;
        if (global_ns() > t_end) {
            *abort = 1;
            report(status, kErrTimeout);
            if (dirty) *dirty = 1u;
            return false;
        }
        return true;
    }
};

__device__ __forceinline__ bool wait_count(const unsigned* ctr, unsigned want, Waiter& wt) {
    unsigned spins = 0;
    while (ld_acquire(ctr) != want)
        if (!wt.keep_waiting(spins)) return false;
    return true;
}

// Behind the plan: checksums [R] of 8 bytes or, with the protocols that have none, the regions' first rows [R + 1] (one or the
// other: with both there was no room for tables that had been taken, of 5200 ranks for instance); the quantised row.
__host__ __device__ inline int sync_qrow(const Params& p) { return (p.R * 8 + 15) / 16 * 16; }
__host__ __device__ inline int qrow_bytes(const Params& p) { return p.payload ? ((p.H + 4 * p.G + 15) / 16) * 16 : 0; }
__host__ __device__ inline bool strips_in_ring(const Params& p) {   // (a plan has four rows at least, two for FP8 rows)
    return (p.payload ? 2 : 4) * 2 * p.H >= kWarps * kStripWords * 4;
}

// kFp8: rows travel quantised (e4m3 payload, then the fp32 scales of the row's 128-channel groups, as one
// wire row of H + 4 * H / 128 bytes); the sender quantises a row once into shared memory and sends from
// there; what arrives goes to the payload and the scale array of the receive region.  The checksum
// markers of Data-for-Checksum are taken from the payload bytes.
// kLayout: kLaunched, from count_kernel / scan_kernel, launched before over the same chunks: the CTA stages only its own tokens
// and reads the rows of earlier chunks, the expert offsets and the region sizes.  kWhole: every CTA counts the whole routing table.
// K > 0, small tables of K slots per token: a warp per slot (ubep_few.cuh); the CTAs of a chunk share its rows, a range of their
// blocks each.
constexpr int kLaunched = 0, kWhole = -1;
template <int kProto, bool kFp8, int kLayout>
__global__ void __launch_bounds__(kThreads, 1) sync_dispatch_kernel(const Params p, const SmemPlan pl,
                                                                   const SyncParams sp) {
    constexpr bool kTable = kLayout == kWhole, kFew = kLayout > 0;
    constexpr int K = kFew ? kLayout : 1;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ unsigned seq_sm;
    __shared__ int abort_flag;
    __shared__ unsigned long long wsum[2][kWarps];   // DC: per-warp marker sums (two tokens in flight)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = blockIdx.x;
    const int k = p.k, R = p.R;
    unsigned long long* times = sp.times + (size_t)c * kSyncTimeSlots;
    if (tid == 0) times[0] = global_ns();

    int* ids_sm = reinterpret_cast<int*>(smem + pl.off_ids);
    int* pos = reinterpret_cast<int*>(smem + pl.off_pos);
    int* key = reinterpret_cast<int*>(smem + pl.off_key);
    float* w_sm = reinterpret_cast<float*>(smem + pl.off_w);
    int* hist = reinterpret_cast<int*>(smem + pl.off_hist);
    int* nrows = reinterpret_cast<int*>(smem + pl.off_arr);     // rows every region receives
    int* first = reinterpret_cast<int*>(smem + pl.total);   // Token-Flag and Sentinel receivers: [R + 1]
    int* order_sm = reinterpret_cast<int*>(smem + pl.off_order);
    unsigned long long* chk_sm = reinterpret_cast<unsigned long long*>(smem + pl.total);   // DC: [R]
    uint8_t* qrow = smem + pl.total + sync_qrow(p);                                         // FP8: the quantised row
    // TFF: [kWarps, kStripWords]; in the ring of rows, which the receiver no longer needs, where that is large enough
    uint32_t* strips = reinterpret_cast<uint32_t*>(kFew || strips_in_ring(p) ? smem : qrow + qrow_bytes(p));
    __shared__ __align__(8) uint64_t row_bar[2];   // the row of an even / odd token has landed in ring stage 0 / 1
    const BinMaps bmaps{reinterpret_cast<unsigned*>(smem + pl.off_mask), reinterpret_cast<unsigned*>(smem + pl.off_bm),
                        pl.map_wb, pl.map_bp, pl.map_groups};
    const int parts = kFew ? p.parts : 1, part = kFew ? c % parts : 0, ch = kFew ? c / parts : c;
    const int t0 = (int)chunk_begin(ch, p.T, p.nchunks), t1 = (int)chunk_begin(ch + 1, p.T, p.nchunks);
    const int ntok = t1 - t0;
    uint16_t* ids16 = reinterpret_cast<uint16_t*>(smem + pl.off_ids);   // (kFew)
    auto fetch_row = [&](int tl) {   // one thread; the row before the last one has been sent
        mbar_arrive_expect_tx(&row_bar[tl & 1], (unsigned)p.H * 2u);
        bulk_load(smem + (size_t)(tl & 1) * pl.stage_bytes, p.x + (size_t)(t0 + tl) * p.H, (unsigned)p.H * 2u, &row_bar[tl & 1]);
    };
    constexpr int kFetcher = kFew ? 0 : 32;   // (kFew: warp 0 has no part in staging the table)
    if (tid == kFetcher) {
        mbar_init(&row_bar[0], 1);
        mbar_init(&row_bar[1], 1);
        mbar_fence_init();
        if (ntok > 0) fetch_row(0);   // on its way while the layout is computed
        if (ntok > 1) fetch_row(1);
    }

    if (kFew) {
        for (int r = tid; r < R; r += kThreads) nrows[r] = 0;
        __syncthreads();
    }
    if (tid == 0) {
        seq_sm = read_seq_and_check_in(sp, p.grid);
        abort_flag = 0;
        // Sentinel Polling after a call that gave up: blocks of that call may still sit in the wire and
        // would be taken for this call's.  Nothing is sent or received then; the call reports the
        // condition again, and the library re-fills the wire once it has learnt of it (ubep_status).
        if (kProto == kSP && ld_relaxed(sp.sp_dirty) != 0u) {
            abort_flag = 1;
            report(p.status, kErrTimeout);
        }
    }
    if (kProto == kDC)
        for (int r = tid; r < R; r += kThreads) chk_sm[r] = 0ull;

    // ---- layout: counts of every bin over the whole routing table -> totals, the rows before this CTA's tokens,
    // expert offsets, rows of this CTA's slots
    int* tot = hist;
    int* base = hist + p.B;   // rows before the CTA's tokens in the bin's segment
    int* eo = hist + 2 * p.B;
    unsigned* cnt = reinterpret_cast<unsigned*>(smem + pl.off_cnt);   // (kTable)
    unsigned* own = cnt + p.B + 1;
    bool twice = false;
    if (kFew) {
        bool bad = warp != 0 && stage_tokens<K>(p, ids16, nrows, p.dedup != 0, tid - 32, kThreads - 32);
        __syncthreads();
        for (int sl = warp; sl < ntok * K; sl += kWarps) {
            const int t = t0 + sl / K, j = sl % K;
            const float w_i = part == 0 && lane < K ? __ldg(p.topk_w + (size_t)t * K + lane) : 0.0f;
            const SlotRow s = slot_row<K>(p, ids16, t, j, p.dedup != 0, lane);
            bad = bad || s.twice;
            const int gpos = s.valid && s.row < p.cap ? s.r * p.cap + s.row : -1;
            if (lane == 0) pos[sl] = s.first ? gpos : -1;
            if (part == 0) slot_meta<K>(p, s, t, j, gpos, w_i, p.dedup != 0, lane);
        }
        if (bad) report(p.status, kErrBadIndex);
    } else if (kTable) {
        for (int b = tid; b < 3 * (p.B + 1); b += kThreads) cnt[b] = 0u;
        for (int b = tid; b < pl.map_groups * pl.map_bp; b += kThreads) bmaps.bm[b] = 0u;
        __syncthreads();
        twice = stage_own(p, t0, t1, ids_sm, bmaps.bm, bmaps.bp, own, kThreads - 1 - tid, kThreads);
        count_tokens(count_args(p), 0, p.T, t0, true, cnt, tid, kThreads, t1, t1 > t0 ? own_sources_end(p, t1) : t1, cnt + 2 * (p.B + 1));
    } else {
        stage_ids(p, t0, t1, ids_sm, tid, kThreads);
    }
    if (!kFew) {
        for (int r = tid; r < R; r += kThreads) order_sm[r] = __ldg(p.order_pos + r);
        for (int i = tid; i < ntok * k; i += kThreads) w_sm[i] = __ldg(p.topk_w + (size_t)t0 * k + i);
    }
    if (__syncthreads_or(twice)) {
        local_clean_own_duplicates(p, 0, ntok, ids_sm, tid, kThreads);
        __syncthreads();
    }
    const unsigned seq = seq_sm;
    const int par = (int)(seq & 1u);
    if (kTable) {
        for (int b = tid; b < p.B; b += kThreads) {
            tot[b] = (int)(cnt[b] >> 16);
            base[b] = (int)(cnt[b] & 0xffffu);
        }
        __syncthreads();
        for (int e = tid; e < p.E; e += kThreads) {
            int o = 0;
            for (int q = (e / p.L) * p.L; q < e; ++q) o += tot[q];
            eo[e] = o;
            base[e] += o;
        }
        __syncthreads();
        for (int r = tid; r < R; r += kThreads) {
            const int e1 = (r + 1) * p.L - 1;
            nrows[r] = p.dedup ? tot[p.E + r] : eo[e1] + tot[e1];
        }
        finalize_chunk(p, t0, t1, ids_sm, w_sm,
                       [&](int e, int tl) { return base[e] + own_below(bmaps, e, tl); },
                       [&](int r, int tl) { return base[p.E + r] + own_below(bmaps, p.E + r, tl); },
                       true, c, order_sm, pos, key, nullptr, tid, kThreads);
        __syncthreads();
    } else if (!kFew) {
        build_bin_maps(p, ids_sm, ntok, bmaps, warp, kWarps, lane);
        int* base_sm = hist;   // per bin: rows of all earlier chunks (+ the expert's offset in its region)
        for (int b = tid; b < p.B; b += kThreads)
            base_sm[b] = __ldcg(p.chunk_base + (size_t)b * p.nchunks + c) + (b < p.E ? __ldcg(p.expert_offset + b) : 0);
        for (int r = tid; r < R; r += kThreads) nrows[r] = __ldcg(p.num_rows_per_rank + r);
        __syncthreads();
        finalize_chunk(p, t0, t1, ids_sm, w_sm,
                       [&](int e, int tl) { return base_sm[e] + bits_in_range(bmaps, e, 0, tl); },
                       [&](int r, int tl) { return base_sm[p.E + r] + bits_in_range(bmaps, p.E + r, 0, tl); },
                       true, c, order_sm, pos, key, nullptr, tid, kThreads);
        __syncthreads();
    }
    if (tid == 0) times[1] = global_ns();
    // ---- sender: the rows of tokens [t0, t1), one token at a time, all threads on a row
    const int wbytes = kFp8 ? p.H + 4 * p.G : p.rowB;   // bytes of one row on the wire
    const int nvec = (wbytes + 15) / 16;                // its 16-byte blocks (FP8: the last may be cut short)
    const int pvec = p.rowB / 16;                       // blocks of the payload (all of them for bf16 rows)
    const int nwords = wbytes / 4;
    const int pwords = p.rowB / 4;
    const size_t wire_row = (size_t)sp.tff_blocks * 16;
    const size_t sp_row = (size_t)nvec * 16;
    const bool wire_unusable = kProto == kSP && abort_flag != 0;   // (set before the barriers above, uniform in the CTA)
    // word w of the wire row of global row `where` lands in the payload or, beyond it, in the scales
    auto put_word = [&](size_t where, int w, uint32_t val) {
        if (!kFp8 || w < pwords) reinterpret_cast<uint32_t*>(p.recv_x + where * p.rowB)[w] = val;
        else reinterpret_cast<uint32_t*>(p.recv_scale + where * p.G)[w - pwords] = val;
    };
    bool lost = false;   // a row did not come: what is sent is not it, and the call reports the timeout
    if (wire_unusable)
        for (int tl = 0; tl < min(2, ntok); ++tl) (void)mbar_wait(&row_bar[tl], 0, nullptr);
    for (int tl = 0; tl < ntok && !wire_unusable; ++tl) {
        const int* ps = pos + tl * k;
        const uint4* xrow = reinterpret_cast<const uint4*>(smem + (size_t)(tl & 1) * pl.stage_bytes);
        lost = !mbar_wait(&row_bar[tl & 1], (tl >> 1) & 1, nullptr) || lost;
        if (kFp8) {
            // quantise the row once (every copy carries the same bytes)
            const int xvec = p.H / 8;
            for (int v0 = 0; v0 < xvec; v0 += kThreads) {   // same trip count for every thread (the quantiser shuffles)
                const int v = v0 + tid;
                const bool in = v < xvec;
                const uint4 d = in ? xrow[v] : make_uint4(0, 0, 0, 0);
                uint2 q;
                float scale;
                quantize8(d, in, q, scale);
                if (in) {
                    *reinterpret_cast<uint2*>(qrow + (size_t)v * 8) = q;
                    if ((v & 15) == 0) reinterpret_cast<float*>(qrow + p.H)[v >> 4] = scale;
                }
            }
            for (int w = nwords + tid; w < nvec * 4; w += kThreads) reinterpret_cast<uint32_t*>(qrow)[w] = 0u;   // padding
            __syncthreads();
        }
        if (kProto == kTFF) {
            const uint32_t* xw = kFp8 ? reinterpret_cast<const uint32_t*>(qrow) : reinterpret_cast<const uint32_t*>(xrow);
            for (int g = sp.tff_blocks * part / parts + tid; g < sp.tff_blocks * (part + 1) / parts; g += kThreads) {
                const int w0 = 3 * g;
                uint4 blk;
                blk.x = seq;   // the flag leads the block
                blk.y = w0 < nwords ? xw[w0] : 0u;
                blk.z = w0 + 1 < nwords ? xw[w0 + 1] : 0u;
                blk.w = w0 + 2 < nwords ? xw[w0 + 2] : 0u;
                for (int j = 0; j < k; ++j) {
                    const int where = ps[j];
                    if (where >= 0) st_relaxed_v4(sp.tff_wire + (size_t)where * wire_row + (size_t)g * 16, blk);
                }
            }
        } else {
            unsigned long long mine = 0ull;
            for (int v = nvec * part / parts + tid; v < nvec * (part + 1) / parts; v += kThreads) {
                const uint4 d = kFp8 ? reinterpret_cast<const uint4*>(qrow)[v] : xrow[v];
                if (kProto == kDC && v < pvec && (v % kDcBlockVecs) < kDcMarkerVecs) mine += marker_words(d);
                for (int j = 0; j < k; ++j) {
                    const int where = ps[j];
                    if (where < 0) continue;
                    if (kProto == kSP) {
                        st_relaxed_v4(sp.sp_wire + (size_t)where * sp_row + (size_t)v * 16, d);
                    } else if (!kFp8 || v < pvec) {
                        *reinterpret_cast<uint4*>(p.recv_x + (size_t)where * p.rowB + (size_t)v * 16) = d;
                    } else {
                        const uint32_t dw[4] = {d.x, d.y, d.z, d.w};
                        for (int i = 0; i < 4; ++i)
                            if (4 * v + i < nwords) put_word((size_t)where, 4 * v + i, dw[i]);
                    }
                }
            }
            if (kProto == kDC) {
                // marker sum of this row, added to the running sum of every region it goes to
                // (the slot of the token after next is written only after the next barrier)
                mine = warp_sum64(mine);
                if (lane == 0) wsum[tl & 1][warp] = mine;
                __syncthreads();
                if (tid < k && ps[tid] >= 0) {
                    unsigned long long row_sum = 0ull;
                    for (int q = 0; q < kWarps; ++q) row_sum += wsum[tl & 1][q];
                    atomicAdd(&chk_sm[ps[tid] / p.cap], row_sum);
                }
            }
            if (kProto == kSW) {
                // stop-and-wait: the row's stores are fenced before its flag is raised
                __threadfence();
                __syncthreads();
                if (tid < k && ps[tid] >= 0) red_release_add(sp.sw_rows + par * R + ps[tid] / p.cap, 1u);
            }
        }
        if (kFp8 || tl + 2 < ntok) __syncthreads();   // the quantised row and the row's buffer are used again
        if (tid == kFetcher && tl + 2 < ntok) fetch_row(tl + 2);
    }
    if (lost) report(p.status, kErrTimeout);
    if (kProto == kDC) {
        // one fence per sender and batch, then the checksum packet of every region
        __threadfence();
        __syncthreads();
        for (int r = tid; r < R; r += kThreads) {
            if (chk_sm[r]) atomicAdd(sp.checksum + par * R + r, chk_sm[r]);
            red_release_add(sp.announced + par * R + r, 1u);
        }
    }
    if (tid == 0) times[2] = global_ns();
    constexpr bool kByBlock = kProto == kTFF || kProto == kSP;   // receivers look at every block
    if (kByBlock && warp == 0) {   // first[r]: rows of the regions before r
        int run = 0;
        for (int r0 = 0; r0 < R; r0 += 32) {
            const int r = r0 + lane, n = r < R ? min(nrows[r], p.cap) : 0, incl = warp_incl_scan(n, lane);
            if (r < R) first[r + 1] = run + incl;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) first[0] = 0;
    }
    if (kByBlock) __syncthreads();   // (the strips may lie where the rows were)
    if (kFew && warp >= kWarps / 2) {   // (see below)
        for (int u = (warp - kWarps / 2) * p.grid + c; u < p.R * pl.duty_units; u += kWarps / 2 * p.grid)
            write_table_unit<K>(p, ids16, u, pl.duty_units, p.dedup != 0, lane);
    }
    if (kTable && warp >= kWarps / 2) {
        // counts and offsets nobody inside this kernel waits for (the launches before wrote them otherwise); behind the
        // rows, which the receivers wait for, and by half of the warps: the others turn to receiving at once
        constexpr int n = kThreads / 2;
        if (c == 0) write_totals(p, tot, eo, tid - n, n);
        write_own_sources<true>(p, t0, t1, 0, 1, bmaps, base, cnt + 2 * (p.B + 1), tid - n, n, 0);
    }

    // ---- receiver
    Waiter wt{&abort_flag, global_ns() + kWaitLimitNs, p.status, kProto == kSP ? sp.sp_dirty : nullptr};
    const int Q = p.grid / R > 1 ? p.grid / R : 1;
    bool duty = false;
    if (kProto == kTFF || kProto == kSP) {
        // Every CTA takes an equal share of all rows of all regions, a warp kStrip DataBlocks of a row at a time: its
        // lanes look at neighbouring blocks, with all loads of the strip in flight before any of them is looked at.  What a Token-Flag strip carries passes through shared
        // memory, so that it leaves in 16-byte stores.  (Four blocks per thread in flight and three 4-byte stores
        // per block: 12.5 us from the last row sent to the last one confirmed at 128 tokens, now 8.7.)
        constexpr int kBatch = kStrip / 32;
        const int per_row = kProto == kTFF ? sp.tff_blocks : nvec;
        const int strips_per_row = (per_row + kStrip - 1) / kStrip;
        const size_t row_stride = kProto == kTFF ? wire_row : sp_row;
        const uint4 sentinel = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
        uint32_t* const mine = strips + (kProto == kTFF ? warp * kStripWords : 0);
        const int from = (int)((long long)first[R] * c / p.grid), to = (int)((long long)first[R] * (c + 1) / p.grid);
        duty = to > from;   // this CTA's share
        bool ok = true;
        const int count = (to - from) * strips_per_row;
        uint8_t* const wires = kProto == kTFF ? sp.tff_wire : sp.sp_wire;
        struct Strip {
            size_t grow;    // row of the receive regions
            int g0, n;      // its blocks g0 .. g0 + n - 1
        };
        auto strip_at = [&](int i) -> Strip {
            const int row = from + i / strips_per_row, g0 = (i % strips_per_row) * kStrip;
            int r = -1;   // its region
            for (int r0 = 0; r0 <= R; r0 += 32) r += __popc(__ballot_sync(0xffffffffu, r0 + lane <= R && first[r0 + lane] <= row));
            return {(size_t)r * p.cap + (row - first[r]), g0, min(kStrip, per_row - g0)};
        };
        for (int i = warp; ok && i < count; i += kWarps) {
            const Strip at = strip_at(i);
            const size_t grow = at.grow;
            const int g0 = at.g0, n = at.n;
            uint8_t* const wire = wires + grow * row_stride + (size_t)g0 * 16;
            uint4 blk[kBatch];
            unsigned missing = 0u;   // bit b: this lane's b-th block has not arrived
#pragma unroll
            for (int b = 0; b < kBatch; ++b) missing |= b * 32 + lane < n ? 1u << b : 0u;
            unsigned spins = 0;
            for (;;) {   // (all missing blocks side by side: one after the other a late strip cost eight round trips)
#pragma unroll
                for (int b = 0; b < kBatch; ++b)
                    if (missing >> b & 1u) blk[b] = ld_relaxed_v4(wire + (size_t)(b * 32 + lane) * 16);
#pragma unroll
                for (int b = 0; b < kBatch; ++b)
                    if ((missing >> b & 1u) && !(kProto == kTFF ? blk[b].x != seq : is_sentinel(blk[b]))) missing &= ~(1u << b);
                if (missing == 0u) break;
                if (!wt.keep_waiting(spins)) { ok = false; break; }
            }
            ok = __all_sync(0xffffffffu, ok);
            // Payload alone, as every strip of bf16 rows: few conditions, and what leaves leaves side by side.  (Token-Flag, 128 tokens of
            // 7168 channels, from the last row sent to the last one confirmed 7.5 us with a condition per word, now 5.7.)
            if (ok && (kProto != kTFF || sp.tff_strips) && (!kFp8 || (kProto == kTFF ? 3 * (g0 + n) <= pwords : g0 + n <= pvec))) {
                uint4* const to16 = reinterpret_cast<uint4*>(p.recv_x + grow * p.rowB) + (kProto == kTFF ? g0 / 4 * 3 : g0);
                if (kProto == kTFF) {
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) {
                        if (b * 32 + lane >= n) continue;
                        mine[3 * (b * 32 + lane)] = blk[b].y;
                        mine[3 * (b * 32 + lane) + 1] = blk[b].z;
                        mine[3 * (b * 32 + lane) + 2] = blk[b].w;
                    }
                    __syncwarp();
                    const int n16 = min(3 * n, pwords - 3 * g0) / 4;   // (the words behind the row's last block are not written)
#pragma unroll
                    for (int q = 0; q < kBatch * 3 / 4; ++q)
                        if (q * 32 + lane < n16) blk[q] = reinterpret_cast<const uint4*>(mine)[q * 32 + lane];
#pragma unroll
                    for (int q = 0; q < kBatch * 3 / 4; ++q)
                        if (q * 32 + lane < n16) to16[q * 32 + lane] = blk[q];
                    __syncwarp();   // the strip's buffer is used again
                } else {
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) {
                        if (b * 32 + lane >= n) continue;
                        to16[b * 32 + lane] = blk[b];
                        st_relaxed_v4(wire + (size_t)(b * 32 + lane) * 16, sentinel);   // consumed: ready for the next call
                    }
                }
                continue;
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int g = b * 32 + lane;
                if (g >= n || (missing >> b & 1u)) continue;
                if (kProto == kTFF && !sp.tff_strips) {
                    const uint32_t dw[3] = {blk[b].y, blk[b].z, blk[b].w};
                    for (int q = 0; q < 3; ++q)
                        if (3 * (g0 + g) + q < nwords) put_word(grow, 3 * (g0 + g) + q, dw[q]);
                } else if (kProto == kTFF) {
                    mine[3 * g] = blk[b].y;
                    mine[3 * g + 1] = blk[b].z;
                    mine[3 * g + 2] = blk[b].w;
                } else {
                    const int v = g0 + g;
                    if (!kFp8 || v < pvec) {
                        *reinterpret_cast<uint4*>(p.recv_x + grow * p.rowB + (size_t)v * 16) = blk[b];
                    } else {
                        const uint32_t dw[4] = {blk[b].x, blk[b].y, blk[b].z, blk[b].w};
                        for (int q = 0; q < 4; ++q)
                            if (4 * v + q < nwords) put_word(grow, 4 * v + q, dw[q]);
                    }
                    st_relaxed_v4(wire + (size_t)g * 16, sentinel);   // consumed: ready for the next call
                }
            }
            if (kProto == kTFF && sp.tff_strips) {
                __syncwarp();   // the lanes' words are in the strip (the vote orders no memory)
                // words [3 * g0, 3 * g0 + 3 * n) of the wire row (a strip begins on a multiple of four words)
                for (int q = lane; ok && q < kStripWords / 4; q += 32) {
                    const int w = 3 * g0 + 4 * q;
                    if (4 * q >= 3 * n || w >= nwords) break;
                    const uint4 d = *reinterpret_cast<const uint4*>(mine + 4 * q);
                    if (w + 4 <= pwords) {
                        *reinterpret_cast<uint4*>(p.recv_x + grow * p.rowB + (size_t)w * 4) = d;
                    } else {   // (scales; the words behind the row's last block are not written)
                        const uint32_t dw[4] = {d.x, d.y, d.z, d.w};
                        for (int z = 0; z < 4; ++z)
                            if (w + z < nwords) put_word(grow, w + z, dw[z]);
                    }
                }
                __syncwarp();   // the strip's buffer is used again
            }
        }
    }
    for (int u = c; u < R * Q; u += p.grid) {
        const int r = u / Q, q = u % Q;
        const int n_r = nrows[r] < p.cap ? nrows[r] : p.cap;
        if (kProto != kTFF && kProto != kSP && q == 0) {
            duty = true;
            if (kProto == kSW) {
                if (tid == 0) (void)wait_count(sp.sw_rows + par * R + r, (unsigned)n_r, wt);
            } else {
                if (tid == 0) (void)wait_count(sp.announced + par * R + r, (unsigned)p.grid, wt);
                __syncthreads();
                if (!abort_flag) {
                    const int nblk = (pvec + kDcBlockVecs - 1) / kDcBlockVecs;
                    const int per_row = nblk * kDcMarkerVecs;
                    unsigned long long mine = 0ull;
                    for (int i = tid; i < n_r * per_row; i += kThreads) {
                        const int row = i / per_row, rem = i - row * per_row;
                        const int v = (rem / kDcMarkerVecs) * kDcBlockVecs + rem % kDcMarkerVecs;
                        if (v < pvec)
                            mine += marker_words(__ldcg(
                                reinterpret_cast<const uint4*>(p.recv_x + ((size_t)r * p.cap + row) * p.rowB) + v));
                    }
                    mine = warp_sum64(mine);
                    if (lane == 0) wsum[0][warp] = mine;
                    __syncthreads();
                    if (tid == 0) {
                        unsigned long long found = 0ull;
                        for (int q = 0; q < kWarps; ++q) found += wsum[0][q];
                        if (found != ld_relaxed_u64(sp.checksum + par * R + r)) report(p.status, kErrChecksum);
                    }
                }
                __syncthreads();
            }
        }
    }
    __syncthreads();
    if (tid == 0) times[3] = (duty && !abort_flag) ? global_ns() : times[2];
    // the counters of the next call live in the other half: clear them now
    if (c == 0)
        for (int r = tid; r < R; r += kThreads) {
            sp.checksum[(par ^ 1) * R + r] = 0ull;
            sp.announced[(par ^ 1) * R + r] = 0u;
            sp.sw_rows[(par ^ 1) * R + r] = 0u;
        }
    if (tid == 0) times[4] = global_ns();
}

__global__ void __launch_bounds__(256) sentinel_scan_kernel(const uint4* __restrict__ x, long long n_vec,
                                                            unsigned long long* count) {
    unsigned long long mine = 0ull;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_vec;
         i += (long long)gridDim.x * blockDim.x)
        mine += is_sentinel(__ldg(x + i)) ? 1ull : 0ull;
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(count, mine);
}

template <int kProto, int kLayout>
cudaError_t launch_one(const Params& p, const SmemPlan& pl, const SyncParams& sp, cudaStream_t st) {
    auto kern = p.payload ? sync_dispatch_kernel<kProto, true, kLayout> : sync_dispatch_kernel<kProto, false, kLayout>;
    const int smem = pl.total + sync_extra_smem(p, kProto, kLayout <= 0 && sp.tff_strips != 0);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    // Receivers wait for senders that are other CTAs of this grid: a cooperative launch, which the
    // runtime refuses when the grid cannot be resident at once and starts only when it is.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.grid);
    cfg.blockDim = dim3((unsigned)kThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, pl, sp);
}

template <int kProto>
cudaError_t launch_layout(const Params& p, const SmemPlan& pl, const SyncParams& sp, int how, cudaStream_t st) {
    if (how == kSyncLaunched) return launch_one<kProto, kLaunched>(p, pl, sp, st);
    if (how == kSyncWhole) return launch_one<kProto, kWhole>(p, pl, sp, st);
    if (p.k == 2) return launch_one<kProto, 2>(p, pl, sp, st);
    if (p.k == 4) return launch_one<kProto, 4>(p, pl, sp, st);
    return launch_one<kProto, 8>(p, pl, sp, st);
}

}  // namespace

bool plan_sync_few(Params& p, int protocol, int max_smem, SmemPlan* out) {
    // (Two, four and eight slots: every further number would be eight more kernels.  The dispatch of small batches has instances for
    // one and six as well; here those take the whole table's count, which they always took: nobody's main path, not timed.)
    if ((p.k != 2 && p.k != 4 && p.k != 8) || p.L > 32) return false;
    // idle CTAs take a part of the rows (not with stop-and-wait, whose counters count rows)
    while (protocol != kSW && p.T <= p.nchunks / 2 && p.nchunks % 2 == 0 && p.parts < 4) {
        p.nchunks /= 2;
        p.parts *= 2;
    }
    const int most = (p.T + p.nchunks - 1) / p.nchunks;
    auto round_up = [](int64_t v, int m) { return (v + m - 1) / m * m; };
    SmemPlan pl{};
    const int64_t stage = round_up((int64_t)p.H * 2, 128), strips = protocol == kTFF ? kWarps * kStripWords * 4 : 0;
    const int64_t ring = 2 * stage > strips ? 2 * stage : strips;   // (the Token-Flag strips lie where the rows were)
    const int64_t at_pos = ring + round_up((int64_t)p.T * p.k * 2, 128), at_arr = at_pos + (int64_t)most * p.k * 4;
    const int64_t total = round_up(at_arr + (int64_t)p.R * 4, 128);
    if ((int64_t)most * p.k * p.T * (p.k + 8) > kFewWork || total + sync_extra_smem(p, protocol, false) + 1536 > max_smem) {
        p.nchunks *= p.parts;
        p.parts = 1;
        return false;
    }
    pl.stages = 2;
    pl.stage_bytes = (int)stage;
    pl.off_ids = (int)ring;
    pl.off_pos = (int)at_pos;
    pl.off_arr = (int)at_arr;
    pl.duty_units = table_units(p);
    pl.total = (int)total;
    *out = pl;
    return true;
}

int sync_extra_smem(const Params& p, int protocol, bool strips) {
    const bool room = protocol == kTFF && strips && !strips_in_ring(p);
    return p.R * 8 + 128 + qrow_bytes(p) + 16 + (room ? kWarps * kStripWords * 4 : 0);
}

cudaError_t launch_sync_dispatch(const Params& p, const SmemPlan& pl, const SyncParams& sp, int how, cudaStream_t st) {
    switch (sp.protocol) {
        case kSW: return launch_layout<kSW>(p, pl, sp, how, st);
        case kTFF: return launch_layout<kTFF>(p, pl, sp, how, st);
        case kDC: return launch_layout<kDC>(p, pl, sp, how, st);
        case kSP: return launch_layout<kSP>(p, pl, sp, how, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_sentinel_scan(const void* x, long long n_vec, unsigned long long* count, int num_sms,
                                 cudaStream_t st) {
    long long blocks = (n_vec + 255) / 256;
    if (blocks > (long long)num_sms * 8) blocks = (long long)num_sms * 8;
    if (blocks < 1) blocks = 1;
    sentinel_scan_kernel<<<(int)blocks, 256, 0, st>>>(static_cast<const uint4*>(x), n_vec, count);
    return cudaGetLastError();
}

}  // namespace ubep
