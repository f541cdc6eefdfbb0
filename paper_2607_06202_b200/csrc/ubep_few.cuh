// Layout of small batches: the routing table staged as 16-bit expert ids, a warp per slot that counts it for its own expert and
// rank alone, and the counts and offsets of the source ranks a warp per rank and handful of source ranks.  Used by the dispatch of
// small batches (ubep_few.cu) and by the readiness protocols (ubep_sync.cu).
#pragma once

#include "ubep_layout.cuh"

namespace ubep {

constexpr unsigned kAll = 0xffffffffu;

// 1 << n, and 0 from 32 on (also for the large values that negative numbers are).
__device__ __forceinline__ unsigned bit_or_none(unsigned n) {
    unsigned v;
    asm("shl.b32 %0, 1, %1;" : "=r"(v) : "r"(n));
    return v;
}
// The n lowest bits; all of them from 32 on, none up to 0.
__device__ __forceinline__ unsigned low_bits(int n) { return bit_or_none((unsigned)max(n, 0)) - 1u; }

// The staged table: 16-bit physical expert ids, kNone for a slot that is empty or bad.
constexpr unsigned kNone = 0xffffu;
__device__ __forceinline__ unsigned pack16(int a, int b) { return ((unsigned)a & 0xffffu) | (unsigned)b << 16; }

// The experts first .. first + 31 that token t selects, one bit each.  (An expert named twice is one bit.)
template <int K>
__device__ __forceinline__ unsigned experts_of(const uint16_t* ids, int t, unsigned first) {
    unsigned w[4] = {0u, 0u, 0u, 0u};
    if (K == 8) {
        const uint4 v = *reinterpret_cast<const uint4*>(ids + t * 8);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else if (K == 4) {
        const uint2 v = *reinterpret_cast<const uint2*>(ids + t * 4);
        w[0] = v.x; w[1] = v.y;
    } else if (K == 1) {
        w[0] = ids[t] | kNone << 16;
    } else {
#pragma unroll
        for (int i = 0; i < K / 2; ++i) w[i] = reinterpret_cast<const unsigned*>(ids + t * K)[i];
    }
    unsigned m = 0u;
#pragma unroll
    for (int i = 0; i < (K + 1) / 2; ++i) m |= bit_or_none((w[i] & 0xffffu) - first) | bit_or_none((w[i] >> 16) - first);
    return m;
}

// Small batches: every slot of the CTA's tokens has a warp.  A slot's warp reads the whole table (T tokens of k slots and some
// 8 more instructions' worth each) and an SM's four schedulers share the warps of up to `most` tokens, so the line lies at a
// product of these.  Dispatch + combine in one graph, as before and this way: 1 token of 7168 channels, top-8, bf16 8.4 and 5.3 us,
// 16 tokens of 4096 channels 8.6 and 5.5, 128 of 256 channels, top-2 7.9 and 4.6; near the line 256 tokens of 4096 channels,
// top-8 12.0 and 12.0 (FP8 rows 13.3 and 12.9), 444 of 1024, top-4 9.8 and 8.3 (10.2 and 9.9), 592 of 256, top-2 9.6 and 9.6
// (FP8); beyond it 296 tokens of 4096 channels, top-8 12.4 and 13.3, 512 of 1024, top-4 10.1 and 10.5, 740 of 256, top-2, FP8
// 9.9 and 11.1.
constexpr int kFewWork = 65536;

// The whole table into ids[], by n threads.  True if a slot's id was out of range.
template <int K>
__device__ __forceinline__ bool stage_table(const Params& p, uint16_t* ids, int tid, int n) {
    constexpr int kV = K % 4 == 0 ? 4 : K % 2 == 0 ? 2 : 1;   // slots per load
    bool bad = false;
#pragma unroll 1
    for (int i = tid; i < p.T * (K / kV); i += n) {
        const int t = i / (K / kV);
        if (kV == 4) {
            const int4 v = ld_plain(reinterpret_cast<const int4*>(p.topk_idx) + i);
            int e[4] = {v.x, v.y, v.z, v.w};
            resolve_slots(p, t, e, bad);
            reinterpret_cast<uint2*>(ids)[i] = make_uint2(pack16(e[0], e[1]), pack16(e[2], e[3]));
        } else if (kV == 2) {
            const int2 v = ld_plain(reinterpret_cast<const int2*>(p.topk_idx) + i);
            int e[2] = {v.x, v.y};
            resolve_slots(p, t, e, bad);
            reinterpret_cast<unsigned*>(ids)[i] = pack16(e[0], e[1]);
        } else {
            int e[1] = {ld_plain(p.topk_idx + i)};
            resolve_slots(p, t, e, bad);
            ids[i] = (uint16_t)e[0];
        }
    }
    return bad;
}

// The same, a thread per token, and the rows every rank receives added to rows[] (zero before).
template <int K>
__device__ __forceinline__ bool stage_tokens(const Params& p, uint16_t* ids, int* rows, bool dedup, int tid, int n) {
    bool bad = false;
#pragma unroll 1
    for (int t = tid; t < p.T; t += n) {
        int e[K];
#pragma unroll
        for (int j = 0; j < K; ++j) e[j] = 0;
        if (K % 4 == 0) {
#pragma unroll
            for (int j = 0; j < K / 4; ++j) {
                const int4 v = ld_plain(reinterpret_cast<const int4*>(p.topk_idx) + t * (K / 4) + j);
                e[4 * j] = v.x; e[4 * j + 1] = v.y; e[4 * j + 2] = v.z; e[4 * j + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < K; ++j) e[j] = ld_plain(p.topk_idx + t * K + j);
        }
        resolve_slots(p, t, e, bad);
#pragma unroll
        for (int j = 0; j < K / 2; ++j) reinterpret_cast<unsigned*>(ids)[t * (K / 2) + j] = pack16(e[2 * j], e[2 * j + 1]);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const int r = e[j] < 0 ? -1 - j : p.L == 1 ? e[j] : fast_div(e[j], p.L_magic);
            e[j] = dedup || e[j] < 0 ? r : e[j];
            bool first = e[j] >= 0;   // one row per (token, rank), or per (token, expert)
#pragma unroll
            for (int i = 0; i < j; ++i) first = first && e[i] != e[j];
            if (first) atomicAdd(rows + r, 1);
        }
    }
    return bad;
}

// Slot j of token t, by a warp.
struct SlotRow {
    unsigned e_i, f;   // lane i: expert of the token's slot i (kNone: none); first expert of the rank
    int r, row, at;    // rank (0 for an empty slot), row in its region (-1), place in the rank's list of rows by expert
    bool valid, twice; // there is an expert / it is one that an earlier slot of the token names
    bool here;         // lane i: slot i names the same rank
    bool first;        // no earlier slot of the token does, or it does not matter
};
// Rows: tokens before t that chose the expert, behind the experts of the rank in front of it; with one row per (token, rank)
// tokens before t that visit the rank.
template <int K>
__device__ __forceinline__ SlotRow slot_row(const Params& p, const uint16_t* ids, int t, int j, bool dedup, int lane) {
    SlotRow s{};
    s.row = -1;
    s.e_i = lane < K ? ids[t * K + lane] : kNone;
    const unsigned e = __shfl_sync(kAll, s.e_i, j);
    s.twice = e != kNone && __any_sync(kAll, lane < j && s.e_i == e);
    s.valid = e != kNone && !s.twice;
    if (!s.valid) return s;
    s.r = p.L == 1 ? (int)e : fast_div((int)e, p.L_magic);
    s.f = (unsigned)(s.r * p.L);
    const unsigned lbits = low_bits(p.L), d = e - s.f, below = (1u << d) - 1u;
    unsigned acc = 0u;
#pragma unroll 2
    for (int tt = lane; tt < p.T; tt += 32) {
        const unsigned m = experts_of<K>(ids, tt, s.f) & lbits;
        acc += (unsigned)__popc(m & below) << 16;
        if (tt < t) acc += ((m >> d) & 1u) << 16 | (m != 0u ? 1u : 0u);
    }
    acc = __reduce_add_sync(kAll, acc);   // (T * K < 2^16)
    s.at = (int)(acc >> 16);
    s.row = dedup ? (int)(acc & 0xffffu) : s.at;
    s.here = s.e_i - s.f < (unsigned)p.L;
    s.first = !dedup || !__any_sync(kAll, s.here && lane < j);
    return s;
}
// Its metadata; gpos: its row in the receive regions, -1 beyond the capacity; w_i: lane i, gate weight of slot i.
template <int K>
__device__ __forceinline__ void slot_meta(const Params& p, const SlotRow& s, int t, int j, int gpos, float w_i, bool dedup, int lane) {
    const bool send = s.valid && s.first && gpos >= 0;
    bool full = s.valid && gpos < 0;
    if (s.valid && dedup) {
        if (send) {
            bool again = false;   // a slot of the token in front of this lane's names the same expert
#pragma unroll
            for (int i = 1; i < K; ++i) {
                const unsigned other = __shfl_up_sync(kAll, s.e_i, i);
                again = again || (lane >= i && other == s.e_i);
            }
            if (lane < K) {
                p.recv_topk_idx[(size_t)gpos * K + lane] = s.here && !again ? (int)(s.e_i - s.f) : -1;
                p.recv_topk_w[(size_t)gpos * K + lane] = s.here && !again ? w_i : 0.0f;
            }
        }
    } else if (send && lane == j) {
        p.recv_weight[gpos] = w_i;
    }
    if (lane == 0) {
        if (send) p.recv_src_idx[gpos] = t;
        p.slot_row[(size_t)t * K + j] = s.row;
        p.slot_pos[(size_t)t * K + j] = gpos;
    }
    // (Last: in front of the others this store held them up by 0.9 us.)
    if (s.valid && dedup) {
        if (s.at < p.er_cap) {
            if (lane == 0) p.expert_rows[(size_t)s.r * p.er_cap + s.at] = s.row;
        } else {
            full = true;
        }
    }
    if (full) report(p.status, kErrCapacity);
}

// Per rank the totals and the expert offsets, per source rank counts and offsets.  A unit is a rank and as many source ranks
// as there are lanes for, a lane per (source rank, expert); `units` of them per rank (table_units).  (One loop of few instructions
// that keeps nothing per group of tokens: with the groups unrolled and their bitmaps in registers the dispatch of 1 to 13 tokens
// took 0.6 us more.)
__host__ __device__ inline int table_units(const Params& p) {
    int at_once = 32;   // source ranks a warp looks at together
    for (int l = 1; l < p.L; l *= 2) at_once /= 2;
    return (p.S + at_once - 1) / at_once;
}
template <int K>
__device__ __forceinline__ void write_table_unit(const Params& p, const uint16_t* ids, int u, int units, bool dedup, int lane) {
    const int lsh = 32 - __clz(p.L - 1);   // experts of a rank, rounded up to a power of two
    const int ur = u / units, uq = u - ur * units, f = ur * p.L;
    const int l = lane & ((1 << lsh) - 1), s = (uq << (5 - lsh)) + (lane >> lsh);
    const bool mine = s < p.S && l < p.L;
    const int b0 = src_begin(min(s, p.S), p.T, p.S), b1 = src_begin(min(s + 1, p.S), p.T, p.S);
    const unsigned lbits = low_bits(p.L);
    int tot = 0, visits = 0;         // tokens that chose expert `lane` of the rank / that visit it
    int before = 0, after = 0;       // tokens before the source rank's first and behind its last one that chose expert l
#pragma unroll 1
    for (int g = 0; g < p.T; g += 32) {
        const unsigned m = g + lane < p.T ? experts_of<K>(ids, g + lane, (unsigned)f) & lbits : 0u;
        visits += m != 0u ? 1 : 0;
        const unsigned bm = transpose32(m, lane);   // lane = expert, bit = token
        tot += __popc(bm);
        const unsigned of_l = __shfl_sync(kAll, bm, l);
        before += __popc(of_l & low_bits(b0 - g));
        after += __popc(of_l & low_bits(b1 - g));
    }
    const int incl = warp_incl_scan(tot, lane), eo = incl - tot, eo_l = __shfl_sync(kAll, eo, l);
    if (mine) {
        p.cnt[(size_t)s * p.E + f + l] = after - before;
        p.src_offset[(size_t)s * p.E + f + l] = eo_l + before;
    }
    if (uq == 0) {
        if (lane < p.L) {
            p.expert_offset[f + lane] = eo;
            p.num_tokens_per_expert[f + lane] = tot;
        }
        visits = __reduce_add_sync(kAll, visits);
        const int rows = __shfl_sync(kAll, incl, 31);
        if (lane == 0) {
            p.num_tokens_per_rank[ur] = visits;
            p.num_rows_per_rank[ur] = dedup ? visits : rows;
        }
    }
}

}  // namespace ubep
