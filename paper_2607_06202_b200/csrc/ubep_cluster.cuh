// Layout of dispatch by thread-block clusters (sm_100a): the CTAs of a cluster count the whole routing table
// between them and exchange what they counted through distributed shared memory.  Nothing is exchanged between
// clusters, so there are no flags in global memory, no second hop and no wait for CTAs that may not run yet.
//
// Why: exchanging counts between all 148 CTAs through global memory released the first copy 14 - 17 us after the
// kernel's start (counts published 6.4, all of them seen 9.2, prefix sums published 12.6 and seen 14.0, rows
// assigned 17.0 us at 4096 tokens).  Here it leaves 4.4 us after the start at 1537 tokens and 6.9 us at 4096.
#pragma once

#include "ubep_layout.cuh"

namespace ubep {

__device__ __forceinline__ unsigned cluster_ctarank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Barrier of all threads of the cluster in two halves: what precedes an arrive is visible after the wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// A word of another CTA's shared memory.
__device__ __forceinline__ unsigned ld_cluster(const unsigned* mine, unsigned rank) {
    uint32_t a;
    unsigned v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(mine)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// What counting needs of the parameters; by value, so that the (out of line) counting functions do not make the
// kernel keep its parameters in addressable memory.
struct CountArgs {
    const int32_t *topk_idx, *phys, *ncopies;
    int k, E, R, L, E_log, C;
    unsigned L_magic;
};
__device__ __forceinline__ CountArgs count_args(const Params& p) {
    return {p.topk_idx, p.phys, p.ncopies, p.k, p.E, p.R, p.L, p.E_log, p.C, p.L_magic};
}

static __device__ __noinline__ int modulo(int a, int b) { return a % b; }   // (out of line: small code, see count_tokens)

// Physical expert of a slot of token t; a negative number of the slot's own (never equal to another slot's) if
// there is none.
__device__ __forceinline__ int counted_expert(const CountArgs& p, int t, int raw, int slot) {
    int e = raw;
    if (p.phys != nullptr) {
        const int nc = (unsigned)e < (unsigned)p.E_log ? ld_plain(p.ncopies + e) : 0;
        e = nc >= 1 && nc <= p.C ? ld_plain(p.phys + (size_t)e * p.C + modulo(t, nc)) : -1;
    }
    return (unsigned)e < (unsigned)p.E ? e : -1 - slot;
}

// Counts, per bin, the tokens of [lo, hi) -- and how many of them are below `split` -- that selected it, into
// cnt[] as (all << 16 | below); a thread per token.  ranks: rank bins too (from cnt[E] on).  A slot that is empty or
// bad counts nowhere (in cnt[E + R], that is: cnt holds E + R + 1 words, whatever `ranks`), an expert a token names
// twice counts once (the CTA that owns the token reports both).
//
// Written for few instructions: this runs once per launch, so what it costs first of all is fetching its code (a
// first form, which collected a token's slots in 32-bit words of bins and transposed them, was 600 instructions
// and took 5 us for its first 32 tokens).  The adds are cheap: 3.6 cycles per warp for random bins.
// Tokens of [lo2, hi2) are counted into cnt2[] as well (all << 16, experts only).
static __device__ __noinline__ void count_tokens(const CountArgs p, int lo, int hi, int split, bool ranks, unsigned* cnt,
                                                 int tid, int n, int lo2 = 0, int hi2 = 0, unsigned* cnt2 = nullptr) {
    const int k = p.k;
    const bool words = k == 8 || k == 4;   // a token's ids are whole 16-byte words (topk_idx is 16-byte aligned)
    const int none = p.E + p.R;
    auto fetch = [&](int t, int4& a, int4& b) {
        const int4* src = reinterpret_cast<const int4*>(p.topk_idx + (size_t)t * k);
        a = b = make_int4(-1, -1, -1, -1);
        if (t < hi) {
            a = ld_plain(src);
            if (k == 8) b = ld_plain(src + 1);
        }
    };
    int4 na, nb;
    if (words) fetch(lo + tid, na, nb);
    for (int t = lo + tid; t < hi; t += n) {
        const unsigned inc = t < split ? 0x10001u : 0x10000u;
        if (words) {
            int e[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
            fetch(t + n, na, nb);   // the next token's ids while this one's are counted
            if (p.phys != nullptr) {
                int nc[8];
                bool many = false;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    nc[j] = (unsigned)e[j] < (unsigned)p.E_log ? ld_plain(p.ncopies + e[j]) : 0;
                    many = many || nc[j] > 2;
                }
                if (many) {
#pragma unroll 1
                    for (int j = 0; j < 8; ++j) {   // (rotates through the slots so that they stay in registers)
                        const int v = counted_expert(p, t, e[0], 0);
#pragma unroll
                        for (int i = 0; i < 7; ++i) e[i] = e[i + 1];
                        e[7] = v;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        e[j] = nc[j] >= 1 && nc[j] <= p.C ? ld_plain(p.phys + (size_t)e[j] * p.C + (nc[j] == 2 ? t & 1 : 0)) : -1;
                }
            }
            bool twice = false;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                e[j] = (unsigned)e[j] < (unsigned)p.E ? e[j] : -1 - j;
#pragma unroll
                for (int i = 0; i < j; ++i) twice = twice || e[i] == e[j];
            }
            if (twice) {   // (an error case)
#pragma unroll
                for (int j = 1; j < 8; ++j)
#pragma unroll
                    for (int i = 0; i < j; ++i)
                        if (e[i] == e[j]) e[j] = -1 - j;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) atomicAdd(cnt + (e[j] >= 0 ? e[j] : none), inc);
            if (t >= lo2 && t < hi2) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (e[j] >= 0) atomicAdd(cnt2 + e[j], 0x10000u);
            }
            if (ranks) {   // a rank counts a token once: with the first of the slots that name it
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int r = p.L == 1 ? e[j] : fast_div(e[j], p.L_magic);
                    e[j] = e[j] >= 0 ? r : e[j];
                    bool first = e[j] >= 0;
#pragma unroll
                    for (int i = 0; i < j; ++i) first = first && e[i] != e[j];
                    atomicAdd(cnt + (first ? p.E + e[j] : none), inc);
                }
            }
        } else {
            const int32_t* src = p.topk_idx + (size_t)t * k;
            int e[kMaxTopk];
#pragma unroll 1
            for (int j = 0; j < k; ++j) {
                int v = counted_expert(p, t, ld_plain(src + j), j);
#pragma unroll 1
                for (int i = 0; i < j; ++i)
                    if (e[i] == v) v = -1 - j;
                e[j] = v;
                if (v < 0) continue;
                atomicAdd(cnt + v, inc);
                if (t >= lo2 && t < hi2) atomicAdd(cnt2 + v, 0x10000u);
                if (!ranks) continue;
                const int r = p.L == 1 ? v : fast_div(v, p.L_magic);
                bool first = true;
#pragma unroll 1
                for (int i = 0; i < j; ++i) first = first && (e[i] < r * p.L || e[i] >= (r + 1) * p.L);
                if (first) atomicAdd(cnt + p.E + r, inc);
            }
        }
    }
}

// The ids of the CTA's own tokens [t0, t1): packed (expert | rank << 16) into ids[], one bit per token and bin into
// the bitmaps (zero before) and the bins' counts into own[], a thread per slot.  A bad id is reported.  Returns
// true if some expert was named twice by a token (local_clean_own_duplicates then empties the later slot).
__device__ __forceinline__ bool stage_own(const Params& p, int t0, int t1, int* ids, unsigned* bm, int bp, unsigned* own,
                                          int tid, int n) {
    const int nslots = (t1 - t0) * p.k;
    bool bad = false, twice = false;
#pragma unroll 1
    for (int i = tid; i < nslots; i += n) {
        const int tl = i / p.k;
        const int v = pack_slot(p, (size_t)t0 * p.k + i, ld_plain(p.topk_idx + (size_t)t0 * p.k + i), bad);
        ids[i] = v;
        if (v >= 0) {
            const unsigned bit = 1u << (tl & 31);
            unsigned* g = bm + (size_t)(tl >> 5) * bp;
            const int e = slot_expert(v), r = p.E + slot_rank(v);
            const unsigned be = atomicOr(g + e, bit), br = atomicOr(g + r, bit);
            if (be & bit) twice = true;
            else atomicAdd(own + e, 1u);
            if (!(br & bit)) atomicAdd(own + r, 1u);
        }
    }
    if (bad) report(p.status, kErrBadIndex);
    return twice;
}

// Tokens before the CTA's own token tl that selected `bin`.
__device__ __forceinline__ int own_below(const BinMaps& m, int bin, int tl) {
    const int g1 = tl >> 5;
    int c = __popc(m.bm[(size_t)g1 * m.bp + bin] & ((1u << (tl & 31)) - 1u));
#pragma unroll 1
    for (int g = 0; g < g1; ++g) c += __popc(m.bm[(size_t)g * m.bp + bin]);
    return c;
}

// What the source ranks whose tokens begin among [t0, t1) report (cnt, src_offset).  base[e]: rows before the CTA's
// tokens in expert e's segment.  Tokens of the last such rank beyond the CTA's own are counted from the table into
// cnt (E + R + 1 words), unless that has been done.  The column parts of a chunk share its source ranks.  Run by n threads that share barrier `bar`.
__device__ __forceinline__ int own_sources_end(const Params& p, int t1) {   // first token beyond the source ranks that begin below t1
    return src_begin(min(p.S, (int)(((int64_t)t1 * p.S + p.T - 1) / p.T)), p.T, p.S);
}
template <bool kCounted>
static __device__ void write_own_sources(const Params& p, int t0, int t1, int part, int parts, const BinMaps& bmaps, const int* base, unsigned* cnt,
                                         int tid, int n, int bar) {
    // source ranks s_lo .. s_hi - 1
    const int s_lo = (int)(((int64_t)t0 * p.S + p.T - 1) / p.T);
    const int s_hi = min(p.S, (int)(((int64_t)t1 * p.S + p.T - 1) / p.T));
    if (s_hi - s_lo <= part) return;
    const int last_end = src_begin(s_hi, p.T, p.S);
    if (!kCounted && last_end > t1) {
        for (int e = tid; e < p.E; e += n) cnt[e] = 0u;
        group_sync(bar, n);
        count_tokens(count_args(p), t1, last_end, 0, false, cnt, tid, n);
        group_sync(bar, n);
    }
#pragma unroll 1
    for (int s = s_lo + part; s < s_hi; s += parts) {
        const int b0 = src_begin(s, p.T, p.S), b1 = src_begin(s + 1, p.T, p.S);
#pragma unroll 1
        for (int e = tid; e < p.E; e += n) {
            const int before = own_below(bmaps, e, b0 - t0);
            p.cnt[(size_t)s * p.E + e] = own_below(bmaps, e, min(b1, t1) - t0) - before + (b1 > t1 ? (int)(cnt[e] >> 16) : 0);
            p.src_offset[(size_t)s * p.E + e] = base[e] + before;
        }
    }
}

}  // namespace ubep
