// Host-visible launchers of the readiness-protocol dispatch (ubep_sync.cu).
#pragma once

#include <cuda_runtime.h>

#include "ubep_common.cuh"

namespace ubep {

constexpr int kErrChecksum = -7;     // mirrors UBEP_ERR_CHECKSUM
constexpr int kSyncTimeSlots = 8;    // per-CTA time stamps of the last call

// Wire-buffer arrays and the protocol of one call.
struct SyncParams {
    int protocol;                   // UBEP_SYNC_*
    int tff_blocks;                 // 16-byte DataBlocks per row: ceil(rowB / 12)
    int tff_strips;                 // Token-Flag payload passes through shared memory (else in single words)
    uint8_t* tff_wire;              // [R * cap][16 * tff_blocks]
    uint8_t* sp_wire;               // [R * cap][rowB]
    unsigned long long* checksum;   // [2][R]
    unsigned* announced;            // [2][R] senders that have added their marker sums
    unsigned* sw_rows;              // [2][R] rows whose stores have been fenced
    unsigned* seq_ctr;              // calls completed
    unsigned* seq_ticket;           // CTAs of the running call that have read seq_ctr
    unsigned* sp_dirty;             // != 0: a Sentinel Polling call gave up and may have left arrived blocks in the wire
    unsigned long long* times;      // [grid][kSyncTimeSlots]
};

// Dynamic shared memory the kernel needs beyond the dispatch plan's total; with Token-Flag strips or without.
int sync_extra_smem(const Params& p, int protocol, bool strips);

// Where the layout comes from: the count / prefix-sum launches (launch_count_scan) that have run before over the same
// p.nchunks chunks; the whole routing table, counted by every CTA; for small tables a warp per slot.
constexpr int kSyncLaunched = 0, kSyncWhole = 1, kSyncFew = 2;
cudaError_t launch_sync_dispatch(const Params& p, const SmemPlan& pl, const SyncParams& sp, int how, cudaStream_t st);
// Whether the call is one of the last kind: the plan then, and p's chunks and parts (unchanged otherwise).
bool plan_sync_few(Params& p, int protocol, int max_smem, SmemPlan* out);

// Counts the 16-byte vectors of x that consist of 0xFFFF elements only.
cudaError_t launch_sentinel_scan(const void* x, long long n_vec, unsigned long long* count, int num_sms,
                                 cudaStream_t st);

}  // namespace ubep
