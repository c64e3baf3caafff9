// Batched-launch data structures shared by the batch entry points (batch.cu)
// and the server (server.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "gbaes_internal.h"

namespace gbaes {

struct MsgDev {  // 32 bytes, group order
    uint64_t blk_start;  // first block of the message in its group's block space
    uint64_t in_blk;     // in_off / 16
    uint64_t out_blk;    // out_off / 16
    uint32_t key_slot;   // schedule slot (2 * key_index + decrypt)
    uint32_t src;        // caller's message index
};

struct GroupDev {
    uint32_t tile_start, tile_end;  // tiles [tile_start, tile_end)
    uint32_t msg_start, msg_end;    // messages [msg_start, msg_end) in group order
    uint64_t blocks;                // blocks in the group
    int32_t nr;
    int32_t dir;  // 0 encrypt, 1 decrypt
};

constexpr int kGroups = 6;
constexpr int kCtasDone = 1;  // BatchArgs::counter[kCtasDone]
constexpr int kSlotWords = 64;  // 60 used (Nr = 14), padded to 256 bytes

struct BatchArgs {
    const uint4* in;
    uint4* out;
    const MsgDev* msgs;
    const uint4* keys;  // kSlotWords / 4 uint4 per slot
    const uint32_t* tile_msg;
    unsigned* counter;  // two words, zero at the launch and after it (units taken, CTAs done),
                        // or nullptr: no more units than warps
    uint32_t ntiles;
    uint32_t tile_blocks;
    uint32_t whole;  // the first tiles, which warps take 2^join at a time ...
    uint32_t join;
    uint32_t split;  // ... and of the others 1 / 2^split of one
    GroupDev groups[kGroups];
};

struct HostPlan {
    std::vector<MsgDev> msgs;
    std::vector<uint32_t> tile_msg;
    GroupDev groups[kGroups];
    uint32_t ntiles = 0;
    uint32_t tile_blocks = 0;
    uint64_t total_blocks = 0;
    uint64_t in_extent = 0;   // bytes from in_base the plan reads
    uint64_t out_extent = 0;  // bytes from out_base the plan writes
};

// Validates descriptors and lays out groups and tiles.
int build_host_plan(const aes_msg_desc* d, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx, uint32_t tile_blocks,
                    HostPlan* P);

// How one batched launch shares its tiles among the GPU's warps (BatchArgs::whole, split).
struct BatchSchedule {
    uint32_t whole;
    uint32_t join;
    bool joined;  // whole units have several passes: the kernel that runs each by itself
    uint32_t split;
    uint32_t grid;
    bool counted;  // some warps take more than one unit: the launch needs its counter, zeroed
};
BatchSchedule schedule_batch(const HostPlan& H, int threads, int bpt, int sms);

// Launches the batched kernel (one CTA per SM at most; ntiles > 0): fills in a.whole and a.split and, where the
// schedule needs none, clears a.counter.
int launch_batch_kernel(const HostPlan& H, BatchArgs a, int threads, int bpt, cudaStream_t stream);

int device_status_word(int** p);  // ecb_table.cu

}  // namespace gbaes
