// Batched multi-key AES-ECB: many messages, each with its own key, key size and
// direction, in one persistent launch.
//
// The paper's draw-per-buffer design pays a per-operation overhead that
// dominates small inputs (Section 3.1; its conclusion advises against small
// messages).  Here thousands of messages share one launch:
//
//  * Host plan (batch_plan.h).  Messages are grouped by (direction, key size)
//    -- encryption groups first -- and each group's blocks are numbered
//    contiguously.  The flattened block space is cut into tiles; for every tile
//    the plan records the first message it touches.  Each (key, direction)
//    gets a slot holding its 4*(Nr+1)-word schedule.  Everything sits in one
//    device buffer, uploaded once per plan.
//  * Kernel.  One CTA per SM holds both directions' tables (aes_rounds.cuh).
//    Each *warp* starts on a fixed unit (a few tiles, or a part of one where there are
//    few tiles for the warps to share), then takes units from an atomic
//    counter on its own, so the dependent loads at the start of one warp's unit
//    overlap the other warps' lookups.  Where its blocks lie in one message a warp stages
//    that message's schedule in its shared-memory key slot; elsewhere every block
//    finds its message from the starts of the next 32, and keys come from
//    global memory through L1.  The round count is a run-time loop bound,
//    so one compact body per direction serves all key sizes.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <set>
#include <utility>
#include <vector>

#include "aes_rounds.cuh"
#include "batch_plan.h"
#include "launch.cuh"
#include "rounds_rt.cuh"

namespace gbaes {

constexpr uint32_t kPlanTileMax = 512;  // largest tile of a batch plan, in blocks

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

constexpr uint32_t kNoBoundary = 0x7fffffffu;

// Blocks per thread of the passes that messages start in.  A body of 8 states there, beside
// the one of the passes that lie in one message, is too much for the instruction cache:
// 512 x 8, 3,000 messages of 8,208 bytes (25 MB) 72.3 us with 8, 3.5 cycles of instruction fetch
// per instruction issued (0.5 with the shorter rounds of four tables, 59.6 us), 56.6 with 4;
// 10,000 messages up to 16 KiB (23 MB) 69.8 -> 54.0, up to 64 KiB (77 MB) 139.6 -> 127.2, up to
// 128 KiB (141 MB) 240 -> 221, up to 4 MiB (3.2 GB) 4,102 -> 4,104.  With 2: 51.5, 49.1, 126.9, 216
// and 4,105, but 5-20% more than 4 in batches of up to 5 MB.
constexpr int kMixedBpt = 4;

// Starts of the messages after `base`, relative to tb0: lane l gets message
// base + 1 + l's (kNoBoundary past the group's last message or far away; 0 for
// any start at or before tb0).  One coalesced load tells a warp where 32
// messages begin.
__device__ __forceinline__ uint32_t load_starts(const BatchArgs& a, const GroupDev& G, uint32_t base, uint64_t tb0,
                                                uint32_t lane) {
    const uint32_t m = base + 1u + lane;
    if (m >= G.msg_end || m < base) return kNoBoundary;
    const uint64_t s = __ldg((const unsigned long long*)(a.msgs + m));
    if (s <= tb0) return 0u;
    return s - tb0 < kNoBoundary ? (uint32_t)(s - tb0) : kNoBoundary;
}

// n consecutive blocks from tb0 inside one message m (the common case: 97.5% of
// the 512-block tiles of a batch of 10,000 messages, 16 B - 4 MiB), processed
// 32*BPT at a time (lane l, slot b -> block it + 32b + l, so every load and store
// instruction of the warp covers 512 contiguous bytes).  The descriptor is
// read once and m's schedule is staged in the warp's shared-memory key slot:
// one parallel load instead of a dependent global load per round, issued once
// the first data loads are in flight so that the two overlap.  Lanes past the
// end compute on zeros and store nothing, so the warp stays converged.
template <bool DEC, int BPT>
__device__ __forceinline__ void single_message_unit(const BatchArgs& a, const GroupDev& G, uint32_t m, uint64_t tb0,
                                                    uint32_t n, uint32_t lane, uint32_t L,
                                                    uint32_t kslot) {
    const uint4* mp = (const uint4*)(a.msgs + m);
    const uint4 q0 = __ldg(mp);
    const uint4 q1 = __ldg(mp + 1);
    const uint64_t off = tb0 - (((uint64_t)q0.y << 32) | q0.x);  // tb0 - blk_start
    const uint4* in = a.in + ((((uint64_t)q0.w << 32) | q0.z) + off);
    uint4* out = a.out + ((((uint64_t)q1.y << 32) | q1.x) + off);
    for (uint32_t it = 0; it < n; it += 32u * BPT) {
        uint32_t s[BPT][4];
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const uint32_t i = it + 32u * b + lane;
            const uint4 v = i < n ? ld_stream(in + i) : make_uint4(0, 0, 0, 0);
            s[b][0] = v.x;
            s[b][1] = v.y;
            s[b][2] = v.z;
            s[b][3] = v.w;
        }
        if (it == 0) {  // (every lane is done with the slot: the warp met to choose these blocks)
            if (lane < (uint32_t)G.nr + 1u) {
                const uint4 k = __ldg(a.keys + (uint64_t)q1.z * (kSlotWords / 4) + lane);
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(kslot + 16u * lane), "r"(k.x),
                             "r"(k.y), "r"(k.z), "r"(k.w)
                             : "memory");
            }
            __syncwarp();
        }
        cipher_rt<DEC, BPT>(s, SmemKeys{kslot}, G.nr, L);
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const uint32_t i = it + 32u * b + lane;
            if (i < n) __stcs(out + i, make_uint4(s[b][0], s[b][1], s[b][2], s[b][3]));
        }
    }
}

// The passes (32*BPT blocks) from tb0 + it on up to tb0 + end, in a unit that ends at
// tb0 + n and crosses message boundaries; block `it` is in message m; `starts`:
// load_starts of a message at most 32 before the next boundary.  Both are left as
// the block after the last pass needs them.  Each block finds its message from the
// window of starts: a ballot counts those a pass leaves behind, an OR over the warp
// marks the blocks at which a message begins, and a lane's message is the one of
// block 0 plus the marks up to the lane.  (A binary search per block took five or more dependent loads;
// with the finer units of schedule_batch, the kernel's time for 2,000 messages of
// 16 B - 16 KiB went from 33 to 14 us in a plan of 1024 x 2 and from 199 to 15 us in
// a one-shot call.)  The states of one thread may belong to different messages:
// each reads its own round keys from global memory through L1, where the
// schedule's second line is fetched ahead, and the warp runs one interleaved
// cipher over all of them (no divergent per-block ciphers at a boundary).
template <bool DEC, int BPT>
__device__ __forceinline__ void mixed_passes(const BatchArgs& a, const GroupDev& G, uint32_t& m, uint32_t& starts,
                                             uint64_t tb0, uint32_t it, uint32_t end, uint32_t n, uint32_t lane,
                                             uint32_t L) {
    uint32_t wlast = __shfl_sync(0xffffffffu, starts, 31);  // the window's last entry
    for (; it < end; it += 32u * BPT) {
        uint32_t s[BPT][4];
        uint64_t oidx[BPT];
        uint32_t slot[BPT];
        bool ok[BPT];
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const uint32_t g0 = it + 32u * b;
            if (wlast <= g0 + 32u) {  // the window must reach past these blocks
                starts = load_starts(a, G, m, tb0, lane);
                wlast = __shfl_sync(0xffffffffu, starts, 31);
            }
            const uint32_t marks =
                __reduce_or_sync(0xffffffffu, starts > g0 && starts < g0 + 32u ? 1u << (starts - g0) : 0u);
            const uint32_t own = m + __popc(marks & (0xffffffffu >> (31u - lane)));
            m += __popc(__ballot_sync(0xffffffffu, starts > g0 && starts <= g0 + 32u));
            ok[b] = g0 + lane < n;
            uint4 v = make_uint4(0, 0, 0, 0);
            slot[b] = 0;
            oidx[b] = 0;
            if (ok[b]) {
                const uint4* mp = (const uint4*)(a.msgs + own);
                const uint4 r0 = __ldg(mp);
                const uint4 r1 = __ldg(mp + 1);
                const uint64_t off = tb0 + g0 + lane - (((uint64_t)r0.y << 32) | r0.x);
                v = ld_stream(a.in + ((((uint64_t)r0.w << 32) | r0.z) + off));
                oidx[b] = (((uint64_t)r1.y << 32) | r1.x) + off;
                slot[b] = r1.z;
                prefetch_l1(a.keys + (uint64_t)r1.z * (kSlotWords / 4) + 8);
            }
            s[b][0] = v.x;
            s[b][1] = v.y;
            s[b][2] = v.z;
            s[b][3] = v.w;
        }
        if (ok[0]) {  // (else this lane's blocks are all past the end)
#pragma unroll
            for (int b = 1; b < BPT; ++b)
                if (!ok[b]) slot[b] = slot[0];  // (past the end: computes on zeros with a valid key, stores nothing)
            cipher_rt<DEC, BPT>(s, StateKeys<BPT, kSlotWords / 4>{a.keys, slot}, G.nr, L);
#pragma unroll
            for (int b = 0; b < BPT; ++b)
                if (ok[b]) __stcs(a.out + oidx[b], make_uint4(s[b][0], s[b][1], s[b][2], s[b][3]));
        }
        __syncwarp();
    }
}

// The tiles [t, e) of group G, or part `sub` of tile t, `part` blocks in all (a tile is
// tile_blocks consecutive blocks of the group's block space, fewer in the group's last one).
template <bool DEC, int BPT, bool JOINED>
__device__ __forceinline__ void batch_warp_unit(const BatchArgs& a, const GroupDev& G, uint32_t t, uint32_t e,
                                                uint32_t sub, uint32_t part, uint32_t lane, uint32_t L,
                                                uint32_t kslot) {
    const uint64_t tb0 = (uint64_t)(t - G.tile_start) * a.tile_blocks + sub * part;
    if (tb0 >= G.blocks) return;
    const uint64_t left = G.blocks - tb0;
    const uint32_t n = left < part ? (uint32_t)left : part;
    const uint32_t m_lo = a.tile_msg[t];
    const uint32_t m_hi = e < G.tile_end ? a.tile_msg[e] : G.msg_end - 1;
    uint32_t m = m_lo, starts = kNoBoundary;
    if (m_lo != m_hi) {
        for (;;) {  // find tb0's message; the starts after it stay in the window
            starts = load_starts(a, G, m, tb0, lane);
            const uint32_t passed = __popc(__ballot_sync(0xffffffffu, starts == 0u));
            m += passed;
            if (passed < 32u) break;
        }
    }
    constexpr uint32_t kPass = 32u * BPT;
    constexpr int kMixed = BPT < kMixedBpt ? BPT : kMixedBpt;
    const bool crossing = __any_sync(0xffffffffu, starts != 0u && starts < n);
    if (!JOINED) {
        if (!crossing)
            single_message_unit<DEC, BPT>(a, G, m, tb0, n, lane, L, kslot);
        else
            mixed_passes<DEC, kMixed>(a, G, m, starts, tb0, 0, n, n, lane, L);
        return;
    }
    // Whole passes up to the next message's start (or the end) run with one message's
    // keys, those that cross a start one by one.
    uint32_t len = crossing ? 0u : n;
    for (uint32_t it = 0; it < n;) {
        uint32_t next = 0;
        if (len == 0u) {
            if (__shfl_sync(0xffffffffu, starts, 31) <= it) starts = load_starts(a, G, m, tb0, lane);
            next = __reduce_min_sync(0xffffffffu, starts > it ? starts : kNoBoundary);
            len = next >= n ? n - it : (next - it) & ~(kPass - 1u);
        }
        if (len) {
            single_message_unit<DEC, BPT>(a, G, m, tb0 + it, len, lane, L, kslot);
            it += len;
            m += next == it;
            len = 0;
        } else {
            const uint32_t stop = BPT == kMixed ? it + 1 : it + kPass < n ? it + kPass : n;
            mixed_passes<DEC, kMixed>(a, G, m, starts, tb0, it, stop, n, lane, L);
            it += kPass;
        }
    }
}

// Group table staged in shared memory (read with a runtime index per tile).
__device__ __forceinline__ GroupDev load_group(uint32_t gaddr, int g) {
    GroupDev G;
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = lds(gaddr + 32u * g + 4u * i);
    G.tile_start = w[0];
    G.tile_end = w[1];
    G.msg_start = w[2];
    G.msg_end = w[3];
    G.blocks = ((uint64_t)w[5] << 32) | w[4];
    G.nr = (int32_t)w[6];
    G.dir = (int32_t)w[7];
    return G;
}

// Units: the first `whole` tiles, 2^join of them each (JOINED; a unit that reaches into
// another group takes its tiles group by group), then the others in 2^split parts
// each; encryption first (groups 0-2), then decryption, both directions' tables in
// shared memory throughout.  Every warp starts on a fixed unit (interleaved over the
// CTAs, so a small batch spreads over the SMs), then takes units from a counter,
// independently of the other warps, so their global-memory latencies overlap.
// Without a counter (no more units than warps) that is all.
constexpr uint32_t kBatchSlots = 2 * kTableBytes;         // key slots: 256 B per warp
constexpr uint32_t kBatchGroups = kBatchSlots + 256u * 32;  // group table
constexpr uint32_t kBatchSmem = kBatchGroups + 32u * kGroups;

template <int BPT, bool JOINED>
__global__ void __launch_bounds__(BPT == 8 ? 512 : 1024, 1) batch_kernel(const BatchArgs a) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t A = smem_base(smem_raw);
    const uint32_t gaddr = A + kBatchGroups;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) {
        if (threadIdx.x == (unsigned)i) {
            const GroupDev& G = a.groups[i];
            const uint32_t w[8] = {G.tile_start, G.tile_end, G.msg_start, G.msg_end, (uint32_t)G.blocks,
                                   (uint32_t)(G.blocks >> 32), (uint32_t)G.nr, (uint32_t)G.dir};
#pragma unroll
            for (int k = 0; k < 8; ++k) sts(gaddr + 32u * i + 4u * k, w[k]);
        }
    }
    const uint32_t enc_tiles = a.groups[kGroups / 2 - 1].tile_end;
    if (enc_tiles) fill_table(A, false, threadIdx.x, blockDim.x);
    if (enc_tiles < a.ntiles) fill_table(A + kTableBytes, true, threadIdx.x, blockDim.x);
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t L = A + 4u * lane;
    const uint32_t kslot = A + kBatchSlots + 256u * (threadIdx.x >> 5);
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    const uint32_t units = (a.whole >> a.join) + ((a.ntiles - a.whole) << a.split);
    pdl_wait();
    pdl_trigger();  // (at the start: 136.0 us instead of 131.9 for 85 MB, 45.0 / 44.2 for 27 MB)
    uint32_t u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (u < units) {
        uint32_t nxt = units;
        if (a.counter && lane == 0) nxt = atomicAdd(a.counter, 1u) + warps;  // consumed after this unit
        const uint32_t join = JOINED ? a.join : 0u;
        uint32_t t = u << join, end = t + (1u << join), sub = 0, part = a.tile_blocks;
        if (t >= a.whole) {
            const uint32_t c = u - (a.whole >> join);
            t = a.whole + (c >> a.split);
            end = t + 1;
            sub = c & ((1u << a.split) - 1u);
            part = a.tile_blocks >> a.split;
        }
        do {
            int g = 0;
            while (g < kGroups - 1 && t >= lds(gaddr + 32u * g + 4u)) ++g;  // tile_end of group g
            const GroupDev G = load_group(gaddr, g);
            const uint32_t e = JOINED && end > G.tile_end ? G.tile_end : end;
            if (JOINED) part *= e - t;
            if (G.dir)
                batch_warp_unit<true, BPT, JOINED>(a, G, t, e, sub, part, lane, L + kTableBytes, kslot);
            else
                batch_warp_unit<false, BPT, JOINED>(a, G, t, e, sub, part, lane, L, kslot);
            if (!JOINED) break;
            t = e;
            part = a.tile_blocks;
        } while (t < end);
        u = __shfl_sync(0xffffffffu, nxt, 0);
    }
    if (!a.counter) return;
    // The last CTA to get here leaves the counter at zero for the next launch of
    // these tables (which waits for this one's end).
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.counter + kCtasDone, 1u) == gridDim.x - 1) {
            a.counter[0] = 0;
            a.counter[kCtasDone] = 0;
        }
    }
}

// ------------------------------------------------------------------ host plan

constexpr size_t kMaxMessages = 0xFFFFFFF0u;

static int group_of(int nr, int dir) { return dir * 3 + (nr == 10 ? 0 : nr == 12 ? 1 : 2); }

// Validates the descriptors and lays out groups and tiles: one pass checks and
// counts, a second writes each message to its place.
int build_host_plan(const aes_msg_desc* d, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx, uint32_t tile_blocks,
                    HostPlan* P) {
    if (nmsg && !d) return fail(AES_ERR_ARG, "message descriptors are NULL");
    if (nctx && !ctxs) return fail(AES_ERR_ARG, "key contexts are NULL");
    if (nmsg > kMaxMessages) return fail(AES_ERR_ARG, "too many messages (%zu)", nmsg);
    if (tile_blocks == 0) return fail(AES_ERR_ARG, "tile size is zero");
    for (size_t i = 0; i < nctx; ++i)
        if (!ctxs[i] || ctxs[i]->magic != kCtxMagic) return fail(AES_ERR_ARG, "ctxs[%zu] is not a valid aes_ctx", i);
    uint32_t count[kGroups] = {};
    uint64_t blocks[kGroups] = {};
    std::vector<uint8_t> group;  // of each message; kGroups: no blocks.  Grows with the messages found valid.
    for (size_t i = 0; i < nmsg; ++i) {
        const aes_msg_desc& m = d[i];
        if (m.key_index >= nctx) return fail(AES_ERR_ARG, "message %zu: key_index %u >= %zu", i, m.key_index, nctx);
        if (m.decrypt > 1) return fail(AES_ERR_ARG, "message %zu: decrypt must be 0 or 1", i);
        if ((m.in_off | m.out_off) & 15u) return fail(AES_ERR_ALIGN, "message %zu: offsets must be multiples of 16", i);
        if (m.nblocks > (UINT64_MAX >> 5)) return fail(AES_ERR_ARG, "message %zu: nblocks too large", i);
        const uint64_t bytes = m.nblocks * 16;
        if (m.in_off > UINT64_MAX - bytes || m.out_off > UINT64_MAX - bytes)
            return fail(AES_ERR_ARG, "message %zu: offset + length overflows", i);
        if (i == group.size()) group.resize(std::min(nmsg, std::max<size_t>(2 * i, 1 << 20)));
        group[i] = kGroups;
        if (m.nblocks == 0) continue;
        P->in_extent = std::max<uint64_t>(P->in_extent, m.in_off + bytes);
        P->out_extent = std::max<uint64_t>(P->out_extent, m.out_off + bytes);
        const int g = group_of(ctxs[m.key_index]->nr, (int)m.decrypt);
        group[i] = (uint8_t)g;
        ++count[g];
        blocks[g] += m.nblocks;
    }
    P->tile_blocks = tile_blocks;
    uint64_t tiles = 0, msgs = 0;
    uint32_t next[kGroups];  // where each group's next message goes
    for (int g = 0; g < kGroups; ++g) {
        GroupDev& G = P->groups[g];
        G.nr = g % 3 == 0 ? 10 : g % 3 == 1 ? 12 : 14;
        G.dir = g / 3;
        next[g] = G.msg_start = (uint32_t)msgs;
        G.msg_end = (uint32_t)(msgs += count[g]);
        G.blocks = blocks[g];
        const uint64_t gt = (blocks[g] + tile_blocks - 1) / tile_blocks;
        // headroom: warps read the counter past the last tile, offset by the fixed first tiles
        if (tiles + gt > 0xFFFF0000u) return fail(AES_ERR_ARG, "batch needs too many tiles");
        G.tile_start = (uint32_t)tiles;
        G.tile_end = (uint32_t)(tiles += gt);
        P->total_blocks += blocks[g];
        blocks[g] = 0;  // from here: blocks of the messages placed
    }
    P->ntiles = (uint32_t)tiles;
    P->msgs.resize(msgs);
    for (size_t i = 0; i < nmsg; ++i) {
        const int g = group[i];
        if (g == kGroups) continue;
        const aes_msg_desc& m = d[i];
        P->msgs[next[g]++] = MsgDev{blocks[g], m.in_off >> 4, m.out_off >> 4, 2u * m.key_index + m.decrypt, (uint32_t)i};
        blocks[g] += m.nblocks;
    }
    P->tile_msg.resize(tiles);
    for (const GroupDev& G : P->groups) {  // first message of each tile: walk the group's messages once
        uint32_t m = G.msg_start;
        uint64_t first = 0;
        for (uint32_t t = G.tile_start; t < G.tile_end; ++t, first += tile_blocks) {
            while (m + 1 < G.msg_end && P->msgs[m + 1].blk_start <= first) ++m;
            P->tile_msg[t] = m;
        }
    }
    return AES_OK;
}

}  // namespace gbaes

using namespace gbaes;

struct aes_batch_plan {
    uint32_t magic;
    int device;
    int threads, bpt;
    HostPlan host;
    uint8_t* dev_buf;
    size_t dev_bytes;
    BatchArgs args;  // device pointers and schedule filled in; in/out set per launch
    uint32_t grid;
    bool joined;
    cudaGraphExec_t graph_exec;
    cudaGraph_t graph;
    cudaGraphNode_t kernel_node;
    cudaStream_t capture_stream;
    std::mutex mu;
};

namespace gbaes {

constexpr uint32_t kPlanMagic = 0x504c414eu;  // "PLAN"

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// The device tables of a plan, in one piece: the counter (256 bytes), two
// schedules per context, the messages, the tiles.
struct Tables {
    static constexpr size_t off_keys = 256;
    size_t off_msgs, off_tiles, bytes;
    Tables(const HostPlan& H, size_t nctx) {
        off_msgs = off_keys + nctx * 2 * kSlotWords * 4;
        off_tiles = off_msgs + align256(H.msgs.size() * sizeof(MsgDev));
        bytes = off_tiles + align256(H.tile_msg.size() * 4 + 4);
    }
    // Their host copy (bytes long).
    std::unique_ptr<uint8_t[]> image(const HostPlan& H, const aes_ctx* const* ctxs, size_t nctx) const {
        std::unique_ptr<uint8_t[]> img(new uint8_t[bytes]);
        memset(img.get(), 0, off_keys);
        for (size_t i = 0; i < nctx; ++i) {
            const size_t n = 16 * (size_t)(ctxs[i]->nr + 1), slot = 4 * kSlotWords;
            uint8_t* p = img.get() + off_keys + 2 * i * slot;
            memcpy(p, ctxs[i]->enc_rk, n);
            memset(p + n, 0, slot - n);
            memcpy(p + slot, ctxs[i]->dec_rk, n);
            memset(p + slot + n, 0, slot - n);
        }
        put(img.get(), off_msgs, off_tiles, H.msgs.data(), H.msgs.size() * sizeof(MsgDev));
        put(img.get(), off_tiles, bytes, H.tile_msg.data(), H.tile_msg.size() * 4);
        return img;
    }
    // Points a launch's arguments at the tables at dev.
    void fill_args(const HostPlan& H, uint8_t* dev, BatchArgs* a) const {
        a->msgs = (const MsgDev*)(dev + off_msgs);
        a->keys = (const uint4*)(dev + off_keys);
        a->tile_msg = (const uint32_t*)(dev + off_tiles);
        a->counter = (unsigned*)dev;
        a->ntiles = H.ntiles;
        a->tile_blocks = H.tile_blocks;
        memcpy(a->groups, H.groups, sizeof a->groups);
    }

  private:
    static void put(uint8_t* img, size_t from, size_t to, const void* src, size_t n) {
        if (n) memcpy(img + from, src, n);
        memset(img + from + n, 0, to - from - n);
    }
};

using BatchKernel = void (*)(const BatchArgs);

static BatchKernel pick_batch(int bpt, bool joined = false) {
    switch (bpt) {
        case 1: return batch_kernel<1, false>;
        case 2: return joined ? batch_kernel<2, true> : batch_kernel<2, false>;
        case 4: return batch_kernel<4, false>;
        case 8: return joined ? batch_kernel<8, true> : batch_kernel<8, false>;  // (512 threads at most: 128 registers)
        default: return nullptr;
    }
}


static int check_bases(const HostPlan& H, const void* in_base, size_t in_bytes, const void* out_base,
                       size_t out_bytes) {
    if (in_bytes < H.in_extent || out_bytes < H.out_extent)
        return fail(AES_ERR_ARG, "buffers (%zu in, %zu out bytes) are smaller than the messages need (%llu, %llu)",
                    in_bytes, out_bytes, (unsigned long long)H.in_extent, (unsigned long long)H.out_extent);
    if (H.ntiles) {
        int rc = check_device_range(in_base, H.in_extent, "in_base");
        if (rc) return rc;
        rc = check_device_range(out_base, H.out_extent, "out_base");
        if (rc) return rc;
    }
    return AES_OK;
}

static int plan_launch_args(aes_batch_plan* P, const void* in_base, size_t in_bytes, void* out_base,
                            size_t out_bytes, BatchArgs* a) {
    if (!P || P->magic != kPlanMagic) return fail(AES_ERR_ARG, "invalid aes_batch_plan");
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != P->device)
        return fail(AES_ERR_ARG, "plan was built on device %d, current device is %d", P->device, dev);
    int rc = check_bases(P->host, in_base, in_bytes, out_base, out_bytes);
    if (rc) return rc;
    *a = P->args;
    a->in = (const uint4*)in_base;
    a->out = (uint4*)out_base;
    return AES_OK;
}

// A batch with fewer than kTilesPerWarp tiles for every warp has its tiles cut
// into parts, down to one pass of a warp, until there are kPartsPerWarp of them per
// warp.  A larger one keeps whole tiles (fewer unit starts) but for the last ones
// of every warp, cut the same way, so that the SMs end together: 85 MB
// 131.0 -> 123.7 us (1024 x 2), 291 MB 399.5 -> 392.8 (512 x 8), 849 MB 1,103.4 -> 1,097.4,
// 3.4 GB 4,293 -> 4,288.  Cutting every tile instead gives 126-129 at 85 MB and 403.6 at
// 291 MB (1024 x 2), the unit starts costing what the even end gains.
//
// Whole tiles are then taken 2^join at a time, as long as that leaves kTilesPerWarp
// units per warp, up to kJoinMax blocks and a kJoinPerMsg-th of the mean message
// (messages up to 4 MiB, 512 x 8: 3.37 GB 4,285 us with tiles of 512 blocks one at a
// time, 4,246 with 1,024 blocks, 4,234 with 2,048, 4,230 with 4,096; 10,000 messages up
// to 256 KiB, 1,700 blocks on average, 271 MB: 382 with 512, 398 with 1,024, 455 with 2,048;
// here and below as measured before crossing passes ran 4 blocks at a time).
constexpr uint64_t kTilesPerWarp = 4;
constexpr uint64_t kPartsPerWarp = 8;
constexpr uint64_t kJoinMax = 2048;  // blocks
constexpr uint64_t kJoinPerMsg = 4;

// The kernel for whole tiles runs each pass of a unit by itself: in a unit that
// messages start in, the passes without a start keep to one message's keys.  It pays
// where units have several passes: 512 x 8, 10,000 messages up to 128 KiB (146 MB)
// 259 -> 242 us, up to 256 KiB 398 -> 382, up to 1 MiB 1,234 -> 1,218.  With 2 blocks
// per thread (146 MB: 207.0 -> 204.6) it costs 0.6% where few units cross (250
// messages up to 4 MiB, 92 MB: 128.1 -> 128.9), so there it wants joined tiles or a
// mean message below kShortTiles tiles; with 4 it would spill.  In launches of cut
// tiles it costs 0.5-4%.
constexpr uint64_t kShortTiles = 16;

BatchSchedule schedule_batch(const HostPlan& H, int threads, int bpt, int sms) {
    BatchSchedule s{};
    const uint64_t warps = (uint64_t)threads / 32 * (uint64_t)sms;
    const uint32_t pass = 32u * (uint32_t)bpt;
    if (H.ntiles >= kTilesPerWarp * warps) {
        if (bpt == 2 || bpt == 8) {
            const uint64_t mean = H.total_blocks / H.msgs.size(), most = std::min(kJoinMax, mean / kJoinPerMsg);
            while (H.ntiles >= (kTilesPerWarp * warps << (s.join + 1)) && H.ntiles < 1u << 30 &&
                   (uint64_t)H.tile_blocks << (s.join + 1) <= most)
                ++s.join;
            s.joined = (uint64_t)H.tile_blocks << s.join > pass &&
                       (bpt == 8 || s.join || mean < kShortTiles * H.tile_blocks);
        }
        s.whole = (uint32_t)(H.ntiles - (warps << s.join)) >> s.join << s.join;
    }
    const uint64_t cut = H.ntiles - s.whole;
    while ((cut << s.split) < kPartsPerWarp * warps && (H.tile_blocks >> s.split) % (2u * pass) == 0) ++s.split;
    const uint64_t units = (s.whole >> s.join) + (cut << s.split);
    s.grid = (uint32_t)std::min<uint64_t>(units, (uint64_t)sms);
    s.counted = units > (uint64_t)s.grid * ((uint64_t)threads / 32);
    return s;
}

static BatchSchedule current_schedule(const HostPlan& H, int threads, int bpt) {
    DeviceInfo info;
    return schedule_batch(H, threads, bpt, current_device_info(&info) ? 1 : info.sms);
}

int launch_batch_kernel(const HostPlan& H, BatchArgs a, int threads, int bpt, cudaStream_t stream) {
    if (!pick_batch(bpt)) return fail(AES_ERR_ARG, "blocks_per_thread %d: need 1, 2, 4 or 8", bpt);
    if (bpt == 8 && threads > 512) return fail(AES_ERR_ARG, "8 blocks per thread need threads <= 512");
    const BatchSchedule sch = current_schedule(H, threads, bpt);
    const BatchKernel fn = pick_batch(bpt, sch.joined);
    int rc = set_max_dynamic_smem((const void*)fn, (int)kBatchSmem);
    if (rc) return rc;
    a.whole = sch.whole;
    a.join = sch.join;
    a.split = sch.split;
    if (!sch.counted) a.counter = nullptr;
    const cudaError_t e = launch_overlapped(fn, sch.grid, (unsigned)threads, kBatchSmem, stream, a);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "batch kernel launch: %s", cudaGetErrorString(e));
    return AES_OK;
}

// Largest tile of a call that plans for one launch, in blocks.
constexpr uint32_t kOneShotTileMax = 2048;

// Tiles of 512 blocks, which above 2^23 blocks would only lengthen the upload.
static uint32_t one_shot_tile(const aes_msg_desc* d, size_t nmsg) {
    uint64_t total = 0;
    if (nmsg > kMaxMessages) nmsg = 0;  // (build_host_plan refuses the count before it reads a message)
    for (size_t i = 0; d && i < nmsg; ++i) total += std::min<uint64_t>(d[i].nblocks, 1ull << 32);
    return total <= 1u << 23 ? 512 : kOneShotTileMax;
}

// A launch whose shape the caller left open runs 1024 threads x 2 blocks, or 512 x 8:
// there a warp reads each round's key for 8 states instead of 2 (4 cycles of the L1
// data stage per read, beside 16 per state), which counts from kWideBlocks on, once
// unit starts and tails do not; but a message that starts inside a pass makes all 256
// blocks of it, not 64, read keys for each state.  512 x 8
// over 1024 x 2, kept plans of 190-910 MB, by the share of such passes: 0.8% 0.961-1.000,
// 2.5% 0.970-0.990, 4.5% 0.977-1.000 (messages up to 512 KiB), 8% 0.984-1.011 (up to 256 KiB),
// 14% 0.999-1.030, 23% 1.019-1.055, 60% 1.07-1.10 (up to 16 KiB).  By size,
// messages up to 4 MiB: 42.5 us with 1024 x 2 and 44.7 with 512 x 8 at 24 MB, 124 / 124 at
// 89 MB, 213 / 210 at 149 MB, 315 / 305 at 231 MB, 1,218 / 1,175 at 918 MB, 4,395 / 4,235 at 3.4 GB.
constexpr uint64_t kWideBlocks = 3ull << 22;
constexpr uint64_t kWidePass = 256;     // blocks of a warp's pass with 8 blocks per thread
constexpr uint64_t kWideCrossed = 12;  // at most one pass in this many crossed

struct Shape {
    int threads, bpt;
};

static Shape open_shape(const HostPlan& H) {
    const Shape narrow{1024, 2}, wide{512, 8};
    if (H.total_blocks < kWideBlocks) return narrow;
    uint64_t left = H.total_blocks / kWidePass / kWideCrossed;
    for (const GroupDev& G : H.groups) {
        uint64_t last = UINT64_MAX;  // the pass that was counted last
        for (uint32_t m = G.msg_start; m < G.msg_end; ++m) {
            const uint64_t start = H.msgs[m].blk_start;
            if (start % kWidePass == 0 || start / kWidePass == last) continue;
            if (left-- == 0) return narrow;
            last = start / kWidePass;
        }
    }
    return wide;
}

}  // namespace gbaes

extern "C" {

aes_batch_plan* aes_batch_plan_create(const aes_msg_desc* msgs, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx,
                                      int threads, int blocks_per_thread) {
    const bool open = threads == 0 && blocks_per_thread == 0;
    if (threads == 0) threads = 1024;
    if (blocks_per_thread == 0) blocks_per_thread = 2;
    if (threads < 64 || threads > 1024 || threads % 32) {
        fail(AES_ERR_ARG, "threads %d: need a multiple of 32 in [64, 1024]", threads);
        return nullptr;
    }
    if (!pick_batch(blocks_per_thread)) {
        fail(AES_ERR_ARG, "blocks_per_thread %d: need 1, 2, 4 or 8", blocks_per_thread);
        return nullptr;
    }
    if (blocks_per_thread == 8 && threads > 512) {
        fail(AES_ERR_ARG, "8 blocks per thread need threads <= 512 (128 registers per thread)");
        return nullptr;
    }
    aes_batch_plan* P = new (std::nothrow) aes_batch_plan();
    if (!P) {
        fail(AES_ERR_NOMEM, "out of host memory");
        return nullptr;
    }
    P->threads = threads;
    P->bpt = blocks_per_thread;
    // Tiles of 128*BPT blocks, at most 512.  A batch of 10,000 messages (16 B - 4 MiB, log-uniform) ran at
    // 0.8847 of its lookup roofline with 1,024-block tiles at 8 blocks per thread and at 0.8878 with 512
    // (less work left over in the last wave); at 4 blocks per thread 256-block tiles lost (0.8705 against
    // 0.8745 at 512).
    const uint32_t tile_blocks = std::min(128u * (uint32_t)blocks_per_thread, kPlanTileMax);
    if (build_host_plan(msgs, nmsg, ctxs, nctx, tile_blocks, &P->host)) {
        delete P;
        return nullptr;
    }
    if (open) {  // (the tiles stay 1024 x 2's)
        const Shape shape = open_shape(P->host);
        P->threads = shape.threads;
        P->bpt = shape.bpt;
    }
    if (cudaGetDevice(&P->device) != cudaSuccess) {
        fail(AES_ERR_CUDA, "no CUDA device");
        delete P;
        return nullptr;
    }
    const HostPlan& H = P->host;
    const Tables tables(H, nctx);
    P->dev_bytes = tables.bytes;
    cudaError_t e = cudaMalloc(&P->dev_buf, P->dev_bytes);
    if (e != cudaSuccess) {
        fail(AES_ERR_NOMEM, "cudaMalloc(%zu): %s", P->dev_bytes, cudaGetErrorString(e));
        delete P;
        return nullptr;
    }
    e = cudaMemcpy(P->dev_buf, tables.image(H, ctxs, nctx).get(), P->dev_bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        fail(AES_ERR_CUDA, "uploading the batch plan: %s", cudaGetErrorString(e));
        cudaFree(P->dev_buf);
        delete P;
        return nullptr;
    }
    BatchArgs& a = P->args;
    memset(&a, 0, sizeof a);
    tables.fill_args(H, P->dev_buf, &a);
    if (H.ntiles) {
        const BatchSchedule sch = current_schedule(H, P->threads, P->bpt);
        a.whole = sch.whole;
        a.join = sch.join;
        a.split = sch.split;
        if (!sch.counted) a.counter = nullptr;
        P->grid = sch.grid;
        P->joined = sch.joined;
    }
    P->magic = kPlanMagic;
    return P;
}

int aes_batch_plan_launch(aes_batch_plan* P, const void* in_base, size_t in_bytes, void* out_base, size_t out_bytes,
                          void* stream) {
    BatchArgs a;
    int rc = plan_launch_args(P, in_base, in_bytes, out_base, out_bytes, &a);
    if (rc) return rc;
    if (P->host.ntiles == 0) return AES_OK;
    BatchKernel fn = pick_batch(P->bpt, P->joined);
    rc = set_max_dynamic_smem((const void*)fn, (int)kBatchSmem);
    if (rc) return rc;
    const cudaError_t e = launch_overlapped(fn, P->grid, (unsigned)P->threads, kBatchSmem, (cudaStream_t)stream, a);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "batch kernel launch: %s", cudaGetErrorString(e));
    return AES_OK;
}

int aes_batch_plan_launch_graph(aes_batch_plan* P, const void* in_base, size_t in_bytes, void* out_base,
                                size_t out_bytes, void* stream) {
    BatchArgs a;
    int rc = plan_launch_args(P, in_base, in_bytes, out_base, out_bytes, &a);
    if (rc) return rc;
    if (P->host.ntiles == 0) return AES_OK;
    std::lock_guard<std::mutex> lk(P->mu);
    BatchKernel fn = pick_batch(P->bpt, P->joined);
    rc = set_max_dynamic_smem((const void*)fn, (int)kBatchSmem);
    if (rc) return rc;
    cudaError_t e = cudaSuccess;
    if (!P->graph_exec) {
        if (!P->capture_stream) {
            e = cudaStreamCreateWithFlags(&P->capture_stream, cudaStreamNonBlocking);
            if (e != cudaSuccess) return fail(AES_ERR_CUDA, "capture stream: %s", cudaGetErrorString(e));
        }
        e = cudaStreamBeginCapture(P->capture_stream, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            fn<<<P->grid, P->threads, kBatchSmem, P->capture_stream>>>(a);
            e = cudaStreamEndCapture(P->capture_stream, &P->graph);
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&P->graph_exec, P->graph, 0);
        if (e == cudaSuccess) {
            size_t n = 0;
            cudaGraphGetNodes(P->graph, nullptr, &n);
            std::vector<cudaGraphNode_t> nodes(n);
            cudaGraphGetNodes(P->graph, nodes.data(), &n);
            for (auto node : nodes) {
                cudaGraphNodeType ty;
                if (cudaGraphNodeGetType(node, &ty) == cudaSuccess && ty == cudaGraphNodeTypeKernel)
                    P->kernel_node = node;
            }
        }
        if (e != cudaSuccess || !P->kernel_node) {
            cudaGetLastError();
            return fail(AES_ERR_CUDA, "capturing the batch graph: %s", cudaGetErrorString(e));
        }
    } else {
        void* params[1] = {&a};
        cudaKernelNodeParams kp;
        memset(&kp, 0, sizeof kp);
        kp.func = (void*)fn;
        kp.gridDim = dim3(P->grid);
        kp.blockDim = dim3(P->threads);
        kp.sharedMemBytes = kBatchSmem;
        kp.kernelParams = params;
        e = cudaGraphExecKernelNodeSetParams(P->graph_exec, P->kernel_node, &kp);
        if (e != cudaSuccess) return fail(AES_ERR_CUDA, "updating the batch graph: %s", cudaGetErrorString(e));
    }
    e = cudaGraphLaunch(P->graph_exec, (cudaStream_t)stream);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "graph launch: %s", cudaGetErrorString(e));
    return AES_OK;
}

int aes_batch_plan_info(const aes_batch_plan* P, uint64_t* total_blocks, uint32_t* ntiles, uint32_t* tile_blocks) {
    if (!P || P->magic != kPlanMagic) return fail(AES_ERR_ARG, "invalid aes_batch_plan");
    if (total_blocks) *total_blocks = P->host.total_blocks;
    if (ntiles) *ntiles = P->host.ntiles;
    if (tile_blocks) *tile_blocks = P->host.tile_blocks;
    return AES_OK;
}

void aes_batch_plan_free(aes_batch_plan* P) {
    if (!P || P->magic != kPlanMagic) return;
    P->magic = 0;
    if (P->graph_exec) cudaGraphExecDestroy(P->graph_exec);
    if (P->graph) cudaGraphDestroy(P->graph);
    if (P->capture_stream) cudaStreamDestroy(P->capture_stream);
    cudaFree(P->dev_buf);
    delete P;
}

int aes_ecb_batch(const aes_msg_desc* msgs, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx, const void* in_base,
                  size_t in_bytes, void* out_base, size_t out_bytes, void* stream) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing((cudaStream_t)stream, &cap);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "cudaStreamIsCapturing: %s", cudaGetErrorString(e));
    if (cap != cudaStreamCaptureStatusNone)
        return fail(AES_ERR_STATE,
                    "aes_ecb_batch uploads from host memory freed on return and cannot be captured; "
                    "use aes_batch_plan_launch_graph");
    HostPlan H;
    int rc = build_host_plan(msgs, nmsg, ctxs, nctx, one_shot_tile(msgs, nmsg), &H);
    if (rc) return rc;
    if (H.ntiles == 0) return AES_OK;
    rc = check_bases(H, in_base, in_bytes, out_base, out_bytes);
    if (rc) return rc;
    // Stream-ordered scratch: plan tables live only as long as the launch.
    cudaStream_t s = (cudaStream_t)stream;
    const Tables tables(H, nctx);
    uint8_t* buf = nullptr;
    e = cudaMallocAsync((void**)&buf, tables.bytes, s);
    if (e != cudaSuccess) return fail(AES_ERR_NOMEM, "cudaMallocAsync(%zu): %s", tables.bytes, cudaGetErrorString(e));
    const auto img = tables.image(H, ctxs, nctx);
    e = cudaMemcpyAsync(buf, img.get(), tables.bytes, cudaMemcpyHostToDevice, s);  // pageable: staged before return
    if (e != cudaSuccess) {
        cudaFreeAsync(buf, s);
        return fail(AES_ERR_CUDA, "uploading the batch tables: %s", cudaGetErrorString(e));
    }
    BatchArgs a;
    memset(&a, 0, sizeof a);
    a.in = (const uint4*)in_base;
    a.out = (uint4*)out_base;
    tables.fill_args(H, buf, &a);
    const Shape shape = open_shape(H);
    rc = launch_batch_kernel(H, a, shape.threads, shape.bpt, s);
    cudaFreeAsync(buf, s);
    return rc;
}

int aes_batch_tiles(const aes_msg_desc* msgs, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx, int tile_blocks,
                    uint32_t* first_msg, size_t cap) {
    if (tile_blocks <= 0) return fail(AES_ERR_ARG, "tile_blocks must be positive");
    HostPlan H;
    int rc = build_host_plan(msgs, nmsg, ctxs, nctx, (uint32_t)tile_blocks, &H);
    if (rc) return rc;
    if (first_msg) {
        if (cap < H.ntiles) return fail(AES_ERR_ARG, "first_msg holds %zu entries, the batch has %u tiles", cap, H.ntiles);
        for (uint32_t t = 0; t < H.ntiles; ++t) first_msg[t] = H.msgs[H.tile_msg[t]].src;
    }
    return (int)std::min<uint32_t>(H.ntiles, 0x7FFFFFFF);
}

}  // extern "C"

// ------------------------------------------------ batch without allocation
//
// Some callers cannot call cudaMalloc: code whose device memory is owned by
// another runtime or allocator (a cudaMalloc behind its back breaks its
// accounting, or fails once it has reserved the device), and latency-critical
// paths that must not pay an allocation's synchronisation or unbounded cost.
// aes_ecb_batch_noalloc serves them: it runs the same batched kernel as
// aes_ecb_batch, but its plan tables and tile counter live in the fixed array
// below, which every GPU that loads this library holds until the process exits.

namespace gbaes {

constexpr size_t kNoAllocScratchBytes = (size_t)8 << 20;  // 8 MiB

static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocScratchBytes];

static std::mutex g_noalloc_mu;
static std::vector<std::pair<unsigned long long, uint8_t*>> g_noalloc_addr;  // (context id, device address)

// Device address of g_noalloc_scratch in the current context.  Host code must
// not pass the array's own name to a kernel: on the host that name denotes a
// host-side stand-in, not device memory.  The address belongs to the module
// loaded in one CUDA context, so it is looked up (cudaGetSymbolAddress, with
// that context current) on the first call in each context -- normally once per
// device, in its primary context -- and cached under the context's id.
static int noalloc_scratch(uint8_t** out) {
    unsigned long long ctx = 0;
    int rc = current_context_id(&ctx);
    if (rc) return rc;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    for (const auto& e : g_noalloc_addr)
        if (e.first == ctx) {
            *out = e.second;
            return AES_OK;
        }
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) return fail(AES_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
    g_noalloc_addr.emplace_back(ctx, (uint8_t*)p);
    *out = (uint8_t*)p;
    return AES_OK;
}

}  // namespace gbaes

extern "C" {

int aes_ecb_batch_noalloc(const aes_msg_desc* msgs, size_t nmsg, const aes_ctx* const* ctxs, size_t nctx,
                          const void* in_base, size_t in_bytes, void* out_base, size_t out_bytes, void* stream) {
    HostPlan H;
    int rc = build_host_plan(msgs, nmsg, ctxs, nctx, one_shot_tile(msgs, nmsg), &H);
    if (rc) return rc;
    if (Tables(H, nctx).bytes > kNoAllocScratchBytes && H.tile_blocks != kOneShotTileMax) {
        H = HostPlan();
        rc = build_host_plan(msgs, nmsg, ctxs, nctx, kOneShotTileMax, &H);  // the smallest tables
        if (rc) return rc;
    }
    if (H.ntiles == 0) return AES_OK;
    rc = check_bases(H, in_base, in_bytes, out_base, out_bytes);
    if (rc) return rc;
    const Tables tables(H, nctx);
    if (tables.bytes > kNoAllocScratchBytes)
        return fail(AES_ERR_ARG,
                    "batch needs %zu bytes of tables (keys: 512 B per context; 32 B per message; 4 B per tile), "
                    "the allocation-free entry point holds at most %zu",
                    tables.bytes, kNoAllocScratchBytes);
    uint8_t* buf = nullptr;
    rc = noalloc_scratch(&buf);
    if (rc) return rc;
    const auto img = tables.image(H, ctxs, nctx);  // host staging only; the counter words are zero
    cudaStream_t s = (cudaStream_t)stream;
    // Stream-ordered after earlier work on `stream`; from pageable memory the
    // call returns once the image is staged, so img may be released after it.
    cudaError_t e = cudaMemcpyAsync(buf, img.get(), tables.bytes, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "uploading the batch tables: %s", cudaGetErrorString(e));
    BatchArgs a;
    memset(&a, 0, sizeof a);
    a.in = (const uint4*)in_base;
    a.out = (uint4*)out_base;
    tables.fill_args(H, buf, &a);
    const Shape shape = open_shape(H);
    return launch_batch_kernel(H, a, shape.threads, shape.bpt, s);
}

}  // extern "C"
