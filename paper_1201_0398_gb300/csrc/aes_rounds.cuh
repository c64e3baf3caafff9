// Device-side AES rounds in the T-table form of Eq. 1, shared by every table
// kernel.
//
// Shared-memory layout: one table per direction, 32 KiB.  Entry x of T_0 is stored
// 32 times side by side (128 bytes at 128 x); lane l reads copy l, so lane l always
// hits the same bank whatever byte it looks up.  The other three tables of Eq. 1
// are rotations, T_k[x] = rotl(T_0[x], 8k), and cost one byte permute of the
// entry read.
//
// A lookup address is one dp4a: byte k of a state word times 128 plus the lane's
// base, the other three bytes times 0.  dp4a runs on the multiply-add pipe at the
// ALU's rate (64 lanes/clk/SM), beside it: dp4a and lop3 in turn issue 3.63 warp
// instructions per clock and SM, prmt and lop3 1.99.  A round of a warp is 16
// lookups (16 clocks of the shared-memory pipe, the bound), 16 dp4a (8 clocks), and
// 12 permutes and 8 three-input XORs (10 clocks of the ALU).
//
// Measured, AES-128, 1 GiB, cycles of an SM per 32 blocks (160 are lookups):
//   four tables of 32 KiB, PRMT addresses (64 KiB aligned)   177  (909 GB/s)
//   the same with dp4a addresses                             177
//   four tables at the start of the shared-memory window     172
//   one table, two CTAs of 512 threads per SM                172  (937 GB/s)
//   one table 128 KiB into the window                        179
// The global loads and stores (about 12 of the 172) share the L1 data stage with the
// lookups, and tables far into the window get more in their way.  One table is also
// a quarter of the fill (256 store cycles instead of 1,024), lets two CTAs share an
// SM, and leaves room for both directions' tables at once.
#pragma once

#include <cstdint>

#include "aes_tables.h"
#include "gbaes_internal.h"

namespace gbaes {

// Source of the shared-memory fills, read through the read-only global path.
static __device__ AesTables g_tab = make_aes_tables();

constexpr uint32_t kTableBytes = 0x8000u;  // 256 entries x 32 lanes x 4 B

__device__ __forceinline__ uint32_t lds(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

template <uint32_t OFF>
__device__ __forceinline__ uint32_t lds_off(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}

__device__ __forceinline__ void sts(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// 16-byte input loads, read once (not kept in L1) or read again soon.  Not .nc: a
// kernel may start while the one that writes its input still runs (launch.cuh), and
// only the coherent path is bound to see those writes after the wait.  Volatile, so
// that a load meant to go out before the rounds stays there.
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ uint4 ld_keep(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint32_t smem_base(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Fill store: ordered before the table's first use by the barrier that follows
// every fill, so it needs no compiler memory clobber (which would keep the next
// entry's global load from being issued early).
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(v));
}

// Writes one direction's table at A (16-byte aligned); threads tid = 0..nt-1 take
// part and the caller synchronises them.  Four threads share an entry's 128 bytes:
// piece p in 0..1023 is two of the eight 16-byte parts of entry p / 4, rotated so
// that the 8 threads of a quarter-warp's store hit 8 different bank groups.  A thread
// loads the entries of up to kFillChunk pieces (p0 and every nt after it) before
// storing any.
constexpr uint32_t kFillPieces = 1024, kFillChunk = 4;

__device__ __forceinline__ void fill_load(bool decrypt, uint32_t p0, uint32_t nt, uint32_t (&v)[kFillChunk]) {
    const uint32_t* t0 = decrypt ? g_tab.td0 : g_tab.te0;
#pragma unroll
    for (uint32_t u = 0; u < kFillChunk; ++u) {
        const uint32_t p = p0 + u * nt;
        v[u] = 0u;
        // (volatile: issued here, ahead of what stands between this and fill_store)
        if (p < kFillPieces) asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v[u]) : "l"(t0 + (p >> 2)));
    }
}

__device__ __forceinline__ void fill_store(uint32_t A, uint32_t p0, uint32_t nt, const uint32_t (&v)[kFillChunk]) {
#pragma unroll
    for (uint32_t u = 0; u < kFillChunk; ++u) {
        const uint32_t p = p0 + u * nt;
        if (p < kFillPieces) {
            const uint32_t part = 2u * (p & 3u) + ((p >> 2) & 1u);
            const uint32_t base = A + (p >> 2) * 128u;
            sts128(base + 16u * part, v[u]);
            sts128(base + 16u * (part ^ 1u), v[u]);
        }
    }
}

__device__ __forceinline__ void fill_table(uint32_t A, bool decrypt, uint32_t tid, uint32_t nt) {
    for (uint32_t p = tid; p < kFillPieces; p += kFillChunk * nt) {
        uint32_t v[kFillChunk];
        fill_load(decrypt, p, nt, v);
        fill_store(A, p, nt, v);
    }
}

// Entry [byte K of w] of T_0 for the lane whose base is L = A + 4 * lane.
template <int K>
__device__ __forceinline__ uint32_t look(uint32_t w, uint32_t L) {
    return lds(__dp4a(w, 0x80u << (8 * K), L));
}

// Rotation of an entry left by K bytes: T_0's entry as T_K's.
template <int K>
__device__ __forceinline__ uint32_t as_table(uint32_t v) {
    return K == 0 ? v : __byte_perm(v, v, K == 1 ? 0x2103u : K == 2 ? 0x1032u : 0x0321u);
}

// (a & m) | (b & ~m): bytes of a where m is set, of b elsewhere.
__device__ __forceinline__ uint32_t merge(uint32_t a, uint32_t b, uint32_t m) { return (a & m) | (b & ~m); }

// One inner round (Eq. 1): the word that gives byte k of output word j is I_{j+k,k},
// for the inverse cipher I_{j-k,k}.
template <bool DECRYPT>
__device__ __forceinline__ void round_inner(uint32_t (&s)[4], uint32_t L, uint4 k) {
    constexpr int D = DECRYPT ? 3 : 1;
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        t[j] = as_table<0>(look<0>(s[j], L)) ^ as_table<1>(look<1>(s[(j + D) & 3], L)) ^
               as_table<2>(look<2>(s[(j + 2) & 3], L)) ^ as_table<3>(look<3>(s[(j + 3 * D) & 3], L)) ^ kk[j];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

// Last round: SubBytes + ShiftRows + AddRoundKey.  S[x] is bytes 1 and 2 of Te0's
// entry (02 S, S, S, 03 S).  Of Td0's entry (0e Si, 09 Si, 0d Si, 0b Si) the four
// bytes XOR to Si, as 0e ^ 09 ^ 0d ^ 0b = 01: the inverse S-box needs no table.
template <bool DECRYPT>
__device__ __forceinline__ void round_last(uint32_t (&s)[4], uint32_t L, uint4 k) {
    constexpr int D = DECRYPT ? 3 : 1;
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t e0 = look<0>(s[j], L), e1 = look<1>(s[(j + D) & 3], L);
        const uint32_t e2 = look<2>(s[(j + 2) & 3], L), e3 = look<3>(s[(j + 3 * D) & 3], L);
        if (DECRYPT) {  // byte k: the XOR of e_k's bytes
            const uint32_t x = __byte_perm(e0, e1, 0x5410u) ^ __byte_perm(e0, e1, 0x7632u);
            const uint32_t y = __byte_perm(e2, e3, 0x5410u) ^ __byte_perm(e2, e3, 0x7632u);
            t[j] = __byte_perm(x, y, 0x6420u) ^ __byte_perm(x, y, 0x7531u) ^ kk[j];
        } else {  // byte 1 of e0, e1 and byte 2 of e2, e3 (e1's and e2's are in place)
            t[j] = merge(merge(e1, e2, 0x0000ffffu), __byte_perm(e0, e3, 0x6001u), 0x00ffff00u) ^ kk[j];
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

// Round keys from the kernel parameters (uniform constant-bank operands).
struct ParamKeys {
    const uint32_t (&rk)[60];
    __device__ __forceinline__ uint4 get(int r) const {
        return make_uint4(rk[4 * r], rk[4 * r + 1], rk[4 * r + 2], rk[4 * r + 3]);
    }
};

template <int BPT, class KS>
__device__ __forceinline__ void whiten(uint32_t (&s)[BPT][4], const KS& ks) {
    const uint4 k = ks.get(0);
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        s[b][0] ^= k.x;
        s[b][1] ^= k.y;
        s[b][2] ^= k.z;
        s[b][3] ^= k.w;
    }
}

// Rounds FIRST..NR (after the whitening) on BPT independent states sharing one
// schedule, UNROLL rounds per iteration: unrolled in full (UNROLL >= NR) the round
// keys are constant operands of the XORs, rolled they are loads.
template <int NR, bool DECRYPT, int FIRST, int BPT, int UNROLL, class KS>
__device__ __forceinline__ void rounds_from(uint32_t (&s)[BPT][4], const KS& ks, uint32_t L) {
#pragma unroll UNROLL
    for (int r = FIRST; r < NR; ++r) {
        const uint4 k = ks.get(r);
#pragma unroll
        for (int b = 0; b < BPT; ++b) round_inner<DECRYPT>(s[b], L, k);
    }
    const uint4 k = ks.get(NR);
#pragma unroll
    for (int b = 0; b < BPT; ++b) round_last<DECRYPT>(s[b], L, k);
}

}  // namespace gbaes
