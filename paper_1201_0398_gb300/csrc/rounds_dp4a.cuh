// Eq. 1's rounds with lookup addresses from byte dot products.
//
// The layout of aes_rounds.cuh takes one PRMT per lookup address, on the integer
// ALU, beside the XORs.  Here an address is one dp4a: byte k of a state word times
// 128 plus the lane's base, the other three bytes times 0.  dp4a runs at the
// ALU's rate (64 lanes/clk/SM) on the multiply-add pipe, so a round leaves the
// ALU with the XORs alone (8 of 24 instructions), free for other warps.
// Measured on the GB300: dp4a and lop3 in turn issue 3.63 warp instructions per
// clock and SM, prmt and lop3 1.99; the rounds alone take 160.5 cycles per 32
// blocks of AES-128 either way (160 is the lookups' bound).
//
// Tables: T_k at A + 32 KiB * k, entry x at 128 x, its 32 lane copies side by
// side, so lane l always hits the same bank; the inverse S-box follows as a fifth
// table.  The factor 128 fits dp4a's bytes, the table is the load's immediate
// offset, and A needs no alignment beyond 16 bytes.
#pragma once

#include "aes_rounds.cuh"

namespace gbaes {
namespace dp {

constexpr uint32_t kTable = 0x8000u;  // 256 entries x 32 lanes x 4 B
constexpr uint32_t kEncBytes = 4 * kTable;
constexpr uint32_t kDecBytes = 5 * kTable;

// Writes one direction's tables at A; the CTA's THREADS threads take part and the
// caller synchronises them.  Pair p = (entry p/4, table p%4): 128 contiguous
// bytes, stored 16 at a time in an order rotated by p, so that 8 neighbouring
// threads hit 8 different bank groups.
template <int THREADS, bool DECRYPT>
__device__ __forceinline__ void fill_tables(uint32_t A) {
    constexpr int N = 1024 / THREADS, NS = DECRYPT ? (256 + THREADS - 1) / THREADS : 0;
    static_assert(1024 % THREADS == 0, "pairs per thread");
    const uint32_t* t0 = DECRYPT ? g_tab.td0 : g_tab.te0;
    uint32_t v[N + NS];  // every entry's load goes out before the first store
#pragma unroll
    for (int u = 0; u < N; ++u) v[u] = __ldg(t0 + ((threadIdx.x + u * THREADS) >> 2));
#pragma unroll
    for (int u = 0; u < NS; ++u) v[N + u] = __ldg(g_tab.si4 + ((threadIdx.x + u * THREADS) & 255u));
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const uint32_t p = threadIdx.x + u * THREADS;
        const uint32_t k = p & 3u;
        const uint32_t val = __funnelshift_l(v[u], v[u], 8u * k);  // T_k[x] = rotl(T_0[x], 8k)
        const uint32_t base = A + k * kTable + (p >> 2) * 128u;
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) sts128(base + 16u * ((j + p) & 7u), val);
    }
#pragma unroll
    for (int u = 0; u < NS; ++u) {
        const uint32_t x = threadIdx.x + u * THREADS;
        if (x < 256u) {
            const uint32_t base = A + 4 * kTable + x * 128u;
#pragma unroll
            for (uint32_t j = 0; j < 8; ++j) sts128(base + 16u * ((j + x) & 7u), v[N + u]);
        }
    }
}

// Entry [byte K of w] of table T for the lane whose base is L = A + 4 * lane.
template <int K, uint32_t T>
__device__ __forceinline__ uint32_t look(uint32_t w, uint32_t L) {
    return lds_off<T * kTable>(__dp4a(w, 0x80u << (8 * K), L));
}

template <bool DECRYPT>
__device__ __forceinline__ void round_inner(uint32_t (&s)[4], uint32_t L, uint4 k) {
    constexpr int D = DECRYPT ? 3 : 1;  // Eq. 1 takes I_{j+k,k}, the inverse cipher I_{j-k,k}
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        t[j] = look<0, 0>(s[j], L) ^ look<1, 1>(s[(j + D) & 3], L) ^ look<2, 2>(s[(j + 2) & 3], L) ^
               look<3, 3>(s[(j + 3 * D) & 3], L) ^ kk[j];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

// Last round: S[x] is byte 0 of T2, byte 1 of T3, byte 2 of T0 and byte 3 of T1;
// the inverse S-box has a table of its own, its value in all four bytes.
template <bool DECRYPT>
__device__ __forceinline__ void round_last(uint32_t (&s)[4], uint32_t L, uint4 k) {
    constexpr int D = DECRYPT ? 3 : 1;
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t o = merge(look<0, DECRYPT ? 4 : 2>(s[j], L), look<1, DECRYPT ? 4 : 3>(s[(j + D) & 3], L), 0x000000ffu);
        o = merge(o, look<2, DECRYPT ? 4 : 0>(s[(j + 2) & 3], L), 0x0000ffffu);
        o = merge(o, look<3, DECRYPT ? 4 : 1>(s[(j + 3 * D) & 3], L), 0x00ffffffu);
        t[j] = o ^ kk[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

// Rounds FIRST..NR (the whitening is the caller's) on BPT independent states
// sharing one schedule, the round loop kept rolled: the body of one round is all
// that a warp's instruction fetch has to hold, and a rolled loop measured the same
// as an unrolled one (916 GB/s at 1 GiB).
template <int NR, bool DECRYPT, int FIRST, int BPT, class KS>
__device__ __forceinline__ void rounds_from(uint32_t (&s)[BPT][4], const KS& ks, uint32_t L) {
#pragma unroll 1
    for (int r = FIRST; r < NR; ++r) {
        const uint4 k = ks.get(r);
#pragma unroll
        for (int b = 0; b < BPT; ++b) round_inner<DECRYPT>(s[b], L, k);
    }
    const uint4 k = ks.get(NR);
#pragma unroll
    for (int b = 0; b < BPT; ++b) round_last<DECRYPT>(s[b], L, k);
}

}  // namespace dp
}  // namespace gbaes
