// Loading and storing one block in each mode, shared by the single-call kernels
// (ecb_table.cu, ctr.cu).
#pragma once

#include "aes_rounds.cuh"

namespace gbaes {

__device__ __forceinline__ uint32_t bswap32(uint32_t x) { return __byte_perm(x, 0, 0x0123u); }

// Counter block for counter index i (128-bit base + i, modulo 2^128).
__device__ __forceinline__ void counter_words(const EcbArgs& a, uint64_t i, uint32_t (&w)[4]) {
    uint64_t lo = a.ctr_lo + i;
    uint64_t hi = a.ctr_hi + (lo < a.ctr_lo ? 1u : 0u);
    if (a.ctr_be) {
        w[0] = bswap32((uint32_t)(hi >> 32));
        w[1] = bswap32((uint32_t)hi);
        w[2] = bswap32((uint32_t)(lo >> 32));
        w[3] = bswap32((uint32_t)lo);
    } else {
        w[0] = (uint32_t)lo;
        w[1] = (uint32_t)(lo >> 32);
        w[2] = (uint32_t)hi;
        w[3] = (uint32_t)(hi >> 32);
    }
}

// Loads block idx of the input (ok: idx < n) into the cipher state s, and what
// the mode combines with the cipher output into aux: CTR encrypts the counter
// block and keeps the data, CBC decryption keeps the previous ciphertext block
// (the IV for block 0).  Lanes past the end compute on zeros.
template <int MODE>
__device__ __forceinline__ void load_block(const EcbArgs& a, uint64_t idx, bool ok, uint32_t (&s)[4], uint4& aux) {
    uint4 v = make_uint4(0, 0, 0, 0);
    if (MODE == kCtr) {
        counter_words(a, a.first + idx, s);
        if (ok) v = ld_stream(a.in + idx);
        aux = v;
    } else {
        // (CBC decryption reads every block twice, the second time as its successor's
        // predecessor: kept in L1 for that, 1 GiB takes 0.3-0.4% less)
        if (ok) v = MODE == kCbcDec ? ld_keep(a.in + idx) : ld_stream(a.in + idx);
        s[0] = v.x;
        s[1] = v.y;
        s[2] = v.z;
        s[3] = v.w;
        if (MODE == kCbcDec) {
            uint4 p = make_uint4(a.iv[0], a.iv[1], a.iv[2], a.iv[3]);
            if (ok && idx > 0) p = ld_keep(a.in + idx - 1);
            aux = p;
        }
    }
}

template <int MODE>
__device__ __forceinline__ void store_block(const EcbArgs& a, uint64_t idx, const uint32_t (&s)[4], const uint4& aux) {
    uint4 o = make_uint4(s[0], s[1], s[2], s[3]);
    if (MODE == kCtr || MODE == kCbcDec) {
        o.x ^= aux.x;
        o.y ^= aux.y;
        o.z ^= aux.z;
        o.w ^= aux.w;
    }
    __stcs(a.out + idx, o);
}

}  // namespace gbaes
