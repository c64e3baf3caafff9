// T-table AES kernels for sm_103a: ECB encryption/decryption, CTR, CBC decryption.
//
// Each round is Eq. 1 of the paper: four output words, each the XOR of four
// 32-bit table lookups and a round-key word,
//     O_j = T0[I_{j,0}] ^ T1[I_{j+1,1}] ^ T2[I_{j+2,2}] ^ T3[I_{j+3,3}] ^ K_j
// (indices of I mod 4), and for the inverse cipher the same with Td tables and
// I_{j-k,k}.  The paper keeps the tables in a texture (Section 3); here one of them,
// 32 times replicated, sits in shared memory (aes_rounds.cuh), the others are
// rotations of it.
//
// Two CTAs of 512 threads per SM (one for short calls), persistent over the input; each block is a
// coalesced 16-byte load and store, and round keys come from the kernel parameters.
#include <algorithm>

#include "block_io.cuh"
#include "launch.cuh"

namespace gbaes {

__device__ int g_status;  // nonzero: a kernel reported an error (resident.cu)

// Blocks i, i + step, ... of a thread: loads, rounds and stores.  Blocks from `end`
// on are computed on zeros and not stored.
template <int MODE, int BPT>
__device__ __forceinline__ void load_blocks(const EcbArgs& a, uint64_t i, uint32_t step, uint64_t end,
                                            uint32_t (&s)[BPT][4], uint4 (&aux)[BPT]) {
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const uint64_t idx = i + (uint64_t)b * step;
        load_block<MODE>(a, idx, idx < end, s[b], aux[b]);
    }
}

template <int NR, int MODE, int BPT>
__device__ __forceinline__ void cipher_blocks(const EcbArgs& a, uint64_t i, uint32_t step, uint64_t end,
                                              uint32_t (&s)[BPT][4], const uint4 (&aux)[BPT], uint32_t L) {
    constexpr bool DECRYPT = (MODE == kDec || MODE == kCbcDec);
    whiten<BPT>(s, ParamKeys{a.rk});
    // In full: 1 GiB 1,148 us (AES-256 decryption 1,583), three rounds per iteration 1,156 (1,683).
    rounds_from<NR, DECRYPT, 1, BPT, NR>(s, ParamKeys{a.rk}, L);
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const uint64_t idx = i + (uint64_t)b * step;
        if (idx < end) store_block<MODE>(a, idx, s[b], aux[b]);
    }
}

// The CTAs take passes of blockDim.x * BPT blocks in turn, as many as there are for
// all of them, then equal shares of the rest (less than a pass each; they differ by
// 32 blocks at most, whatever n is), one state at a time so that whole warps past
// the end of a share skip it.  The next pass's input -- the rest's, after the last
// full pass -- is loaded before the rounds of the pass before it, except with 4
// blocks per thread, where holding both would spill.
template <int NR, int MODE, int BPT>
__global__ void __launch_bounds__(1024, 1) table_kernel(const EcbArgs a) {
    constexpr bool DECRYPT = (MODE == kDec || MODE == kCbcDec);
    constexpr bool kAhead = BPT <= 2;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const uint32_t A = smem_base(smem_raw);
    // The table's last pieces stay in registers until the first blocks' loads are out,
    // where those come first.
    uint32_t piece[kFillChunk], p = threadIdx.x;
    for (; p + kFillChunk * blockDim.x < kFillPieces; p += kFillChunk * blockDim.x) {
        fill_load(DECRYPT, p, blockDim.x, piece);
        fill_store(A, p, blockDim.x, piece);
    }
    fill_load(DECRYPT, p, blockDim.x, piece);
    const uint32_t L = A + 4u * (threadIdx.x & 31u);
    const uint32_t step = blockDim.x;
    const uint64_t stride = (uint64_t)step * BPT * gridDim.x;  // blocks of one pass of every CTA
    const uint64_t n = a.nblocks, first = n / stride * stride, units = (n - first + 31) / 32;
    uint64_t i = (uint64_t)step * BPT * blockIdx.x + threadIdx.x;
    uint64_t rest = first + units * blockIdx.x / gridDim.x * 32 + threadIdx.x;  // this thread's first block of the rest
    uint64_t end = first + units * (blockIdx.x + 1) / gridDim.x * 32;
    if (end > n) end = n;
    uint32_t next[BPT][4];
    uint4 next_aux[BPT];  // CTR: data; CBC: previous ciphertext block
    const bool any = i < first;
    if (a.loads_first) {
        pdl_wait();
        if (kAhead) load_blocks<MODE, BPT>(a, any ? i : rest, step, any ? first : end, next, next_aux);
    }
    fill_store(A, p, blockDim.x, piece);
    if (!a.loads_first) {
        pdl_wait();
        if (kAhead) load_blocks<MODE, BPT>(a, any ? i : rest, step, any ? first : end, next, next_aux);
    }
    __syncthreads();
    pdl_trigger();  // (after the barrier: 0.2 us less per call than at the kernel's start)
    while (i < first) {
        uint32_t s[BPT][4];
        uint4 aux[BPT];
        const uint64_t ni = i + stride;
        if (kAhead) {
#pragma unroll
            for (int b = 0; b < BPT; ++b) {
                aux[b] = next_aux[b];
#pragma unroll
                for (int w = 0; w < 4; ++w) s[b][w] = next[b][w];
            }
            const bool full = ni < first;
            load_blocks<MODE, BPT>(a, full ? ni : rest, step, full ? first : end, next, next_aux);
        } else {
            load_blocks<MODE, BPT>(a, i, step, first, s, aux);
        }
        cipher_blocks<NR, MODE, BPT>(a, i, step, first, s, aux, L);
        i = ni;
    }
#pragma unroll 1
    for (int b = 0; b < BPT && rest < end; ++b, rest += step) {
        uint32_t s[1][4];
        uint4 aux[1];
        if (kAhead) {
            aux[0] = next_aux[0];
#pragma unroll
            for (int w = 0; w < 4; ++w) s[0][w] = next[0][w];
            next_aux[0] = next_aux[BPT - 1];
#pragma unroll
            for (int w = 0; w < 4; ++w) next[0][w] = next[BPT - 1][w];
        } else {
            load_blocks<MODE, 1>(a, rest, step, end, s, aux);
        }
        cipher_blocks<NR, MODE, 1>(a, rest, step, end, s, aux, L);
    }
}

// ------------------------------------------------------------ compact tables
//
// AES_KERNEL_TABLE_COMPACT: each of T0..T3 (and the inverse S-box) once, 4-5 KiB of
// shared memory, one word per thread to write.  Its lookups may meet bank conflicts
// (32 lanes, random bytes, one copy).  Nothing chooses it by itself any more: with
// one replicated table of 32 KiB per CTA short calls are faster than with this
// (AES-128 / 256 encryption, captured calls, this against table_kernel: 1 block
// 2.01 / 2.24 and 1.90 / 2.08 us, 4,096 blocks 2.40 / 2.72 and 2.10 / 2.28, 9,728 blocks
// 2.27 / 2.56 and 2.12 / 2.29).
// Word x of table k sits at byte 1024*k + 4*x; the inverse S-box (its value in
// all four bytes) follows at 4096.

constexpr uint32_t kCompactWords = 5 * 256;

template <int K>
__device__ __forceinline__ uint32_t byte4(uint32_t w) {  // 4 * (byte K of w)
    return __byte_perm(w, 0u, 0x4440u | K) << 2;
}

__device__ __forceinline__ void fill_compact(uint32_t T, bool decrypt) {
    const uint32_t* t0 = decrypt ? g_tab.td0 : g_tab.te0;
    for (uint32_t x = threadIdx.x; x < 256u; x += blockDim.x) {
        const uint32_t v = __ldg(t0 + x);
        const uint32_t si = decrypt ? __ldg(g_tab.si4 + x) : 0u;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) sts(T + 1024u * k + 4u * x, __funnelshift_l(v, v, 8u * k));
        if (decrypt) sts(T + 4096u + 4u * x, si);
    }
}

__device__ __forceinline__ void enc_round_c(uint32_t (&s)[4], uint32_t T, uint4 k) {
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        t[j] = lds(T + byte4<0>(s[j])) ^ lds_off<1024>(T + byte4<1>(s[(j + 1) & 3])) ^
               lds_off<2048>(T + byte4<2>(s[(j + 2) & 3])) ^ lds_off<3072>(T + byte4<3>(s[(j + 3) & 3])) ^ kk[j];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

// S[x] is byte 0 of T2[x], byte 1 of T3[x], byte 2 of T0[x], byte 3 of T1[x].
__device__ __forceinline__ void enc_last_c(uint32_t (&s)[4], uint32_t T, uint4 k) {
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t o = merge(lds_off<2048>(T + byte4<0>(s[j])), lds_off<3072>(T + byte4<1>(s[(j + 1) & 3])), 0xffu);
        o = merge(o, lds(T + byte4<2>(s[(j + 2) & 3])), 0xffffu);
        o = merge(o, lds_off<1024>(T + byte4<3>(s[(j + 3) & 3])), 0xffffffu);
        t[j] = o ^ kk[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

__device__ __forceinline__ void dec_round_c(uint32_t (&s)[4], uint32_t T, uint4 k) {
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        t[j] = lds(T + byte4<0>(s[j])) ^ lds_off<1024>(T + byte4<1>(s[(j + 3) & 3])) ^
               lds_off<2048>(T + byte4<2>(s[(j + 2) & 3])) ^ lds_off<3072>(T + byte4<3>(s[(j + 1) & 3])) ^ kk[j];
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

__device__ __forceinline__ void dec_last_c(uint32_t (&s)[4], uint32_t T, uint4 k) {
    uint32_t t[4];
    const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t o = merge(lds_off<4096>(T + byte4<0>(s[j])), lds_off<4096>(T + byte4<1>(s[(j + 3) & 3])), 0xffu);
        o = merge(o, lds_off<4096>(T + byte4<2>(s[(j + 2) & 3])), 0xffffu);
        o = merge(o, lds_off<4096>(T + byte4<3>(s[(j + 1) & 3])), 0xffffffu);
        t[j] = o ^ kk[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = t[j];
}

template <int NR, bool DECRYPT>
__device__ __forceinline__ void cipher_compact(uint32_t (&s)[4], const ParamKeys& ks, uint32_t T) {
    const uint4 k0 = ks.get(0);
    s[0] ^= k0.x;
    s[1] ^= k0.y;
    s[2] ^= k0.z;
    s[3] ^= k0.w;
#pragma unroll
    for (int r = 1; r < NR; ++r) {
        if (DECRYPT)
            dec_round_c(s, T, ks.get(r));
        else
            enc_round_c(s, T, ks.get(r));
    }
    if (DECRYPT)
        dec_last_c(s, T, ks.get(NR));
    else
        enc_last_c(s, T, ks.get(NR));
}

// One block per thread, grid-stride.  The trigger comes after the wait, so that at
// most one later call's CTAs (which fit beside these) wait on the SMs: triggering
// first let several pile up (9.4 us per call of 304 KiB against 3.7).
template <int NR, int MODE>
__global__ void __launch_bounds__(256) table_compact_kernel(const EcbArgs a) {
    constexpr bool DECRYPT = (MODE == kDec || MODE == kCbcDec);
    __shared__ __align__(16) uint32_t tab[kCompactWords];
    const uint64_t n = a.nblocks;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t T = smem_base(tab);
    uint32_t s[4];
    uint4 aux;
    if (!a.loads_first) fill_compact(T, DECRYPT);
    pdl_wait();
    pdl_trigger();
    load_block<MODE>(a, i, i < n, s, aux);
    if (a.loads_first) fill_compact(T, DECRYPT);
    __syncthreads();
    while (i < n) {
        cipher_compact<NR, DECRYPT>(s, ParamKeys{a.rk}, T);
        store_block<MODE>(a, i, s, aux);
        i += stride;
        if (i >= n) break;
        load_block<MODE>(a, i, true, s, aux);
    }
}

// ------------------------------------------------------------------ launcher

namespace {

using KernelFn = void (*)(const EcbArgs);

template <int NR, int MODE>
KernelFn pick_bpt(int bpt) {
    switch (bpt) {
        case 1: return table_kernel<NR, MODE, 1>;
        case 2: return table_kernel<NR, MODE, 2>;
        case 4: return table_kernel<NR, MODE, 4>;
        default: return nullptr;
    }
}

template <int NR>
KernelFn pick_mode(int mode, int bpt, bool compact) {
    switch (mode) {
        case kEnc: return compact ? table_compact_kernel<NR, kEnc> : pick_bpt<NR, kEnc>(bpt);
        case kDec: return compact ? table_compact_kernel<NR, kDec> : pick_bpt<NR, kDec>(bpt);
        case kCtr: return compact ? nullptr : pick_bpt<NR, kCtr>(bpt);
        case kCbcDec: return compact ? nullptr : pick_bpt<NR, kCbcDec>(bpt);
        default: return nullptr;
    }
}

KernelFn pick(int nr, int mode, int bpt, bool compact) {
    switch (nr) {
        case 10: return pick_mode<10>(mode, bpt, compact);
        case 12: return pick_mode<12>(mode, bpt, compact);
        case 14: return pick_mode<14>(mode, bpt, compact);
        default: return nullptr;
    }
}

}  // namespace

// A CTA with less than one pass of blocks keeps at least this many threads, one chunk
// of its table's pieces each: with 128, which fill in two steps, 13,000 blocks take
// 2.71 us in a captured call instead of 2.43 (2.06 in a stream instead of 1.98).
constexpr int kMinThreads = (int)(kFillPieces / kFillChunk);

// Up to this many blocks per SM a call runs one CTA on each SM, above it two: a second
// table to write costs more than the warps of a second CTA give.  Captured calls with two
// CTAs and with one: 9,728 blocks 2.29 / 2.12 us (AES-256 decryption 2.49 / 2.29), 19,456
// 2.44 / 2.14 (2.75 / 2.31); at 256 blocks per SM (32,768 blocks) 2.53 / 2.38 (2.83 / 2.64), but
// in a stream, where the fill overlaps the call before, 2.02 / 2.52 (2.27 / 3.08).
constexpr uint64_t kOneCtaBlocksPerSm = 128;

int launch_table(EcbArgs a, int nr, Mode mode, int threads, int bpt, int variant, cudaStream_t stream) {
    DeviceInfo info;
    int rc = current_device_info(&info);
    if (rc) return rc;
    const uint64_t n = a.nblocks;
    const uint64_t sms = (uint64_t)info.sms;
    const bool compact = variant == AES_KERNEL_TABLE_COMPACT;
    // The automatic shape: one block per thread while that covers the input, which
    // spreads a short call over the most warps.  The shortest take it whatever shape is
    // asked for, unless the variant is too.
    if (variant == AES_KERNEL_TABLE && n <= kOneCtaBlocksPerSm * sms) threads = bpt = 0;
    if (threads == 0) threads = 512;
    if (bpt == 0) bpt = n <= 2 * sms * (uint64_t)threads ? 1 : 2;
    KernelFn fn = pick(nr, mode, bpt, compact);
    if (!fn) return fail(AES_ERR_ARG, "no table kernel for nr=%d mode=%d blocks_per_thread=%d", nr, (int)mode, bpt);
    unsigned grid;
    int smem = 0;
    if (compact) {
        // A warp per 32 blocks, spread over the SMs (at most 8 warps per CTA, 8 CTAs per SM).
        const uint64_t warps = (n + 31) / 32;
        uint64_t per_cta = (warps + sms - 1) / sms;
        if (per_cta > 8) per_cta = 8;
        const uint64_t ctas = (warps + per_cta - 1) / per_cta;
        grid = (unsigned)(ctas < 8 * sms ? ctas : 8 * sms);
        threads = (int)(32 * per_cta);
    } else {
        // Two CTAs per SM (64 registers a thread); one above 512 threads, and for short
        // calls if a pass of it covers its blocks.
        const bool brief = n <= sms * std::min<uint64_t>(kOneCtaBlocksPerSm, (uint64_t)threads);
        const uint64_t ctas = brief || threads > 512 ? sms : 2 * sms;
        const uint64_t units = (n + 31) / 32;
        grid = (unsigned)(units < ctas ? units : ctas);
        // A CTA with less than one pass of blocks needs no more threads than those.
        const uint64_t share = (units + grid - 1) / grid * 32;
        if (share < (uint64_t)threads) threads = (int)(share < kMinThreads ? std::min(kMinThreads, threads) : (int)share);
        // With one block per thread (40 registers) three CTAs and more would fit, and a
        // call's CTAs, placed while the call before it still runs, would crowd some SMs and
        // leave others idle (65,536 blocks 3.1-4.1 us per call of a stream, 100,000 blocks
        // 3.3-4.5): with this much shared memory two do (2.7, 3.1).
        smem = (int)kTableBytes;
        if (bpt == 1 && threads <= 512 && !brief) {
            smem = 100 << 10;
            rc = set_max_dynamic_smem((const void*)fn, smem);
            if (rc) return rc;
        }
    }
    const bool overlap = may_overlap(stream);
    a.loads_first = !overlap;
    const cudaError_t e = launch_overlapped(fn, grid, (unsigned)threads, (size_t)smem, stream, a, overlap);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "table kernel launch: %s", cudaGetErrorString(e));
    return AES_OK;
}

int device_status_word(int** p) {
    cudaError_t e = cudaGetSymbolAddress((void**)p, g_status);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "status word address: %s", cudaGetErrorString(e));
    return AES_OK;
}

int read_device_status(int clear) {
    int v = 0;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&v, g_status, sizeof(int));
    if (e == cudaSuccess && clear) {
        const int zero = 0;
        e = cudaMemcpyToSymbol(g_status, &zero, sizeof(int));
    }
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "reading device status: %s", cudaGetErrorString(e));
    return v;
}

}  // namespace gbaes
