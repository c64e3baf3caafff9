// CTR mode on long inputs: the first two rounds shared between blocks.
//
// Section 3's CTR listing enciphers a counter per block, and counters that follow
// one another differ in one or two bytes.  Take the blocks whose counters agree in
// the upper 14 bytes, and call the two lowest bytes y and x.  After round 1 of
// Eq. 1 column 0 depends on x alone, another column on y alone (1 for the
// big-endian counter, 3 for the little-endian one) and two on neither; round 2
// XORs one lookup of each column into every word, so the state after it is
//     F(x, y) = A(x) ^ B(y) = F(x, y0) ^ F(0, y0) ^ F(0, y).
// (Sharing the first rounds of neighbouring counters is Bernstein and Schwabe's
// "counter-mode caching", New AES Software Speed Records, 2008; splitting round 2
// in two parts, each common to many blocks, spares all 32 lookups of both rounds.)
//
// Rows of 256 counters share y.  A thread takes the counters x and x + 128 of
// consecutive rows: it keeps F(x, y0) ^ F(0, y0) of both in registers while the
// upper 14 bytes last (2^16 counters), and its warp F(0, y) of the next 32 rows --
// the same for all lanes -- in shared memory, one 16-byte broadcast load per row in
// place of 2 x 32 lookups.  All come from two ordinary rounds, 32 lookups per lane
// each.
//
// Bound: the shared-memory lookups of the remaining Nr - 2 rounds (16 per block and
// round, 32 lanes per clock and SM) and the L1 cycles of the global loads and
// stores (about 12 per 32 blocks): 1 GiB of AES-128 takes 143 of the 128 + 12
// cycles per 32 blocks, where ten rounds take 173.  Measured, with all the rounds in
// the table kernel and here: 1 GiB 1,153 -> 954 us (1,125 GB/s; AES-256 1,583 -> 1,382),
// 256 MiB 291 -> 242 (400 -> 349), 16 MiB 20.6 -> 17.4 (27.0 -> 24.1).  An input whose first
// counter is odd, so that a warp's 512 bytes straddle five lines, takes 1% more.
// One counter a row (four rows at a time) measured 969 us at 1 GiB, four counters 947
// (AES-256 1,433); two CTAs per SM with 64 registers a thread 984.
#include "block_io.cuh"
#include "launch.cuh"

namespace gbaes {

constexpr int kCtrThreads = 512;
constexpr int kCtrX = 2;                             // counters of a row per thread
constexpr uint32_t kCtrSpan = 256 / kCtrX;           // threads across a row
constexpr int kCtrRanges = kCtrThreads / kCtrSpan;   // row ranges per CTA
constexpr uint32_t kCtrSlots = 32;                   // rows whose F(0, y) a warp keeps
constexpr uint32_t kCtrSmem = kTableBytes + (kCtrThreads / 32) * kCtrSlots * 16u;

// This thread's counters of one row: v = 256 row + x + kCtrSpan * g is a block's
// counter less the (2^16-aligned) counter base, and v - a.first its place in the
// input; places outside the input (before its first counter, past its last) compute
// and store nothing.
template <int NR>
__device__ __forceinline__ void ctr_row(const EcbArgs& a, uint64_t row, uint32_t x, const uint32_t (&ax)[kCtrX][4],
                                        uint32_t slots, uint32_t L) {
    uint32_t s[kCtrX][4];
    uint4 data[kCtrX];
    const uint64_t i0 = (row << 8) + x - a.first;
#pragma unroll
    for (int g = 0; g < kCtrX; ++g) {
        const uint64_t i = i0 + kCtrSpan * g;
        data[g] = i < a.nblocks ? ld_stream(a.in + i) : make_uint4(0, 0, 0, 0);
    }
    uint4 f;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(f.x), "=r"(f.y), "=r"(f.z), "=r"(f.w)
                 : "r"(slots + 16u * ((uint32_t)row % kCtrSlots)));
#pragma unroll
    for (int g = 0; g < kCtrX; ++g) {
        s[g][0] = ax[g][0] ^ f.x;
        s[g][1] = ax[g][1] ^ f.y;
        s[g][2] = ax[g][2] ^ f.z;
        s[g][3] = ax[g][3] ^ f.w;
    }
    rounds_from<NR, false, 3, kCtrX, NR>(s, ParamKeys{a.rk}, L);
#pragma unroll
    for (int g = 0; g < kCtrX; ++g) {
        const uint64_t i = i0 + kCtrSpan * g;
        if (i < a.nblocks) store_block<kCtr>(a, i, s[g], data[g]);
    }
}

// The states after two rounds of the counters v[i] past the base.
template <int N>
__device__ __forceinline__ void two_rounds(const EcbArgs& a, const uint64_t (&v)[N], uint32_t L, uint32_t (&s)[N][4]) {
    const ParamKeys ks{a.rk};
#pragma unroll
    for (int i = 0; i < N; ++i) {
        counter_words(a, v[i], s[i]);
        const uint4 k = ks.get(0);
        s[i][0] ^= k.x;
        s[i][1] ^= k.y;
        s[i][2] ^= k.z;
        s[i][3] ^= k.w;
    }
#pragma unroll
    for (int r = 1; r <= 2; ++r)
#pragma unroll
        for (int i = 0; i < N; ++i) round_inner<false>(s[i], L, ks.get(r));
}

// a.ctr_hi, a.ctr_lo: the counter base, its low 16 bits 0; a.first: the first
// block's counter less the base (below 2^16).
template <int NR>
__global__ void __launch_bounds__(kCtrThreads, 1) ctr_kernel(const EcbArgs a) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    pdl_trigger();
    const uint32_t A = smem_base(smem_raw);
    fill_table(A, false, threadIdx.x, kCtrThreads);
    __syncthreads();
    pdl_wait();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t L = A + 4u * lane;
    const uint32_t slots = A + kTableBytes + (threadIdx.x >> 5) * kCtrSlots * 16u;
    const uint32_t x = threadIdx.x % kCtrSpan;
    // Rows with blocks of the input, shared out evenly over the row ranges of all CTAs.
    const uint64_t row0 = a.first >> 8;
    const uint64_t rows = ((a.first + a.nblocks - 1) >> 8) - row0 + 1;
    const uint64_t range = (uint64_t)blockIdx.x * kCtrRanges + threadIdx.x / kCtrSpan;
    const uint64_t ranges = (uint64_t)gridDim.x * kCtrRanges;
    uint64_t row = row0 + rows * range / ranges;
    const uint64_t end = row0 + rows * (range + 1) / ranges;
    uint64_t high = ~0ull;  // row / 256 that ax belongs to
    uint32_t ax[kCtrX][4] = {};
    while (row < end) {
        const uint64_t slot_row = row & ~(uint64_t)(kCtrSlots - 1);
        uint32_t f[4];
        if (row >> 8 != high) {
            high = row >> 8;
            uint64_t v[kCtrX + 1];
            uint32_t t[kCtrX + 1][4];
            v[kCtrX] = (slot_row + lane) << 8;
#pragma unroll
            for (int g = 0; g < kCtrX; ++g) v[g] = (slot_row << 8) + x + kCtrSpan * g;
            two_rounds<kCtrX + 1>(a, v, L, t);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                f[w] = t[kCtrX][w];
                const uint32_t f0 = __shfl_sync(0xffffffffu, f[w], 0);
#pragma unroll
                for (int g = 0; g < kCtrX; ++g) ax[g][w] = t[g][w] ^ f0;
            }
        } else {
            uint32_t t[1][4];
            two_rounds<1>(a, {(slot_row + lane) << 8}, L, t);
#pragma unroll
            for (int w = 0; w < 4; ++w) f[w] = t[0][w];
        }
        __syncwarp();  // every lane is done with the slots' previous rows
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(slots + 16u * lane), "r"(f[0]), "r"(f[1]),
                     "r"(f[2]), "r"(f[3])
                     : "memory");
        __syncwarp();
        const uint64_t stop = slot_row + kCtrSlots < end ? slot_row + kCtrSlots : end;
        for (; row < stop; ++row) ctr_row<NR>(a, row, x, ax, slots, L);
    }
}

// Shortest input that takes this kernel: 2.5 rows for every row range, so that half of
// the ranges have three rows and half two.  With fewer, the two rounds ahead of a range's
// first row cost more than the rounds spared; from 330,000 to 470,000 blocks the two kernels
// are within 2% of one another either way, by how the rows and passes divide.  The table
// kernel against this one, captured calls / calls of a stream, in us: AES-128 272,384
// blocks 6.98 / 6.09 and 7.14 / 6.65, 389,120 9.16 / 8.42 and 8.82 / 8.36, 544,768 11.81 / 11.10 and
// 11.03 / 10.61; AES-256 8.81 / 7.88 and 9.16 / 8.69, 11.74 / 10.97 and 11.61 / 11.15, 15.38 / 14.63 and
// 14.82 / 14.39.
uint64_t ctr_min_blocks(int sms) { return (uint64_t)sms * kCtrRanges * 256u * 5u / 2u; }

int launch_ctr(EcbArgs a, int nr, cudaStream_t stream) {
    DeviceInfo info;
    int rc = current_device_info(&info);
    if (rc) return rc;
    using Fn = void (*)(const EcbArgs);
    const Fn fn = nr == 10 ? ctr_kernel<10> : nr == 12 ? ctr_kernel<12> : nr == 14 ? ctr_kernel<14> : nullptr;
    if (!fn) return fail(AES_ERR_ARG, "no CTR kernel for nr=%d", nr);
    // The first counter, split into a base with 16 zero low bits and the rest.
    const uint64_t lo = a.ctr_lo + a.first;
    if (lo < a.ctr_lo) ++a.ctr_hi;
    a.ctr_lo = lo & ~0xffffull;
    a.first = lo & 0xffffull;
    const cudaError_t e = launch_overlapped(fn, (unsigned)info.sms, kCtrThreads, kCtrSmem, stream, a);
    if (e != cudaSuccess) return fail(AES_ERR_CUDA, "CTR kernel launch: %s", cudaGetErrorString(e));
    return AES_OK;
}

}  // namespace gbaes
