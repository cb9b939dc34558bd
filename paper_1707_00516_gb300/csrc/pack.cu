// Profile preparation kernels: packing (Sec. II-A), mixtures (per-word OR),
// database rows with popcounts, and the per-query operands of the plain form.
#include "common.cuh"

namespace fastid {

namespace {

// Bit 7 of each byte of the result: that byte of x is not 0.
__device__ __forceinline__ uint32_t nonzero4(uint32_t x) {
    return (((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) & 0x80808080u;
}

// Eight allele bytes -> eight bits in the top byte.  Bytes of x go to bits 8i
// and bytes of y to bits 8i + 4; the multiplier 2^24 + 2^17 + 2^10 + 2^3 moves
// bit 8i to 24 + i and bit 8i + 4 to 28 + i by its term 2^(24 - 7i), the terms
// j > i land at distinct positions below bit 24 (no carries) and j < i
// overflow.
__device__ __forceinline__ uint32_t bytes8_to_top(uint32_t x, uint32_t y) {
    return ((nonzero4(x) >> 7) | (nonzero4(y) >> 3)) * 0x01020408u;
}

// Sixteen allele bytes -> 16 bits.
__device__ __forceinline__ uint32_t bytes16_to_bits(const uint4 v) {
    return __byte_perm(bytes8_to_top(v.x, v.y), bytes8_to_top(v.z, v.w), 0x4473) & 0xFFFFu;
}

// The word of `live` (1..64) loci at a, byte by byte.
__device__ __noinline__ uint64_t word_bytewise(const uint8_t *a, int live) {
    uint64_t word = 0;
#pragma unroll 16
    for (int t = 0; t < live; ++t) word |= (uint64_t)(a[t] != 0) << t;
    return word;
}

// The same from the aligned 16-byte blocks that hold the loci, shifted into
// place: all of the word's loads are in flight together, whatever its
// alignment and length.  The blocks may reach into the next row or the gap
// between rows, never outside the buffer's first to last allele [lo, hi).
__device__ __forceinline__ uint64_t word_of(const uint8_t *a, int live, const uint8_t *lo, const uint8_t *hi) {
    const uint32_t s = (uint32_t)(reinterpret_cast<uintptr_t>(a) & 15);
    const uint8_t *p = a - s;
    const int blocks = ((int)s + live + 15) >> 4;  // up to five
    if (p < lo || p + 16 * blocks > hi) return word_bytewise(a, live);  // the buffer's first or last word
    uint4 v[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) v[c] = c < blocks ? __ldg(reinterpret_cast<const uint4 *>(p) + c) : make_uint4(0, 0, 0, 0);
    uint64_t word = (uint64_t)(bytes16_to_bits(v[0]) | (bytes16_to_bits(v[1]) << 16)) |
                    ((uint64_t)(bytes16_to_bits(v[2]) | (bytes16_to_bits(v[3]) << 16)) << 32);
    if (s) word = (word >> s) | ((uint64_t)bytes16_to_bits(v[4]) << (64 - s));
    return live < 64 ? word & ((1ull << live) - 1ull) : word;
}
__device__ __noinline__ uint64_t word_of_call(const uint8_t *a, int live, const uint8_t *lo, const uint8_t *hi) {
    return word_of(a, live, lo, hi);
}

// G = 1 << log_g lanes share a row and make its 64-bit words, one a lane and
// step; without norms the words of a row are also spread over cpr groups.
// ALIGNED: rows start on 16 bytes, so every word but a row's last is four
// whole blocks.  HBM-bound at size; the register limits keep enough warps to
// cover the loads (60 registers: 262,144 x 2048 at 101 us instead of 87), and
// the conversion is 21 instructions for 16 bytes.  Against a warp a row with
// words off 16 bytes and last words read byte by byte: 262,144 x 2047 890 ->
// 105 us, 1M x 1000 1768 -> 205, 1M x 1024 273 -> 169, 2M x 200 1560 -> 95,
// 1000 x 65,536 17.5 -> 12.5, 262,144 x 2048 88 -> 87 (6.9 TB/s).  Coalesced
// blocks with four lanes a word and shuffles between them were slower (151 us).
template <bool ALIGNED>
__global__ void __launch_bounds__(256, ALIGNED ? 8 : 5)
    pack_kernel(const uint8_t *__restrict__ alleles, int64_t n, int32_t n_loci, int64_t ld_alleles,
                uint64_t *__restrict__ packed, int64_t ld_words, uint32_t *__restrict__ norms, int log_g,
                int64_t cpr) {
    const int g = 1 << log_g, lane = threadIdx.x & (g - 1);
    const int64_t units = n * cpr, step = ((int64_t)gridDim.x * blockDim.x) >> log_g;
    const uint8_t *lo = alleles, *hi = alleles + (n - 1) * ld_alleles + n_loci;
    // (whole warps stay in the loop, for the norms' shuffles)
    for (int64_t u0 = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) >> log_g; u0 < units; u0 += step) {
        const int64_t u = u0 + ((threadIdx.x & 31) >> log_g);
        const int64_t row = cpr == 1 ? u : u / cpr, part = cpr == 1 ? 0 : u - row * cpr;
        const uint8_t *a = alleles + row * ld_alleles;
        uint32_t pc = 0;
        for (int64_t w = part * g + lane; u < units && w < ld_words; w += g * cpr) {
            uint64_t word = 0;
            const int64_t l0 = w * 64;
            if (ALIGNED && l0 + 64 <= n_loci) {
                const uint4 *p = reinterpret_cast<const uint4 *>(a + l0);
                const uint4 v0 = __ldg(p), v1 = __ldg(p + 1), v2 = __ldg(p + 2), v3 = __ldg(p + 3);
                word = (uint64_t)(bytes16_to_bits(v0) | (bytes16_to_bits(v1) << 16)) |
                       ((uint64_t)(bytes16_to_bits(v2) | (bytes16_to_bits(v3) << 16)) << 32);
            } else if (l0 < n_loci) {
                const int live = n_loci - l0 < 64 ? (int)(n_loci - l0) : 64;
                word = ALIGNED ? word_of_call(a + l0, live, lo, hi) : word_of(a + l0, live, lo, hi);
            }
            packed[row * ld_words + w] = word;
            pc += __popcll(word);
        }
        if (norms) {
            for (int off = g >> 1; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
            if (lane == 0 && u < units) norms[row] = pc;
        }
    }
}

__global__ void mix_kernel(const uint64_t *__restrict__ src, int64_t ld_src, int32_t n_words,
                           const int32_t *__restrict__ offsets, int64_t n_mix,
                           uint64_t *__restrict__ out, int64_t ld_out, uint32_t *__restrict__ norms) {
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t m = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); m < n_mix;
         m += warps_total) {
        const int32_t s0 = offsets[m], s1 = offsets[m + 1];
        uint32_t pc = 0;
        for (int64_t w = lane; w < ld_out; w += 32) {
            uint64_t v = 0;
            if (w < n_words)
                for (int32_t s = s0; s < s1; ++s) v |= __ldg(src + (int64_t)s * ld_src + w);
            out[m * ld_out + w] = v;
            pc += __popcll(v);
        }
        if (norms) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
            if (lane == 0) norms[m] = pc;
        }
    }
}

// dst[r][w] = src[r][w] for r < n, w < n_words; zero elsewhere up to n_pad
// rows and ld_dst words.  norms[r] = popcount of the row (0 for padding rows).
__global__ void copy_rows_kernel(const uint64_t *__restrict__ src, int64_t n, int64_t ld_src,
                                 int32_t n_words, uint64_t *__restrict__ dst, int64_t n_pad,
                                 int64_t ld_dst, uint32_t *__restrict__ norms) {
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n_pad;
         r += warps_total) {
        uint32_t pc = 0;
        for (int64_t w = lane; w < ld_dst; w += 32) {
            uint64_t v = (r < n && w < n_words) ? __ldg(src + r * ld_src + w) : 0ull;
            dst[r * ld_dst + w] = v;
            pc += __popcll(v);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
        if (lane == 0 && norms) norms[r] = pc;
    }
}

// Plain-form query operands: rows of 32-bit words at stride ld32 (padded to
// n_q_pad rows, zero beyond n_q / n_words) and per-query coefficients.
__global__ void query_prep_kernel(const uint64_t *__restrict__ q, int64_t ld_q, int64_t n_q,
                                  int32_t n_words, const uint8_t *__restrict__ modes,
                                  uint32_t *__restrict__ q32, int64_t n_q_pad, int64_t ld32,
                                  QueryCoef *__restrict__ coef) {
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t ld64 = ld32 / 2;
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n_q_pad;
         r += warps_total) {
        uint32_t pc = 0;
        for (int64_t w = lane; w < ld64; w += 32) {
            uint64_t v = (r < n_q && w < n_words) ? __ldg(q + r * ld_q + w) : 0ull;
            reinterpret_cast<uint2 *>(q32 + r * ld32)[w] = make_uint2((uint32_t)v, (uint32_t)(v >> 32));
            pc += __popcll(v);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
        if (lane == 0) {
            QueryCoef c;
            if (r < n_q && modes[r] == FASTID_MODE_MISMATCH) {
                c.a = 2u;  // popc(R ^ Q) = |R| + |Q| - 2 popc(R & Q)
                c.b = pc;
            } else {
                c.a = 1u;  // Eq. 1: popc(R & ~Q) = |R| - popc(R & Q)
                c.b = 0u;
            }
            coef[r] = c;
        }
    }
}

int warp_grid(int64_t rows, int warps_per_block) {
    int64_t blocks = (rows + warps_per_block - 1) / warps_per_block;
    if (blocks > 65535 * 8) blocks = 65535 * 8;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

}  // namespace

cudaError_t launch_pack(const uint8_t *alleles, int64_t n, int32_t n_loci, int64_t ld_alleles,
                        uint64_t *packed, int64_t ld_words, uint32_t *norms, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    // lanes a row: as many as it has words, up to a warp; more words than
    // that go to further groups where no norm joins them
    int log_g = 0;
    while (log_g < 5 && (1 << log_g) < ld_words) ++log_g;
    const int64_t cpr = norms ? 1 : (ld_words + (1 << log_g) - 1) >> log_g;
    const bool aligned = ((ld_alleles | (int64_t)reinterpret_cast<uintptr_t>(alleles)) & 15) == 0;
    const int grid = warp_grid(((n * cpr << log_g) + 31) >> 5, 8);
    if (aligned)
        pack_kernel<true><<<grid, 256, 0, s>>>(alleles, n, n_loci, ld_alleles, packed, ld_words, norms, log_g, cpr);
    else
        pack_kernel<false><<<grid, 256, 0, s>>>(alleles, n, n_loci, ld_alleles, packed, ld_words, norms, log_g, cpr);
    return cudaGetLastError();
}

cudaError_t launch_mix(const uint64_t *src, int64_t ld_src, int32_t n_words, const int32_t *offsets,
                       int64_t n_mix, uint64_t *out, int64_t ld_out, uint32_t *norms, cudaStream_t s) {
    if (n_mix == 0) return cudaSuccess;
    mix_kernel<<<warp_grid(n_mix, 8), 256, 0, s>>>(src, ld_src, n_words, offsets, n_mix, out, ld_out, norms);
    return cudaGetLastError();
}

cudaError_t launch_copy_rows(const uint64_t *src, int64_t n, int64_t ld_src, int32_t n_words,
                             uint64_t *dst, int64_t n_pad, int64_t ld_dst, uint32_t *norms,
                             cudaStream_t s) {
    if (n_pad == 0) return cudaSuccess;
    copy_rows_kernel<<<warp_grid(n_pad, 8), 256, 0, s>>>(src, n, ld_src, n_words, dst, n_pad, ld_dst, norms);
    return cudaGetLastError();
}

cudaError_t launch_query_prep(const uint64_t *q, int64_t ld_q, int64_t n_q, int32_t n_words,
                              const uint8_t *modes, uint32_t *q32, int64_t n_q_pad, int64_t ld32,
                              QueryCoef *coef, cudaStream_t s) {
    if (n_q_pad == 0) return cudaSuccess;
    query_prep_kernel<<<warp_grid(n_q_pad, 8), 256, 0, s>>>(q, ld_q, n_q, n_words, modes, q32, n_q_pad,
                                                            ld32, coef);
    return cudaGetLastError();
}

}  // namespace fastid
