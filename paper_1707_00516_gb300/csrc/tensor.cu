// Tensor-core form of the overloaded matrix multiply on 5th-generation
// tensor cores (tcgen05), FP32 accumulation in TMEM, with the 0/+-1 operands
// in one of two encodings:
//   FP8   kind::f8f6f4, e4m3 bytes (0x00, 0x38 = +1, 0xB8 = -1), K = 32 a MMA
//   FP4   kind::mxf4 block-scaled, e2m1 nibbles (0x0, 0x2 = +1, 0xA = -1)
//         with every ue8m0 scale factor 2^0, K = 64 a MMA: twice the FP8
//         rate per SM clock on GB300, and a quarter of the FP8 copy's bytes.
//
// The paper computes POPC(AND(XOR(R, Q), R)) word by word (Eq. 1,
// Algorithm 3).  On 0/1 vectors the same counts are ordinary dot products,
// so the contraction can run as a real GEMM D = A B^T if the query side is
// encoded per mode (l < N; padding loci are 0 on both sides):
//     mode 1 (Eq. 1):  a_l = 1 - Q_l      D = sum_l R_l (1 - Q_l) = popc(R AND NOT Q)
//     mode 0 (XOR):    a_l = 1 - 2 Q_l    D = |R| - 2 G,   popc(R XOR Q) = D + |Q|
// with b_l = R_l.  So score = D + c_q (c_q = |Q| in mode 0, 0 in mode 1) and
// no reference popcount is needed.  Every partial sum is an integer of
// magnitude <= N <= 65536 < 2^24, exact in FP32 whatever the order of the
// additions; 0, +1 and -1 are exact in e4m3 (0x00, 0x38, 0xB8).
//
// Tile: M = 128 queries (TMEM lanes) x N = 256 references (TMEM columns;
// 224 for FP4, whose two accumulators then leave TMEM columns 448-511 for the
// scale factors), K staged one 128-byte swizzle atom per pipeline stage by
// TMA (128 loci in FP8, 256 in FP4).
// Warp roles in a 192-thread CTA, one CTA per SM (persistent):
//   warp 0       TMA producer (one lane)
//   warp 1       TMEM allocation + MMA issue (one lane)
//   warps 2..5   epilogue: TMEM -> registers -> score filter -> per-query
//                top-k (thread = query), hit list or full score matrix; a second
//                set as the last four warps where ES = 2
//   warps 6..    packed-reference launches only (PK): expansion of the packed
//                reference stage into the FP8 stage (see expand_stage)
// Two accumulators (2 x 256 TMEM columns) let the epilogue of one reference
// tile overlap the MMAs of the next.  Every mbarrier wait is bounded: on
// timeout the thread records FASTID_ETIMEOUT in the status word and the CTA
// drains and exits.
#include <cuda.h>

#include <cstring>

#include "tc_ptx.cuh"

namespace fastid {

namespace {

constexpr int TC_BM = 128;          // queries per tile
constexpr int TC_BK = 128;          // loci (bytes) per stage
constexpr int TC_THREADS = 192;     // producer, MMA issuer, 4 epilogue warps (a second set: 128 more)
// PK: warps expanding packed references, after the 6 others.  Blocks of 257 to
// 384 threads get at most 168 registers a thread.  The 16-slot top-k runs with
// that (4 expanding warps), its queues spilling 92 (FP8) and 100 (FP4) bytes a
// thread: without queues nothing spilled and it was slower everywhere (96
// queries, N = 2048, k = 10, FP4, us: 20,000 references 83 -> 35, 500,000 211 ->
// 96, 2M 363 -> 225, 20M 1942 -> 1809).  The 32-slot one does not fit (2 warps).
__host__ __device__ constexpr int pk_threads(int km) { return km == 16 ? 128 : 64; }
constexpr uint32_t TC_A_BYTES = TC_BM * TC_BK;  // 16 KB
// Packed reference stage of PK launches: BN rows of the stage's loci (128
// bits for FP8, 256 for FP4).
__host__ __device__ constexpr uint32_t pk_stage_bytes(int bn, bool f4) { return (uint32_t)bn * (f4 ? 32u : 16u); }
// FP4 launches: reference tiles of 224, unit scale factors in TMEM columns
// TC_SF_COL.. (A's from TC_SF_COL, B's from TC_SF_COL + 16), all lanes.
constexpr int TC_BN4 = 224;
constexpr uint32_t TC_SF_COL = 448;
// Full-matrix launches: each epilogue warp turns a 32 x 32 block of scores
// from thread-per-query to query-major through a buffer of 32 rows of 36
// words (16-byte rows; a quarter-warp's 16-byte accesses meet every bank once
// both ways).
constexpr int SC_LD = 36;
constexpr uint32_t SC_BYTES = 4 * 32 * SC_LD * 4;
constexpr uint64_t RENDEZVOUS_NS = 50000000ull;  // 50 ms per panel entry, then go on alone

// What a launch's epilogue does with the scores (its own instances: lists take
// 32 to 64 registers a thread, transpose buffers a stage).
enum { MODE_TOPK, MODE_SCORES, MODE_HITS };

// Epilogue sets ES: for hit launches two sets of four warps, one an accumulator
// (even and odd tiles): one set is one warp a scheduler, whose latencies
// nothing hides (512 queries x 1M references, N = 1024, 0.6 hits a 32-column
// chunk, a call: 212 -> 203 us).  One for top-k -- two sets' own lists take
// twice the insertions, and their cuts come later (500 queries x 2M, N = 2048,
// k = 16: 604 -> 658 us) -- and for full matrices, which gain nothing (500 x
// 60,001 uint32: 55.9 and 56.1).
__host__ __device__ constexpr int tc_threads(int km, bool pk, int es) {
    return TC_THREADS + (pk ? pk_threads(km) : 0) + (es - 1) * 128;
}

// Kernel variants: references per tile (the MMA's N) and pipeline depth (as
// many stages as shared memory holds: the pipeline is latency-bound, and on
// GB300 going from 3 to 4 stages took the FP4 2048 x 20M launch from 27.5 to
// 24.5 ms).
//   BN = 256: 32 KB reference stage, 4 stages, 2 x 256 TMEM columns
//   BN = 224: 28 KB reference stage, 5 stages (4 with a packed stage), 2 x 224
//             TMEM columns + scale factors (FP4)
//   BN = 128: 16 KB reference stage, 6 stages, 2 x 128 TMEM columns
//   CG2 (2-SM MMA, see tensor_kernel): each CTA holds half of every reference
//             stage, 7 stages (FP8 32 KB, FP4 30 KB a stage)
//   SC (full-matrix launches): one stage less where the transpose buffers
//   (SC_BYTES) would not fit beside the ring
template <int BN, bool PK = false, bool CG2 = false, int MODE = MODE_TOPK>
struct TcShape {
    static constexpr bool SC = MODE == MODE_SCORES;
    static constexpr int RING = CG2 ? 7 : BN == 128 ? 6 : (BN == 224 && !PK) ? 5 : 4;
    static constexpr int STAGES = RING - (SC && (BN == 224) != PK ? 1 : 0);
    static constexpr uint32_t B_BYTES = (uint32_t)(CG2 ? BN / 2 : BN) * TC_BK;
    static constexpr uint32_t TMEM_COLS = BN == 128 ? 256 : 512;
    // beside the ring: transpose buffers, or the candidate queues (QD entries
    // a query row and epilogue set: what the fullest rings leave)
    static constexpr int ES = MODE == MODE_HITS ? 2 : 1;
    static constexpr int QD = ES == 2 ? (BN == 224 && !PK ? 5 : 8) : CG2 && BN == 256 ? 3 : 11;
    static constexpr int QG = QD < 8 ? 2 : 4;  // columns queued at a time, while QD - QG or fewer are
    static constexpr uint32_t EX_BYTES = SC ? SC_BYTES : (uint32_t)(ES * QD) * TC_BM * 4;
};

// One database ("panel") of a launch, with its schedule (TcSched).
struct PanelDesc {
    int64_t n_refs;
    int64_t n_q;          // real query rows (the operand is padded to whole tiles)
    int64_t n_rt;         // reference tiles
    int32_t n_kb;         // K stages of 128 operand bytes
    TcSched sc;
    const float *qconst;  // c_q per padded query row
    int32_t *gcut;        // shared cut per padded query row, or nullptr, and the
    int64_t gcut_ld;      // slices' published bounds (see TcLaunch)
    int32_t n_pub, pub_rank, pub_need;
    int32_t qspread;      // see spread_row_to_query
};

struct TcMaps {
    CUtensorMap a[TC_MAXP];  // query operand of each panel (boxes 128 loci x 128 queries)
    // reference operand of each panel: boxes of 128 bytes x BN refs (BN/2 when
    // paired), or, for PK launches, packed boxes of 2 (FP8) or 4 (FP4) words
    // x BN refs
    CUtensorMap b[TC_MAXP];
};

struct TensorArgs {
    int32_t n_panels;
    PanelDesc panel[TC_MAXP];
    int32_t order[TC_MAXP];  // panels in the order every group walks them
    uint32_t threshold;    // already clamped to <= N
    int32_t k;
    int32_t epi;
    void *out;  // EPI_SCORES*: panel 0's [n_q][ld_out]
    int64_t ld_out;
    int64_t capacity;  // EPI_HITS: panel 0
    int64_t *hit_q;
    int64_t *hit_r;
    uint32_t *hit_score;
    unsigned long long *hit_count;
    uint64_t *partial;  // EPI_TOPK: [slots][k][128], see TcSched
    uint32_t *status;
    unsigned int *arrive;  // panel-entry counters (see the producer), or nullptr
};

// The 4 MMAs of one 128-byte K stage into accumulator d: operand descriptors
// +0, +2, +4, +6 (32 bytes of K each in the address field), the first MMA
// accumulating only when acc != 0, the others always; one asm block with its
// predicates set once, issued by the warp's elected lane.  At FP4 speed a
// stage is ~450 cycles of MMA work and the tensor pipe holds little more
// than one MMA in its queue, so the issuer's own path between stages (wait,
// descriptors, commit) must stay within about one MMA's time.
template <bool F4, bool CG2>
__device__ __forceinline__ void mma_stage4(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t sfa,
                                           uint32_t sfb, uint32_t acc) {
    const uint64_t a1 = ad + 2u, a2 = ad + 4u, a3 = ad + 6u, b1 = bd + 2u, b2 = bd + 4u, b3 = bd + 6u;
    if constexpr (F4) {
#define FASTID_MMA4_F4(CG)                                                                                         \
    asm volatile("{\n\t.reg .pred p, q, e;\n\t" FASTID_ELECT                                                                    \
                 "setp.ne.b32 p, %12, 0;\n\t"                                                                  \
                 "setp.ne.b32 q, %12, 0xFFFFFFFF;\n\t"                                                         \
                 "@e tcgen05.mma.cta_group::" CG ".kind::mxf4.block_scale.scale_vec::2X [%0], %1, %5, %9, [%10], [%11], p;\n\t" \
                 "@e tcgen05.mma.cta_group::" CG ".kind::mxf4.block_scale.scale_vec::2X [%0], %2, %6, %9, [%10], [%11], q;\n\t" \
                 "@e tcgen05.mma.cta_group::" CG ".kind::mxf4.block_scale.scale_vec::2X [%0], %3, %7, %9, [%10], [%11], q;\n\t" \
                 "@e tcgen05.mma.cta_group::" CG ".kind::mxf4.block_scale.scale_vec::2X [%0], %4, %8, %9, [%10], [%11], q;\n\t}" \
                 ::"r"(d), "l"(ad), "l"(a1), "l"(a2), "l"(a3), "l"(bd), "l"(b1), "l"(b2), "l"(b3), "r"(idesc),      \
                 "r"(sfa), "r"(sfb), "r"(acc)                                                                     \
                 : "memory")
        if constexpr (CG2)
            FASTID_MMA4_F4("2");
        else
            FASTID_MMA4_F4("1");
#undef FASTID_MMA4_F4
    } else {
        (void)sfa;
        (void)sfb;
#define FASTID_MMA4_F8(CG)                                                                                         \
    asm volatile("{\n\t.reg .pred p, q, e;\n\t" FASTID_ELECT                                                                    \
                 "setp.ne.b32 p, %10, 0;\n\t"                                                                  \
                 "setp.ne.b32 q, %10, 0xFFFFFFFF;\n\t"                                                         \
                 "@e tcgen05.mma.cta_group::" CG ".kind::f8f6f4 [%0], %1, %5, %9, p;\n\t"                          \
                 "@e tcgen05.mma.cta_group::" CG ".kind::f8f6f4 [%0], %2, %6, %9, q;\n\t"                          \
                 "@e tcgen05.mma.cta_group::" CG ".kind::f8f6f4 [%0], %3, %7, %9, q;\n\t"                          \
                 "@e tcgen05.mma.cta_group::" CG ".kind::f8f6f4 [%0], %4, %8, %9, q;\n\t}"                         \
                 ::"r"(d), "l"(ad), "l"(a1), "l"(a2), "l"(a3), "l"(bd), "l"(b1), "l"(b2), "l"(b3), "r"(idesc),      \
                 "r"(acc)                                                                                         \
                 : "memory")
        if constexpr (CG2)
            FASTID_MMA4_F8("2");
        else
            FASTID_MMA4_F8("1");
#undef FASTID_MMA4_F8
    }
}

// Per-thread top-k list held in registers, ascending by score; entries of
// equal score keep arrival order (references arrive in increasing order, so
// the earlier entry has the lower index).  Inserting (xs, xr) is a fixed
// compare-select network, so all lanes of a warp insert in lock-step; a lane
// with nothing to insert passes xs = INT32_MAX, which changes nothing.
// The network has KM slots (16 or 32, chosen per launch from k).  For a
// runtime k <= KM the first KM - k slots hold INT32_MIN place-holders that
// nothing displaces, so the k kept entries sit in slots KM-k .. KM-1 and the
// k-th smallest is always slot KM-1 (static register indices only).
constexpr int TC_KMAX = 32;
constexpr int32_t NET_HOLD = (int32_t)0x80000000;

template <int KM>
__device__ __forceinline__ void net_insert(int32_t (&ls)[KM], uint32_t (&lr)[KM], int32_t xs, uint32_t xr) {
#pragma unroll
    for (int i = KM - 1; i > 0; --i) {
        const bool shift = xs < ls[i - 1];
        const bool here = xs < ls[i];
        ls[i] = shift ? ls[i - 1] : (here ? xs : ls[i]);
        lr[i] = shift ? lr[i - 1] : (here ? xr : lr[i]);
    }
    const bool first = xs < ls[0];
    ls[0] = first ? xs : ls[0];
    lr[0] = first ? xr : lr[0];
}

// Candidate queues.  A candidate (a score that beats its query's current
// cut) goes to its query's queue in shared memory -- score in the high bits,
// reference relative to a window of TC_QSPAN in the low ones -- and the 32
// lanes of a warp insert their queues together when one of them is full.
// Inserting each candidate on arrival ran the 80 to 160 instructions of
// net_insert for one lane's candidate while the other 31 had none: with short
// streams, whose lists are still filling, that took most of a launch (a block
// of 131,072 references against 2048 queries, k = 32: 737 us, of which the
// MMAs are 107).  Entries leave in arrival order, so equal scores still keep
// the lower reference first; one that no longer beats the list changes
// nothing.  The cut is that of the last insertion, so a deeper queue lets more
// late candidates in: with k = 16 and 8 entries about a fifth more.
// Adding a column: its entry is stored after the queue's last, and the queue
// grows by it if it beats the cut -- without a predicate, whose latency is the
// longest of the steps, and without a branch.  While lists of short streams
// fill, a third of the 32-column chunks hold a candidate or two, and one warp
// a scheduler issues all of it; with the chunk's 32 columns unrolled such a
// chunk took 830 cycles, mostly fetching instructions, which was half of the
// launch; a short loop over groups of 4 columns, re-read from TMEM, takes 500
// (FP4, k = 16, no threshold: 1792 queries x 250,000 references N = 512 329 ->
// 261 us, N = 2048 362 -> 309; 512 x 1M N = 1024 312 -> 260; 2048 x 2M 2010 ->
// 1936; the FP8 form, MMA-bound at 500 x 2M: 1029 -> 1015).  The score leaves FP32 as the
// low bits of score + 2^23, which the shift leaves alone in the high bits.
constexpr uint32_t SCORE_MAGIC = 0x4B000000u;  // 2^23

// The sign of d - cut: an infinite cut keeps its sign, and no d is NaN.
__device__ __forceinline__ uint32_t queue_step(float d, float cut) {
    return (__float_as_uint(d - cut) >> 31) * (TC_BM * 4);
}

__device__ __forceinline__ float min3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
template <int N, class T>
__device__ __forceinline__ float group_min(const T *v) {
    float t[N];
#pragma unroll
    for (int j = 0; j < N; ++j) t[j] = __builtin_bit_cast(float, v[j]);
#pragma unroll
    for (int n = N; n > 1; n = (n + 2) / 3) {
#pragma unroll
        for (int j = 0; j < (n + 2) / 3; ++j)
            t[j] = 3 * j + 2 < n ? min3(t[3 * j], t[3 * j + 1], t[3 * j + 2])
                                 : 3 * j + 1 < n ? fminf(t[3 * j], t[3 * j + 1]) : t[3 * j];
    }
    return t[0];
}

template <int KM>
__device__ __forceinline__ void queue_insert(const uint32_t *queue, int queued, int64_t qbase, int32_t (&ls)[KM],
                                             uint32_t (&lr)[KM]) {
    const int n = (int)__reduce_max_sync(0xffffffffu, (uint32_t)queued);
    for (int i = 0; i < n; ++i) {
        int32_t xs = NET_EMPTY;
        uint32_t xr = 0u;
        if (i < queued) {
            const uint32_t e = queue[i * TC_BM];
            xs = (int32_t)(e >> TC_QBITS);
            xr = (uint32_t)qbase + (e & (uint32_t)(TC_QSPAN - 1));
        }
        if (__any_sync(0xffffffffu, xs < ls[KM - 1])) net_insert(ls, lr, xs, xr);
    }
}

// The need-th smallest of a group's published bounds (see TcLaunch::gcut) for
// this lane's query row: n values at stride ld, the first TC_UNION of them.
// A slice's own k-th is the k-th of what that slice has seen; the union's is
// near the k-th of what all of them have, so with b slices the lists fill with
// a b-th of the candidates.  Read and sorted (1000 cycles, 16 loads at once)
// only at the tile after a flush.  Measured, k = 16, no threshold, FP4: 1792
// queries x 250,000 references, N = 512 399 -> 329 us, N = 2048 424 -> 362;
// 2048 queries x 2M, N = 2048 2140 -> 2010; 500 x 2M 703 -> 604.
__device__ __forceinline__ int32_t union_cut(const int32_t *pub, int64_t ld, int n, int need) {
    int32_t u[TC_UNION];
#pragma unroll
    for (int i = 0; i < TC_UNION; ++i) u[i] = i < n ? load_cut(pub + i * ld) : NET_EMPTY;
#pragma unroll
    for (int size = 2; size <= TC_UNION; size *= 2)
#pragma unroll
        for (int step = size / 2; step > 0; step /= 2)
#pragma unroll
            for (int i = 0; i < TC_UNION; ++i) {
                const int j = i ^ step;
                if (j <= i) continue;
                const int32_t lo = min(u[i], u[j]), hi = max(u[i], u[j]);
                u[i] = (i & size) == 0 ? lo : hi;
                u[j] = (i & size) == 0 ? hi : lo;
            }
    int32_t x = u[0];  // (u ascends)
#pragma unroll
    for (int i = 1; i < TC_UNION; ++i) x = max(x, i < need ? u[i] : u[0]);
    return x;
}

struct TcSmem {
    uint64_t full[8];
    uint64_t empty[8];
    uint64_t bfull[8];  // PK: reference stage expanded
    uint64_t tfull[2];
    uint64_t tempty[2];
    uint64_t done;
    uint32_t tmem_base;
    int abort_flag;
};

// Writes a warp's 32 x 32 block of full-matrix scores (v: lane's operand row,
// 32 columns) with rows of the output written whole.  Each lane storing its
// own row touched 32 rows an instruction, 2 or 4 useful bytes of every
// 32-byte sector; through the transpose buffer an instruction writes whole
// 64-byte (uint16) or 128-byte (uint32) row segments (500 x 60,001 uint32 at
// N = 1500, 120 MB: 209 -> 56 us a call): 16-byte stores where every row
// starts on a 16-byte boundary (vec), else a column a lane.
// out: the block's first element; row_step: bytes between the warp's rows;
// rows, cols: live rows and columns.  One warp a scheduler issues all of it,
// so the loops carry pointers instead of indices (108 us with an index and a
// bounds check a row), and the score leaves FP32 as the low bits of
// score + 2^23 (exact: 0 <= score <= 65536).
template <int ESZ>
__device__ __forceinline__ void store_scores(uint8_t *out, int64_t row_step, int rows, int cols, bool vec,
                                             uint32_t *buf, const uint32_t (&v)[32], float cq, int lane) {
    constexpr uint32_t MAGIC = SCORE_MAGIC;
    const float cm = cq + __uint_as_float(MAGIC);
    __syncwarp();  // the previous block's reads are done
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        uint4 o;
        o.x = __float_as_uint(__uint_as_float(v[j]) + cm) - MAGIC;
        o.y = __float_as_uint(__uint_as_float(v[j + 1]) + cm) - MAGIC;
        o.z = __float_as_uint(__uint_as_float(v[j + 2]) + cm) - MAGIC;
        o.w = __float_as_uint(__uint_as_float(v[j + 3]) + cm) - MAGIC;
        *reinterpret_cast<uint4 *>(buf + lane * SC_LD + j) = o;
    }
    __syncwarp();
    if (vec && cols >= 32) {
        constexpr int LPR = 2 * ESZ;       // lanes a row segment of 16-byte stores
        constexpr int RPI = 32 / LPR;      // rows an instruction
        const int r0 = lane / LPR, c = lane % LPR;
        uint8_t *p = out + r0 * row_step + c * 16;
        const uint32_t *b = buf + r0 * SC_LD + c * (16 / ESZ);
#pragma unroll
        for (int i = 0; i < 32 / RPI; ++i) {
            if (r0 + i * RPI < rows) {
                uint4 x = *reinterpret_cast<const uint4 *>(b + i * RPI * SC_LD);
                if (ESZ == 2) {
                    const uint4 y = *reinterpret_cast<const uint4 *>(b + i * RPI * SC_LD + 4);
                    x = make_uint4(x.x | (x.y << 16), x.z | (x.w << 16), y.x | (y.y << 16), y.z | (y.w << 16));
                }
                *reinterpret_cast<uint4 *>(p) = x;
            }
            p += RPI * row_step;
        }
    } else if (lane < cols) {
        uint8_t *p = out + lane * ESZ;
        const uint32_t *b = buf + lane;
        if (rows == 32) {
#pragma unroll
            for (int i = 0; i < 32; ++i, p += row_step) {
                if (ESZ == 2)
                    *reinterpret_cast<uint16_t *>(p) = (uint16_t)b[i * SC_LD];
                else
                    *reinterpret_cast<uint32_t *>(p) = b[i * SC_LD];
            }
        } else {
            for (int i = 0; i < rows; ++i, p += row_step) {
                if (ESZ == 2)
                    *reinterpret_cast<uint16_t *>(p) = (uint16_t)b[i * SC_LD];
                else
                    *reinterpret_cast<uint32_t *>(p) = b[i * SC_LD];
            }
        }
    }
}

// Panel-entry rendezvous.  Groups that share a reference slice read its
// tiles through L2 only while they walk it in step; entering a panel at
// different times (the previous panel's drift) breaks that.  So each CTA's
// producer counts itself in at every panel after the first and, if it has
// work there, waits for the whole grid before loading the panel's tiles.
// It is a hint, not a barrier the results depend on: the wait gives up
// after RENDEZVOUS_NS (a CTA that is not resident, or one that aborted) and
// the producer goes on alone.
__device__ __forceinline__ void panel_rendezvous(unsigned int *ctr, bool wait) {
    atomicAdd(ctr, 1u);
    if (!wait) return;
    const unsigned int n = gridDim.x;
    const uint64_t t0 = globaltimer();
    for (;;) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= n || globaltimer() - t0 > RENDEZVOUS_NS) return;
        __nanosleep(200);
    }
}

// The work of one group (see TcSched) in panel p: reference tiles
// [r_lo, r_hi) walked in chunks, query tiles (pairs) [q_lo, q_hi), top-k
// slots from slot (this CTA's first; one per query tile).  Empty
// (q_lo == q_hi) when the panel's grid and tail have no group wg.
struct GroupWork {
    int64_t r_lo, r_hi;
    int32_t q_lo, q_hi, chunk;
    int64_t slot;
    int32_t slice;  // reference slice: y, or b for the tail
};

// cpg: CTAs per group (2 when paired), rank: this CTA's rank in its group.
__device__ __forceinline__ GroupWork group_work(const TensorArgs &a, int64_t wg, int p, int cpg, int rank) {
    GroupWork w;
    w.r_lo = w.r_hi = 0;
    w.q_lo = w.q_hi = 0;
    w.chunk = 1;
    w.slot = 0;
    w.slice = 0;
    const TcSched &sc = a.panel[p].sc;
    const int64_t grid = (int64_t)sc.a * sc.b;
    if (sc.n_qq <= 0) return w;
    if (wg < grid) {
        const int64_t x = wg / sc.b, y = wg - x * sc.b;
        w.r_lo = y * (int64_t)sc.r_main / sc.b;
        w.r_hi = (y + 1) * (int64_t)sc.r_main / sc.b;
        w.q_lo = (int32_t)(x * sc.tpx);
        w.q_hi = (int32_t)min((int64_t)sc.n_qq, (x + 1) * sc.tpx);
        w.chunk = sc.chunk;
        w.slot = (int64_t)sc.slot0 + (wg * cpg + rank) * sc.tpx;
        w.slice = (int32_t)y;
    } else if (wg < grid + sc.t_groups) {
        const int64_t t = wg - grid;
        w.r_lo = sc.r_main;
        w.r_hi = a.panel[p].n_rt;
        w.q_lo = (int32_t)min((int64_t)sc.n_qq, t * sc.t_tpx);
        w.q_hi = (int32_t)min((int64_t)sc.n_qq, (t + 1) * sc.t_tpx);
        w.chunk = sc.t_chunk;
        w.slot = (int64_t)sc.slot0 + grid * cpg * sc.tpx + (t * cpg + rank) * sc.t_tpx;
        w.slice = sc.b;
    }
    return w;
}

// Appends the hits in a warp's queues (entries as in queue_insert) to the hit
// list: one atomicAdd for all of them, then an entry of every lane at a time.
// Hits take the same way to the queues as top-k candidates; appended chunk by
// chunk, each waited for an atomic on the list's counter and ran code unrolled
// over the columns (512 queries x 1M references, N = 1024, 0.6 hits a chunk:
// a call 226 -> 212 us).
__device__ __forceinline__ void append_hits(const TensorArgs &args, const uint32_t *queue, int queued, int64_t qbase,
                                            int64_t q, int lane) {
    const uint32_t total = __reduce_add_sync(0xffffffffu, (uint32_t)queued);
    if (total == 0u) return;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(args.hit_count, (unsigned long long)total);
    base = __shfl_sync(0xffffffffu, base, 0);
    const int n = (int)__reduce_max_sync(0xffffffffu, (uint32_t)queued);
    for (int i = 0; i < n; ++i) {
        const uint32_t b = __ballot_sync(0xffffffffu, i < queued);
        const unsigned long long pos = base + __popc(b & ((1u << lane) - 1u));
        base += __popc(b);
        if (i < queued && pos < (unsigned long long)args.capacity) {
            const uint32_t e = queue[i * TC_BM];
            args.hit_q[pos] = q;
            args.hit_r[pos] = qbase + (e & (uint32_t)(TC_QSPAN - 1));
            args.hit_score[pos] = e >> TC_QBITS;
        }
    }
}

// Save / resume one thread's top-k list.  Slot layout [slot][k][128]: entry i
// of the 128 rows is contiguous, so a warp's accesses coalesce.  Keys
// ascending, empty entries KEY_EMPTY.
template <int KM>
__device__ __forceinline__ void list_save(uint64_t *slot_row, const int32_t (&ls)[KM], const uint32_t (&lr)[KM],
                                          int k) {
#pragma unroll
    for (int i = 0; i < KM; ++i)
        if (i >= KM - k)
            slot_row[(int64_t)(i - (KM - k)) * TC_BM] =
                ls[i] == NET_EMPTY ? KEY_EMPTY : make_key((uint32_t)ls[i], lr[i]);
}

template <int KM>
__device__ __forceinline__ void list_load(const uint64_t *slot_row, int32_t (&ls)[KM], uint32_t (&lr)[KM], int k) {
#pragma unroll
    for (int i = 0; i < KM; ++i) {
        if (i >= KM - k) {
            const uint64_t key = slot_row[(int64_t)(i - (KM - k)) * TC_BM];
            ls[i] = key == KEY_EMPTY ? NET_EMPTY : (int32_t)(key >> 32);
            lr[i] = (uint32_t)key;
        } else {
            ls[i] = NET_HOLD;
            lr[i] = 0xFFFFFFFFu;
        }
    }
}

// PK launches: the reference operand arrives packed (TC_P_BYTES per stage,
// row r at r * 16 bytes: loci 0-63 then 64-127 of the stage) and warps 6.. (pk_threads)
// expand it into the FP8 stage the MMA reads.  A reference "1" is e4m3 2.0
// (byte 0x40) and the query operand is encoded at half scale (+-0.5), so D is
// unchanged.
//
// Locus order.  D sums over loci, so both operands may list the loci of a
// 32-locus group in any common order.  PK uses the order that makes expansion
// cheapest: byte 4j + k of the group holds locus 8k + j (j = 0..7, k = 0..3).
// Then the four bytes 4j .. 4j+3 are bit j of each byte of the group's packed
// word w, moved to bit 6 by one shift and kept by one mask:
// (w << (6 - j)) & 0x40404040 (no other bit reaches a bit 6).  The query
// operand of PK launches is written in the same order (encode_query_row).
// The stage layout is the TMA's 128-byte swizzle: 16-byte chunk c of row r
// sits at r * 128 + ((c ^ (r & 7)) << 4) from a 1024-byte aligned base.
constexpr uint32_t PK_BIT6 = 0x40404040u;

template <int NT>
__device__ __forceinline__ void expand_stage(const uint8_t *sp, uint8_t *sb, int t) {
#pragma unroll
    for (int rr = 0; rr < 256 / NT; ++rr) {
        const int r = t + NT * rr;
        const uint2 lo = *reinterpret_cast<const uint2 *>(sp + r * 16);
        const uint2 hi = *reinterpret_cast<const uint2 *>(sp + r * 16 + 8);
        const uint32_t w[4] = {lo.x, lo.y, hi.x, hi.y};  // 32 loci each
#pragma unroll
        for (int m = 0; m < 4; ++m) {  // chunks 2m (j = 0..3) and 2m + 1 (j = 4..7) of group m
            const uint32_t x = w[m];
            const uint4 o0 = make_uint4((x << 6) & PK_BIT6, (x << 5) & PK_BIT6, (x << 4) & PK_BIT6,
                                        (x << 3) & PK_BIT6);
            const uint4 o1 = make_uint4((x << 2) & PK_BIT6, (x << 1) & PK_BIT6, x & PK_BIT6, (x >> 1) & PK_BIT6);
            *reinterpret_cast<uint4 *>(sb + r * 128 + (((2 * m) ^ (r & 7)) << 4)) = o0;
            *reinterpret_cast<uint4 *>(sb + r * 128 + (((2 * m + 1) ^ (r & 7)) << 4)) = o1;
        }
    }
}

// FP4 (PK launches): the stage holds 256 loci of each reference row (4
// packed words, row r at r * 32 bytes) and each 32-locus word becomes one
// 16-byte chunk of e2m1 nibbles, in the same 128-byte swizzle.  Locus order
// inside a chunk: nibble n of its 32-bit word j holds locus 4n + j, so word j
// is bit j of every nibble of the packed word w moved to bit 1 (e2m1 +1.0 =
// 0x2) by one shift and kept by one mask.  The query operand of every FP4
// launch is written in the same order (encode_query_row_f4), and so is the
// database's FP4 copy (refs_e2m1_kernel).
constexpr uint32_t PK4_BIT1 = 0x22222222u;

// Work unit u = one half row (row u / 2, words 4 (u % 2) .. 4 (u % 2) + 3),
// so that a warp reads 512 consecutive bytes of the packed stage -- a thread
// per row read at a 32-byte stride and took twice the shared-memory
// wavefronts -- and each 16-byte chunk store of a warp still meets every bank
// group four times; a thread's loads all go first.  (64 queries x 20M:
// 2.21 -> 2.07 ms at k = 16, 2.83 -> 2.40 ms at k = 32.)
template <int NT, int BN>
__device__ __forceinline__ void expand_stage_f4(const uint8_t *sp, uint8_t *sb, int t) {
    constexpr int ITER = (2 * BN + NT - 1) / NT;
    uint4 xs[ITER];  // every load first, so that their latencies overlap
#pragma unroll
    for (int it = 0; it < ITER; ++it) {
        const int u = t + it * NT;
        if (u < 2 * BN) xs[it] = *reinterpret_cast<const uint4 *>(sp + u * 16);
    }
#pragma unroll
    for (int it = 0; it < ITER; ++it) {
        const int u = t + it * NT;
        if (u >= 2 * BN) break;
        const int r = u >> 1, h = u & 1;
        const uint4 x4 = xs[it];
        const uint32_t w[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = 4 * h + i;
            const uint32_t x = w[i];
            const uint4 o = make_uint4((x << 1) & PK4_BIT1, x & PK4_BIT1, (x >> 1) & PK4_BIT1, (x >> 2) & PK4_BIT1);
            *reinterpret_cast<uint4 *>(sb + r * 128 + ((c ^ (r & 7)) << 4)) = o;
        }
    }
}

// PAIR: 2-CTA clusters; both CTAs walk the same reference tiles for the two
// query tiles of a pair (rank r takes tile 2 qq + r), and each multicasts half
// of every reference stage into both CTAs' shared memory.
// PK: packed reference operand expanded on chip (see expand_stage).
// F4: block-scaled FP4 operands (kind::mxf4, BN = 224); else FP8 (BN = 256 or 128).
// CG2 (with PAIR): the pair's MMA is one 2-SM tcgen05.mma (cta_group::2, M =
// 256) issued by the even CTA: each CTA loads its own query tile and HALF of
// every reference stage into its own shared memory (no multicast), the
// tensor cores of both SMs read both halves, and each CTA's TMEM receives
// its own 128 query rows x BN references.  A stage then costs each SM 16 KB
// of queries + BN/2 references' bytes instead of the whole reference stage,
// which leaves room for 7 stages.  Both CTAs' loads complete on the even
// CTA's full barrier; its commits release both CTAs' stages and accumulators;
// both epilogues release an accumulator on the even CTA's barrier.
// MODE: full-matrix launches (EPI_SCORES*) store through the transpose buffers
// of store_scores; the others filter into top-k lists or hits.
template <int BN, bool PAIR, int KM, bool PK, bool F4, bool CG2 = false, int MODE = MODE_TOPK>
__global__ void __launch_bounds__(tc_threads(KM, PK, TcShape<BN, PK, CG2, MODE>::ES), 1)
    tensor_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ TensorArgs args) {
    using S = TcShape<BN, PK, CG2, MODE>;
    constexpr bool SC = MODE == MODE_SCORES;
    constexpr bool topk = MODE == MODE_TOPK;
    static_assert(topk || (KM == 16 && !CG2 && BN != 128), "full-matrix and hit launches: the single-call shapes");
    static_assert(!CG2 || (PAIR && !PK), "2-SM MMA launches are paired, over an operand copy");
    static_assert(F4 ? BN == TC_BN4 : BN != TC_BN4, "FP4 launches use 224-reference tiles, FP8 ones 256 or 128");
    static_assert(!PAIR || BN != 128, "paired launches use 256- or 224-reference tiles");
    static_assert(!PK || (BN != 128 && !PAIR), "packed-reference launches use unpaired 256- or 224-reference tiles");
    constexpr uint32_t P_BYTES = pk_stage_bytes(BN, F4);
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned operand stages (queries, references, and for PK the
    // packed reference stages), then the control block, then staging.
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
    uint8_t *base = smem_raw + pad;
    uint8_t *sA = base;
    uint8_t *sB = base + S::STAGES * TC_A_BYTES;
    uint8_t *sP = base + S::STAGES * (TC_A_BYTES + S::B_BYTES);  // PK only
    uint8_t *sT = sP + (PK ? S::STAGES * P_BYTES : 0);  // transpose buffers or candidate queues
    TcSmem *ctl = reinterpret_cast<TcSmem *>(sT + S::EX_BYTES);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int64_t c = blockIdx.x;                     // this CTA: owner of top-k slots
    const int rank = PAIR ? (int)cluster_rank() : 0;
    const int64_t wg = PAIR ? (c >> 1) : c;            // work group: cluster or CTA
    volatile int *abort_flag = &ctl->abort_flag;

    if (tid == 0) {
        for (int s = 0; s < S::STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            // multicast pairs: both CTAs' MMAs release a stage; 2-SM pairs: the even CTA's MMA
            mbar_init(smem_u32(&ctl->empty[s]), (PAIR && !CG2) ? 2 : 1);
            if (PK) mbar_init(smem_u32(&ctl->bfull[s]), pk_threads(KM));  // every expanding thread
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&ctl->tfull[a]), 1);
            mbar_init(smem_u32(&ctl->tempty[a]), CG2 ? 256 : 128);  // 2-SM: both CTAs' epilogues
        }
        mbar_init(smem_u32(&ctl->done), 1);
        ctl->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if (CG2) {  // one warp of each CTA of the pair, together: the same columns in both
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&ctl->tmem_base)),
                         "r"(S::TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&ctl->tmem_base)),
                         "r"(S::TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();  // the peer's barriers exist before any multicast targets them
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (F4) {
        // unit scale factors: TMEM columns TC_SF_COL .. TC_SF_COL + 63 of every
        // lane (each epilogue warp fills its lane quadrant) before any MMA
        if (warp >= 2 && warp < 6) {
            const uint32_t t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + TC_SF_COL;
#pragma unroll
            for (int c = 0; c < 64; c += 16) tmem_fill16(t + c, TC_SF_UNIT);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }

    pdl_wait();  // (everything up to here ran beside the query preparation)

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        // Per stage: one wait for the slot (inline when it is already free),
        // the expected bytes, the loads at stage offsets from the first slot and
        // coordinates fixed per reference tile (a short path, like the MMA
        // issuer's, so that the producer keeps up at FP4 speed).
        if (lane == 0) {
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB), sP0 = smem_u32(sP);
            // this CTA's reference rows of a (paired) tile start at rt * BN + boff
            const int32_t boff = PAIR ? rank * (BN / 2) : 0;
            // bytes landing on a full barrier: 2-SM pairs count both CTAs' loads
            // on the even CTA's; multicast pairs both halves on each CTA's
            constexpr uint32_t TX = CG2 ? 2 * (TC_A_BYTES + S::B_BYTES) : TC_A_BYTES + (PK ? P_BYTES : S::B_BYTES);
            uint32_t stage = 0;
            uint32_t phase = 0;
            int64_t issued = 0;
            bool ok = true;
            for (int pi = 0; pi < args.n_panels && ok; ++pi) {
                const int p = args.order[pi];
                const GroupWork W = group_work(args, wg, p, PAIR ? 2 : 1, rank);
                if (pi > 0 && args.arrive) panel_rendezvous(args.arrive + pi, W.q_lo < W.q_hi);
                if (W.q_lo >= W.q_hi) continue;
                const CUtensorMap *ma = &maps.a[p];
                const CUtensorMap *mb = &maps.b[p];
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(ma)) : "memory");
                asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mb)) : "memory");
                const int n_kb = args.panel[p].n_kb;
                const bool pf = args.panel[p].sc.pf != 0 && W.q_hi - W.q_lo == 1;
                for (int64_t rc = W.r_lo; rc < W.r_hi && ok; rc += W.chunk) {
                    const int64_t re = min(rc + W.chunk, W.r_hi);
                    for (int32_t qq = W.q_lo; qq < W.q_hi && ok; ++qq) {
                        const int32_t ya = (int32_t)((PAIR ? 2 * (int64_t)qq + rank : (int64_t)qq) * TC_BM);
                        for (int64_t rt = rc; rt < re && ok; ++rt) {
                            const int32_t yb = (int32_t)(rt * BN) + boff;
                            // A group with one query tile streams its slice once: fetch the
                            // next reference tile into L2 while this one is consumed, so the
                            // group that reaches a tile first does not wait on DRAM (where
                            // the schedule enables it, see TcSched::pf).
                            const bool pft = !PK && pf && rt + 1 < W.r_hi;
                            for (int kb = 0; kb < n_kb; ++kb) {
                                const uint32_t eb = empty0 + 8u * stage;
                                if (!mbar_try_wait(eb, phase ^ 1u)) {
                                    ok = mbar_wait(eb, phase ^ 1u, abort_flag, args.status, 1);
                                    if (!ok) break;
                                }
                                const uint32_t fb = full0 + 8u * stage;
                                const int32_t x = kb * TC_BK;
                                if (CG2) {
                                    // both CTAs' bytes complete on the even CTA's full barrier
                                    const uint32_t fb0 = mapa_rank(fb, 0);
                                    if (rank == 0) mbar_expect_tx(fb, TX);
                                    tma_load_2d_cg2(sA0 + stage * TC_A_BYTES, ma, fb0, x, ya);
                                    tma_load_2d_cg2(sB0 + stage * S::B_BYTES, mb, fb0, x, yb);
                                } else {
                                    mbar_expect_tx(fb, TX);
                                    tma_load_2d(sA0 + stage * TC_A_BYTES, ma, fb, x, ya);
                                    if (PK)  // the stage's loci as packed words (2 FP8, 4 FP4) x BN references
                                        tma_load_2d(sP0 + stage * P_BYTES, mb, fb, kb * (F4 ? 4 : 2), yb);
                                    else if (PAIR)  // this CTA's half, into both CTAs
                                        tma_load_2d_mc(sB0 + stage * S::B_BYTES + rank * (S::B_BYTES / 2), mb, fb, x, yb,
                                                       (uint16_t)0x3);
                                    else
                                        tma_load_2d(sB0 + stage * S::B_BYTES, mb, fb, x, yb);
                                }
                                if (pft) tma_prefetch_2d(mb, x, yb + BN);
                                ++issued;
                                if (++stage == S::STAGES) {
                                    stage = 0;
                                    phase ^= 1u;
                                }
                            }
                        }
                    }
                }
            }
            // Drain: the last fill of every stage has landed before the CTA
            // exits (fill n used stage n % S in phase (n / S) & 1).
            for (int64_t n = issued - 1; n >= 0 && n >= issued - S::STAGES; --n) {
                // (2-SM pairs: the even CTA's full barriers count both CTAs' fills)
                if (!CG2 || rank == 0)
                    mbar_drain(smem_u32(&ctl->full[n % S::STAGES]), (uint32_t)((n / S::STAGES) & 1), args.status, 2);
                // paired: both MMAs' releases of this stage (the peer's arrive
                // remotely) have landed before the CTA exits
                if (PAIR)
                    mbar_drain(smem_u32(&ctl->empty[n % S::STAGES]), (uint32_t)((n / S::STAGES) & 1), args.status, 7);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (2-SM pairs: the even CTA's) ----------------
        // The whole warp, converged; one elected lane issues (see tc_commit).
        // The lanes vote on every wait (warp_wait): where one ran out, all of
        // them leave together, and none is left at an elect.sync that the
        // others never reach.
        // Per stage: one barrier wait (inline when the stage is already full),
        // the stage's descriptors as constant offsets from the first stage's,
        // four MMAs in one asm block, one commit (see mma_stage4).
        if (!CG2 || rank == 0) {
            constexpr int MM = CG2 ? 2 * TC_BM : TC_BM;
            constexpr uint32_t idesc = F4 ? idesc_mxf4(MM, BN) : idesc_f8(MM, BN);
            constexpr uint32_t A_STEP = TC_A_BYTES >> 4, B_STEP = S::B_BYTES >> 4;  // descriptor units a stage
            const uint64_t ad0 = sw128_desc(smem_u32(sA)), bd0 = sw128_desc(smem_u32(sB));
            const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            const uint32_t bfull0 = smem_u32(&ctl->bfull[0]);
            const uint32_t sfa = tmem_base + TC_SF_COL, sfb = tmem_base + TC_SF_COL + 16;
            uint32_t stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int pi = 0; pi < args.n_panels && ok; ++pi) {
                const int p = args.order[pi];
                const GroupWork W = group_work(args, wg, p, PAIR ? 2 : 1, rank);
                if (W.q_lo >= W.q_hi) continue;
                const int n_kb = args.panel[p].n_kb;
                for (int64_t rc = W.r_lo; rc < W.r_hi && ok; rc += W.chunk) {
                    const int64_t re = min(rc + W.chunk, W.r_hi);
                    for (int32_t qq = W.q_lo; qq < W.q_hi && ok; ++qq) {
                        for (int64_t rt = rc; rt < re && ok; ++rt) {
                            const uint32_t tempty = smem_u32(&ctl->tempty[acc]);
                            ok = warp_wait(tempty, acc_phase ^ 1u, abort_flag, args.status, 3);
                            if (!ok) break;
                            tc_fence_after();  // the epilogue's reads of this accumulator come first
                            const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                            for (int kb = 0; kb < n_kb; ++kb) {
                                const uint32_t fb = full0 + 8u * stage;
                                ok = warp_wait(fb, phase, abort_flag, args.status, 4);
                                if (!ok) break;
                                if (PK) {
                                    ok = warp_wait(bfull0 + 8u * stage, phase, abort_flag, args.status, 8);
                                    if (!ok) break;
                                }
                                // (the stage's operands were written by TMA, or by the expanding
                                // warps behind an async-proxy fence, and are ordered by the barrier)
                                mma_stage4<F4, CG2>(d_tmem, ad0 + stage * A_STEP, bd0 + stage * B_STEP, idesc, sfa,
                                                    sfb, kb != 0);
                                const uint32_t eb = empty0 + 8u * stage;
                                if (CG2)
                                    tc_commit_cg2_mc(eb, (uint16_t)0x3);
                                else if (PAIR)
                                    tc_commit_mc(eb, (uint16_t)0x3);
                                else
                                    tc_commit(eb);
                                if (++stage == S::STAGES) {
                                    stage = 0;
                                    phase ^= 1u;
                                }
                            }
                            if (!ok) break;
                            if (CG2)  // both CTAs' accumulators are full
                                tc_commit_cg2_mc(smem_u32(&ctl->tfull[acc]), (uint16_t)0x3);
                            else
                                tc_commit(smem_u32(&ctl->tfull[acc]));
                            if (++acc == 2) {
                                acc = 0;
                                acc_phase ^= 1u;
                            }
                        }
                    }
                }
            }
            // Drain: a commit completes after every MMA this thread issued.
            if (CG2)
                tc_commit_cg2(smem_u32(&ctl->done));
            else
                tc_commit(smem_u32(&ctl->done));
            mbar_drain(smem_u32(&ctl->done), 0, args.status, 5);
        }
    } else if (PK && warp >= 6 && warp < 6 + pk_threads(KM) / 32) {
        // ---------------- PK: reference expansion, warps 6.. ----------------
        const int t = tid - 192;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int pi = 0; pi < args.n_panels && ok; ++pi) {
            const int p = args.order[pi];
            const GroupWork W = group_work(args, wg, p, PAIR ? 2 : 1, rank);
            if (W.q_lo >= W.q_hi) continue;
            const int n_kb = args.panel[p].n_kb;
            for (int64_t rc = W.r_lo; rc < W.r_hi && ok; rc += W.chunk) {
                const int64_t re = min(rc + W.chunk, W.r_hi);
                for (int32_t qq = W.q_lo; qq < W.q_hi && ok; ++qq) {
                    for (int64_t rt = rc; rt < re && ok; ++rt) {
                        for (int kb = 0; kb < n_kb; ++kb) {
                            ok = mbar_wait(smem_u32(&ctl->full[stage]), phase, abort_flag, args.status, 9);
                            if (!ok) break;
                            if (F4)
                                expand_stage_f4<pk_threads(KM), BN>(sP + stage * P_BYTES, sB + stage * S::B_BYTES, t);
                            else
                                expand_stage<pk_threads(KM)>(sP + stage * P_BYTES, sB + stage * S::B_BYTES, t);
                            // generic-proxy writes, read next by the tensor core (async proxy)
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            mbar_arrive(smem_u32(&ctl->bfull[stage]));
                            if (++stage == S::STAGES) {
                                stage = 0;
                                phase ^= 1u;
                            }
                        }
                    }
                }
            }
        }
    } else {
        // ---------------- epilogue: warps 2..5 (and the last four) ----------------
        constexpr int ES = S::ES;
        const int set = warp < 6 ? 0 : 1;
        const int quad = warp & 3;            // TMEM lane quadrant this warp may access
        const int row = quad * 32 + lane;     // query row within the tile
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const float tplus1 = args.threshold == 0xFFFFFFFFu ? __int_as_float(0x7f800000) : (float)args.threshold + 1.0f;
        const int k = args.k;
        // every row of the output starts on a 16-byte boundary
        const bool vec = SC && (reinterpret_cast<uintptr_t>(args.out) & 15) == 0 &&
                         ((args.ld_out * (args.epi == EPI_SCORES16 ? 2 : 4)) & 15) == 0;
        int acc = set;
        uint32_t acc_phase = 0;
        int64_t tiles = 0;  // of the walk so far
        int32_t ls[KM];   // this thread's top-k scores (see net_insert)
        uint32_t lr[KM];  // and their references
        bool ok = true;
        for (int pi = 0; pi < args.n_panels && ok; ++pi) {
            const int p = args.order[pi];
            const GroupWork W = group_work(args, wg, p, PAIR ? 2 : 1, rank);
            if (W.q_lo >= W.q_hi) continue;
            const PanelDesc &P = args.panel[p];
            const int64_t n_refs = P.n_refs;
            for (int64_t rc = W.r_lo; rc < W.r_hi && ok; rc += W.chunk) {
                const int64_t re = min(rc + W.chunk, W.r_hi);
                for (int32_t qq = W.q_lo; qq < W.q_hi && ok; ++qq) {
                    const int64_t qt = PAIR ? 2 * (int64_t)qq + rank : qq;
                    const int64_t qr = qt * TC_BM + row;                     // operand row
                    const int64_t q = spread_row_to_query(qr, P.qspread);  // input query
                    const bool qvalid = q < P.n_q;
                    const float cq = P.qconst[qr];
                    const float cut0 = qvalid ? tplus1 - cq : -__int_as_float(0x7f800000);
                    // SC: the warp's output rows are q0, q0 + st, q0 + 2 st, ... (see spread_row_to_query)
                    uint8_t *sc_out = nullptr;
                    int64_t sc_step = 0;
                    int sc_rows = 0;
                    if constexpr (SC) {
                        const int64_t q0 = spread_row_to_query(qt * TC_BM + quad * 32, P.qspread);
                        const int64_t st = P.qspread <= 1 ? 1 : P.qspread;
                        const int64_t esz = args.epi == EPI_SCORES16 ? 2 : 4;
                        sc_rows = q0 < P.n_q ? (int)min((int64_t)32, (P.n_q - q0 + st - 1) / st) : 0;
                        sc_out = reinterpret_cast<uint8_t *>(args.out) + q0 * args.ld_out * esz;
                        sc_step = st * args.ld_out * esz;
                    }
                    uint64_t *slot = args.partial + (W.slot + (qq - W.q_lo)) * (int64_t)k * TC_BM + row;
                    if (topk && rc > W.r_lo) {
                        list_load(slot, ls, lr, k);
                    } else {
#pragma unroll
                        for (int i = 0; i < KM; ++i) {
                            ls[i] = i < KM - k ? NET_HOLD : NET_EMPTY;
                            lr[i] = 0xFFFFFFFFu;
                        }
                    }
                    // the cut: below this list's k-th, and not above the shared one
                    int32_t *gc = topk && P.gcut ? P.gcut + qr : nullptr;
                    int32_t shared = gc ? load_cut(gc) : NET_EMPTY, newer = shared;
                    float cut;
                    auto set_cut = [&]() {
                        cut = ls[KM - 1] == NET_EMPTY ? cut0 : (float)ls[KM - 1] - cq;
                        if (shared != NET_EMPTY) cut = fminf(cut, (float)(shared + 1) - cq);
                    };
                    const int32_t n_pub = gc ? P.n_pub : 0;
                    const int32_t win = min(W.slice / TC_UNION * TC_UNION, max(0, n_pub - TC_UNION));
                    bool due = false;  // something was published since the last union
                    auto share_cut = [&]() {
                        if (gc && ls[KM - 1] < shared) {
                            shared = ls[KM - 1];
                            atomicMin(gc, shared);
                        }
                        if (n_pub > 0) {
                            int32_t mine = ls[0];  // (ls ascends)
#pragma unroll
                            for (int i = 1; i < KM; ++i) mine = max(mine, i < KM - k + P.pub_rank ? ls[i] : ls[0]);
                            store_cut(gc + (1 + W.slice) * P.gcut_ld, mine);
                            due = true;
                        }
                    };
                    set_cut();
                    uint32_t *queue = reinterpret_cast<uint32_t *>(sT) + set * S::QD * TC_BM + row;  // entry i at i * TC_BM (see queue_insert)
                    int queued = 0;
                    int64_t qbase = rc * BN;
                    auto flush = [&]() {
                        if (topk) {
                            queue_insert(queue, queued, qbase, ls, lr);
                            share_cut();
                            set_cut();
                        } else {
                            append_hits(args, queue, queued, qbase, q, lane);
                        }
                        queued = 0;
                        __syncwarp();  // lanes took their own ways; what follows may be a whole-warp TMEM load
                    };
                    for (int64_t rt = rc + (ES == 2 ? (tiles & 1) ^ set : 0); rt < re; rt += ES) {
                        const bool got = mbar_wait(smem_u32(&ctl->tfull[acc]), acc_phase, abort_flag, args.status, 6);
                        __syncwarp();
                        if (!__all_sync(0xffffffffu, got)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const int64_t r0 = rt * BN;
                        if (gc) {  // what the other slices had reached a tile ago
                            if (newer < shared) {
                                shared = newer;
                                set_cut();
                            }
                            newer = load_cut(gc);
                        }
                        if (due) {  // (the same for the whole warp)
                            due = false;
                            const int32_t x = union_cut(gc + (1 + win) * P.gcut_ld, P.gcut_ld, n_pub - win, P.pub_need);
                            if (x < shared) {
                                shared = x;
                                atomicMin(gc, x);
                                set_cut();
                            }
                        }
                        if (!SC && r0 + BN - qbase > TC_QSPAN) {  // the queues' reference window moves on
                            flush();
                            qbase = r0;
                        }
                        const uint32_t taddr = tmem_base + lane_addr + (uint32_t)(acc * BN);
#pragma unroll 1
                        for (int ch = 0; ch < BN / 32; ++ch) {
                            uint32_t v[32];
                            __syncwarp();  // tcgen05.ld is warp-collective: reconverge first
                            tmem_ld32(taddr + ch * 32, v);
                            const int64_t rch = r0 + ch * 32;
                            if constexpr (SC) {
                                const int cols = (int)min((int64_t)32, n_refs - rch);
                                if (sc_rows > 0 && cols > 0) {
                                    uint32_t *buf = reinterpret_cast<uint32_t *>(sT) + quad * 32 * SC_LD;
                                    if (args.epi == EPI_SCORES16)
                                        store_scores<2>(sc_out + rch * 2, sc_step, sc_rows, cols, vec, buf, v, cq, lane);
                                    else
                                        store_scores<4>(sc_out + rch * 4, sc_step, sc_rows, cols, vec, buf, v, cq, lane);
                                }
                                continue;
                            }
                            // Common case first: nothing in the chunk beats the cut
                            // (the minima of its groups of G columns, and theirs).
                            constexpr int G = S::QG, NG = 32 / G;
                            float gm[NG];
#pragma unroll
                            for (int g = 0; g < NG; ++g) gm[g] = group_min<G>(v + g * G);
                            if (!__any_sync(0xffffffffu, group_min<NG>(gm) < cut)) continue;
                            // The candidates go to the queues, a group that some lane
                            // needs at a time, each re-read from TMEM by the whole
                            // warp (the accumulator is released only after the tile,
                            // below): a short loop, which stays in the instruction
                            // cache where unrolled code over the chunk's registers
                            // did not (see queue_step).
                            uint32_t left = 0;
#pragma unroll
                            for (int g = 0; g < NG; ++g) left |= (uint32_t)(gm[g] < cut) << g;
                            left = __reduce_or_sync(0xffffffffu, left);
                            const float cm = cq + __uint_as_float(SCORE_MAGIC);
#pragma unroll 1
                            while (left != 0u) {
                                const int col = (__ffs(left) - 1) * G;
                                left &= left - 1u;
                                if (__any_sync(0xffffffffu, queued > S::QD - G)) flush();
                                uint32_t w[G], step[G];
                                tmem_ld_group(taddr + ch * 32 + col, w);
                                const int64_t r = rch + col;
#pragma unroll
                                for (int j = 0; j < G; ++j)
                                    step[j] = queue_step(__uint_as_float(w[j]), cut);
                                if (r + G > n_refs) {
#pragma unroll
                                    for (int j = 0; j < G; ++j)
                                        if (r + j >= n_refs) step[j] = 0;
                                }
                                const uint32_t rel = (uint32_t)(r - qbase), at0 = smem_u32(queue);
                                uint32_t at = at0 + (uint32_t)queued * (TC_BM * 4);
#pragma unroll
                                for (int j = 0; j < G; ++j) {
                                    const uint32_t e = __float_as_uint(__uint_as_float(w[j]) + cm);
                                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"((e << TC_QBITS) + (rel + j))
                                                 : "memory");
                                    at += step[j];
                                }
                                queued = (int)((at - at0) / (TC_BM * 4));
                            }
                        }
                        // every column of the tile is processed: the MMA may reuse the accumulator
                        tc_fence_before();
                        if (CG2)  // on the even CTA's barrier
                            mbar_arrive_cluster(mapa_rank(smem_u32(&ctl->tempty[acc]), 0));
                        else
                            mbar_arrive(smem_u32(&ctl->tempty[acc]));
                        if (ES == 2) {
                            acc_phase ^= 1u;
                        } else if (++acc == 2) {
                            acc = 0;
                            acc_phase ^= 1u;
                        }
                    }
                    tiles += re - rc;
                    if (!SC && ok) {
                        flush();
                        if (topk) list_save(slot, ls, lr, k);
                    }
                }
            }
        }
    }

    pdl_trigger();
    tc_fence_before();
    __syncthreads();
    if (PAIR) cluster_sync();  // neither CTA leaves while the other may still address it
    tc_fence_after();
    if (warp == 1) {
        if (CG2)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(S::TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(S::TMEM_COLS)
                         : "memory");
    }
}

// ---- operand expansion ------------------------------------------------------

// Four bits (bit i of x) -> four bytes, byte i = 0x38 (e4m3 +1.0) or 0.
__device__ __forceinline__ uint32_t bits4_to_e4m3(uint32_t x) {
    uint32_t b = ((x & 0xFu) * 0x00204081u) & 0x01010101u;  // bit i -> byte i
    return b * 0x38u;
}

// Reference operand: byte l of row r = R_rl ? 0x38 : 0 for l < kpad, from
// packed rows at stride ld64 of which the first n_src rows and n_words words
// exist (zero elsewhere: padding rows and loci).  One thread per 16 output
// bytes; streaming loads and stores (each byte is touched once, and the
// operand is larger than L2), so that a concurrent comparison keeps its L2.
__global__ void refs_e4m3_kernel(const uint64_t *__restrict__ packed, int64_t ld64, int64_t n_src, int32_t n_words,
                                 int64_t n_rows, int32_t kpad, uint8_t *__restrict__ out) {
    const int64_t per_row = kpad / 16;
    const int64_t total = n_rows * per_row;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / per_row, c = t - r * per_row;
        const int64_t l0 = c * 16;
        const int32_t wi = (int32_t)(l0 >> 6);
        const uint64_t w = (r < n_src && wi < n_words) ? __ldcs(packed + r * ld64 + wi) : 0ull;
        const uint32_t bits = (uint32_t)(w >> (l0 & 63)) & 0xFFFFu;
        uint4 o;
        o.x = bits4_to_e4m3(bits);
        o.y = bits4_to_e4m3(bits >> 4);
        o.z = bits4_to_e4m3(bits >> 8);
        o.w = bits4_to_e4m3(bits >> 12);
        __stcs(reinterpret_cast<uint4 *>(out + r * (int64_t)kpad) + c, o);
    }
}

// Query operand per mode (see the header comment) and c_q for one row, by one
// warp.  src == nullptr (a padding row) writes zeros.
// `one` is the e4m3 byte of +1 on this operand's scale: 0x38 (1.0) against the
// FP8 reference operand, 0x30 (0.5) against PK's expanded references (2.0).
// pk: PK's locus order (see expand_stage), else loci in order.
__device__ __forceinline__ void encode_query_row(const uint64_t *__restrict__ src, bool mis, int32_t n_words,
                                                 int32_t n_loci, int32_t kpad, uint8_t *__restrict__ dst,
                                                 float *__restrict__ qc, int lane, uint32_t one = 0x38u,
                                                 bool pk = false) {
    const bool valid = src != nullptr;
    uint32_t pc = 0;
    if (pk) {
        // chunk c: words i = 0..3 hold j = 4 (c & 1) + i; byte k of word i is
        // locus 32 (c >> 1) + 8k + j
        for (int32_t c = lane; c < kpad / 16; c += 32) {
            const int32_t l0 = (c >> 1) * 32;
            uint32_t bits = 0;
            if (valid && (l0 >> 6) < n_words) bits = (uint32_t)(src[l0 >> 6] >> (l0 & 63));
            const int32_t live = n_loci - l0;
            const uint32_t in_n = !valid ? 0u : live >= 32 ? 0xFFFFFFFFu : live <= 0 ? 0u : ((1u << live) - 1u);
            bits &= in_n;
            const int32_t j0 = 4 * (c & 1);
            pc += __popc(bits & (0x0F0F0F0Fu << j0));
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t qb = (bits >> (j0 + i)) & 0x01010101u;  // Q_l, one per byte
                const uint32_t nb = (in_n >> (j0 + i)) & 0x01010101u;  // l < N
                w[i] = (nb & ~qb) * one | (mis ? qb * (one | 0x80u) : 0u);
            }
            reinterpret_cast<uint4 *>(dst)[c] = make_uint4(w[0], w[1], w[2], w[3]);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
        if (lane == 0) *qc = mis ? (float)pc : 0.f;
        return;
    }
    for (int32_t c = lane; c < kpad / 16; c += 32) {
        const int32_t l0 = c * 16;
        uint32_t bits = 0;
        if (valid && (l0 >> 6) < n_words) bits = (uint32_t)(src[l0 >> 6] >> (l0 & 63)) & 0xFFFFu;
        // loci < N inside this 16-locus group
        const int32_t live = n_loci - l0;
        const uint32_t in_n = !valid ? 0u : live >= 16 ? 0xFFFFu : live <= 0 ? 0u : ((1u << live) - 1u);
        bits &= in_n;
        pc += __popc(bits);
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t qb = (bits >> (4 * i)) & 0xFu;   // Q_l
            const uint32_t nb = (in_n >> (4 * i)) & 0xFu;   // l < N
            // mode 1: 1 - Q_l  -> +1 where l < N and Q_l = 0
            // mode 0: 1 - 2Q_l -> +1 where Q_l = 0, -1 (sign bit 0x80 set) where Q_l = 1
            const uint32_t plus = (((nb & ~qb) * 0x00204081u) & 0x01010101u) * one;
            const uint32_t minus = mis ? ((qb * 0x00204081u) & 0x01010101u) * (one | 0x80u) : 0u;
            w[i] = plus | minus;
        }
        reinterpret_cast<uint4 *>(dst)[c] = make_uint4(w[0], w[1], w[2], w[3]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
    if (lane == 0) *qc = mis ? (float)pc : 0.f;
}

// Reference operand, FP4: row r holds kbytes = (loci padded to 256) / 2
// bytes; its 16-byte chunk c covers loci 32c .. 32c + 31, in the nibble order
// of expand_stage_f4 (nibble n of 32-bit word j = locus 32c + 4n + j).  From
// packed rows at stride ld64 of which the first n_src rows and n_words words
// exist (zero elsewhere).  One thread per 16 output bytes, streaming loads and
// stores as in refs_e4m3_kernel.
__global__ void refs_e2m1_kernel(const uint64_t *__restrict__ packed, int64_t ld64, int64_t n_src, int32_t n_words,
                                 int64_t n_rows, int32_t kbytes, uint8_t *__restrict__ out) {
    const int64_t per_row = kbytes / 16;
    const int64_t total = n_rows * per_row;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / per_row, c = t - r * per_row;
        const int32_t wi = (int32_t)(c >> 1);
        const uint64_t w = (r < n_src && wi < n_words) ? __ldcs(packed + r * ld64 + wi) : 0ull;
        const uint32_t x = (uint32_t)(w >> (32 * (c & 1)));
        const uint4 o = make_uint4((x << 1) & PK4_BIT1, x & PK4_BIT1, (x >> 1) & PK4_BIT1, (x >> 2) & PK4_BIT1);
        __stcs(reinterpret_cast<uint4 *>(out + r * (int64_t)kbytes) + c, o);
    }
}

// Query operand, FP4, per mode and c_q for one row, by one warp: e2m1 +1
// (0x2) where l < N and Q_l = 0; in mode 0 also -1 (0xA) where Q_l = 1; 0
// elsewhere.  Same nibble order as the reference operand.  src == nullptr (a
// padding row) writes zeros.
__device__ __forceinline__ void encode_query_row_f4(const uint64_t *__restrict__ src, bool mis, int32_t n_words,
                                                    int32_t n_loci, int32_t kbytes, uint8_t *__restrict__ dst,
                                                    float *__restrict__ qc, int lane) {
    const bool valid = src != nullptr;
    uint32_t pc = 0;
    for (int32_t c = lane; c < kbytes / 16; c += 32) {
        const int32_t l0 = c * 32;
        uint32_t bits = 0;
        if (valid && (l0 >> 6) < n_words) bits = (uint32_t)(src[l0 >> 6] >> (l0 & 63));
        const int32_t live = n_loci - l0;
        const uint32_t in_n = !valid ? 0u : live >= 32 ? 0xFFFFFFFFu : live <= 0 ? 0u : ((1u << live) - 1u);
        bits &= in_n;
        pc += __popc(bits);
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t qb = (bits >> j) & 0x11111111u;  // Q at nibble n = locus 4n + j
            const uint32_t nb = (in_n >> j) & 0x11111111u;  // l < N
            w[j] = ((nb & ~qb) << 1) | (mis ? qb * 0xAu : 0u);
        }
        reinterpret_cast<uint4 *>(dst)[c] = make_uint4(w[0], w[1], w[2], w[3]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) pc += __shfl_xor_sync(0xffffffffu, pc, off);
    if (lane == 0) *qc = mis ? (float)pc : 0.f;
}

// Initial shared cut of operand row r, holding input query src (see SharedCut).
// Scores are at most 65536, so a larger entry of a caller's list cuts nothing.
__device__ __forceinline__ void init_cut(const SharedCut &cut, int64_t r, int64_t src, bool valid) {
    int32_t c = NET_EMPTY;
    if (valid && cut.run_s) {
        const int64_t last = src * cut.k + cut.k - 1;
        if (cut.run_i[last] >= 0 && cut.run_s[last] <= (uint32_t)FASTID_MAX_LOCI) c = (int32_t)cut.run_s[last];
    }
    cut.out[r] = c;
}
__device__ __forceinline__ void init_pub(int32_t *row, int64_t ld, int32_t n_pub, int lane) {
    for (int i = lane; i < n_pub; i += 32) row[(1 + i) * ld] = NET_EMPTY;
}

// Operand row r encodes input query spread_row_to_query(r, spread).
__global__ void queries_e2m1_kernel(const uint64_t *__restrict__ q, int64_t ld_q, int64_t n_q, int32_t n_words,
                                    int32_t n_loci, const uint8_t *__restrict__ modes, int64_t n_q_pad,
                                    int32_t kbytes, uint8_t *__restrict__ out, float *__restrict__ qconst,
                                    int64_t spread, const SharedCut cut) {
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n_q_pad; r += warps_total) {
        const int64_t src = spread_row_to_query(r, spread);
        const bool valid = src < n_q;
        if (cut.out && lane == 0) init_cut(cut, r, src, valid);
        if (cut.out) init_pub(cut.out + r, cut.ld, cut.n_pub, lane);
        encode_query_row_f4(valid ? q + src * ld_q : nullptr, valid && modes[src] == FASTID_MODE_MISMATCH, n_words,
                            n_loci, kbytes, out + r * (int64_t)kbytes, qconst + r, lane);
    }
}

__global__ void queries_e4m3_kernel(const uint64_t *__restrict__ q, int64_t ld_q, int64_t n_q, int32_t n_words,
                                    int32_t n_loci, const uint8_t *__restrict__ modes, int64_t n_q_pad,
                                    int32_t kpad, uint8_t *__restrict__ out, float *__restrict__ qconst,
                                    uint32_t one, bool pk, int64_t spread, const SharedCut cut) {
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n_q_pad; r += warps_total) {
        const int64_t src = spread_row_to_query(r, spread);
        const bool valid = src < n_q;
        if (cut.out && lane == 0) init_cut(cut, r, src, valid);
        if (cut.out) init_pub(cut.out + r, cut.ld, cut.n_pub, lane);
        encode_query_row(valid ? q + src * ld_q : nullptr, valid && modes[src] == FASTID_MODE_MISMATCH, n_words,
                         n_loci, kpad, out + r * (int64_t)kpad, qconst + r, lane, one, pk);
    }
}

// Batched form: one job per operand row of every panel.
__global__ void prep_jobs_kernel(const PrepJob *__restrict__ jobs, int64_t n_jobs) {
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < n_jobs; j += warps_total) {
        const PrepJob jb = jobs[j];
        const bool mis = jb.src != nullptr && *jb.mode == FASTID_MODE_MISMATCH;
        if (lane == 0) *jb.gc = NET_EMPTY;
        init_pub(jb.gc, jb.gc_ld, jb.n_pub, lane);
        if (jb.f4)
            encode_query_row_f4(jb.src, mis, jb.n_words, jb.n_loci, jb.kpad, jb.dst, jb.qc, lane);
        else
            encode_query_row(jb.src, mis, jb.n_words, jb.n_loci, jb.kpad, jb.dst, jb.qc, lane);
    }
}

template <int BN, bool PK = false, bool CG2 = false, int MODE = MODE_TOPK>
size_t tensor_smem(bool f4 = false) {
    using S = TcShape<BN, PK, CG2, MODE>;
    return 1024 + S::STAGES * (size_t)(TC_A_BYTES + S::B_BYTES + (PK ? pk_stage_bytes(BN, f4) : 0)) +
           S::EX_BYTES + 256;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// dependency on libcuda).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

}  // namespace

cudaError_t make_operand_map(CUtensorMap *map, const uint8_t *base, int64_t rows, int32_t kpad, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kpad};
    cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int tensor_tile_q() { return TC_BM; }
int tensor_tile_r() { return 256; }
int tensor_tile_r4() { return TC_BN4; }
int tensor_kpad(int32_t n_loci) { return (n_loci + TC_BK - 1) / TC_BK * TC_BK; }
int tensor_kbytes4(int32_t n_loci) { return (n_loci + 2 * TC_BK - 1) / (2 * TC_BK) * TC_BK; }

cudaError_t launch_refs_e2m1(const uint64_t *packed, int64_t ld64, int64_t n_src, int32_t n_words, int64_t n_rows,
                             int32_t kbytes, uint8_t *out, int max_blocks, cudaStream_t s) {
    int64_t total = n_rows * (kbytes / 16);
    int64_t blocks = (total + 255) / 256;
    if (blocks > max_blocks) blocks = max_blocks;
    if (blocks < 1) return cudaSuccess;
    refs_e2m1_kernel<<<(unsigned)blocks, 256, 0, s>>>(packed, ld64, n_src, n_words, n_rows, kbytes, out);
    return cudaGetLastError();
}

cudaError_t launch_queries_e2m1(const uint64_t *q, int64_t ld_q, int64_t n_q, int32_t n_words, int32_t n_loci,
                                const uint8_t *modes, int64_t n_q_pad, int32_t kbytes, uint8_t *out, float *qconst,
                                int64_t spread, const SharedCut &cut, cudaStream_t s) {
    int64_t blocks = (n_q_pad + 7) / 8;
    if (blocks > 65535) blocks = 65535;
    queries_e2m1_kernel<<<(unsigned)blocks, 256, 0, s>>>(q, ld_q, n_q, n_words, n_loci, modes, n_q_pad, kbytes, out,
                                                         qconst, spread, cut);
    return cudaGetLastError();
}

cudaError_t launch_refs_e4m3(const uint64_t *packed, int64_t ld64, int64_t n_src, int32_t n_words, int64_t n_rows,
                             int32_t kpad, uint8_t *out, int max_blocks, cudaStream_t s) {
    int64_t total = n_rows * (kpad / 16);
    int64_t blocks = (total + 255) / 256;
    if (blocks > max_blocks) blocks = max_blocks;
    if (blocks < 1) return cudaSuccess;
    refs_e4m3_kernel<<<(unsigned)blocks, 256, 0, s>>>(packed, ld64, n_src, n_words, n_rows, kpad, out);
    return cudaGetLastError();
}

cudaError_t launch_queries_e4m3(const uint64_t *q, int64_t ld_q, int64_t n_q, int32_t n_words, int32_t n_loci,
                                const uint8_t *modes, int64_t n_q_pad, int32_t kpad, uint8_t *out, float *qconst,
                                bool half, int64_t spread, const SharedCut &cut, cudaStream_t s) {
    int64_t blocks = (n_q_pad + 7) / 8;
    if (blocks > 65535) blocks = 65535;
    queries_e4m3_kernel<<<(unsigned)blocks, 256, 0, s>>>(q, ld_q, n_q, n_words, n_loci, modes, n_q_pad, kpad, out,
                                                         qconst, half ? 0x30u : 0x38u, half, spread, cut);
    return cudaGetLastError();
}

// PK reference operand: the packed rows [rows][ld64] uint64 themselves, in
// boxes of box_words words (2 = 128 loci for FP8 stages, 4 = 256 for FP4) x
// box_rows references, unswizzled.
cudaError_t make_packed_map(CUtensorMap *map, const uint64_t *packed, int64_t rows, int64_t ld64, int box_words,
                            int box_rows, bool swizzle64) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorNotSupported;
    cuuint64_t dims[2] = {(cuuint64_t)ld64, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld64 * 8};
    cuuint32_t box[2] = {(cuuint32_t)box_words, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<uint64_t *>(packed), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_prep_jobs(const PrepJob *jobs, int64_t n_jobs, cudaStream_t s) {
    if (n_jobs == 0) return cudaSuccess;
    int64_t blocks = (n_jobs + 7) / 8;
    if (blocks > 65535) blocks = 65535;
    prep_jobs_kernel<<<(unsigned)blocks, 256, 0, s>>>(jobs, n_jobs);
    return cudaGetLastError();
}

// Largest number of 2-CTA clusters of the paired kernel that can be resident
// at once (0 if clusters are unavailable).
int tensor_pair_clusters(int device) {
    size_t smem = tensor_smem<256>();
    if (cudaFuncSetAttribute(tensor_kernel<256, true, TC_KMAX, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(sms & ~1);
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, tensor_kernel<256, true, TC_KMAX, false, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

int tensor_grid_target(int device) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    return sms;
}

namespace {

// One launch of tensor_kernel<BN, PAIR, KM, PK, F4, CG2, MODE> over n_groups work
// groups (2-CTA clusters when paired).
template <int BN, bool PAIR, int KM, bool PK = false, bool F4 = false, bool CG2 = false, int MODE = MODE_TOPK>
cudaError_t launch_variant(const TcMaps &maps, const TensorArgs &a, int32_t n_groups, cudaStream_t s) {
    const size_t smem = tensor_smem<BN, PK, CG2, MODE>(F4);
    cudaError_t e = cudaFuncSetAttribute(tensor_kernel<BN, PAIR, KM, PK, F4, CG2, MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3((PAIR ? 2 : 1) * n_groups);
    cfg.blockDim = dim3(tc_threads(KM, PK, TcShape<BN, PK, CG2, MODE>::ES));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // after the query preparation (see launch_dependent)
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = PAIR ? 2 : 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = PAIR ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, tensor_kernel<BN, PAIR, KM, PK, F4, CG2, MODE>, maps, a);
}

// Full-matrix and hit launches: the shapes of single calls.
template <int MODE>
cudaError_t launch_single(const TcMaps &maps, const TensorArgs &a, const TcLaunch &L, cudaStream_t s) {
    if (L.f4)
        return L.pk     ? launch_variant<TC_BN4, false, 16, true, true, false, MODE>(maps, a, L.n_groups, s)
               : L.pair ? launch_variant<TC_BN4, true, 16, false, true, false, MODE>(maps, a, L.n_groups, s)
                        : launch_variant<TC_BN4, false, 16, false, true, false, MODE>(maps, a, L.n_groups, s);
    return L.pk     ? launch_variant<256, false, 16, true, false, false, MODE>(maps, a, L.n_groups, s)
           : L.pair ? launch_variant<256, true, 16, false, false, false, MODE>(maps, a, L.n_groups, s)
                    : launch_variant<256, false, 16, false, false, false, MODE>(maps, a, L.n_groups, s);
}

}  // namespace

cudaError_t launch_tensor_multi(int bn, const TcLaunch &L, cudaStream_t s) {
    TcMaps maps;
    TensorArgs a;
    memset(&maps, 0, sizeof maps);
    memset(&a, 0, sizeof a);
    if (L.n_panels < 1 || L.n_panels > TC_MAXP) return cudaErrorInvalidValue;
    if (L.n_groups < 1) return cudaSuccess;
    a.n_panels = L.n_panels;
    for (int p = 0; p < L.n_panels; ++p) {
        maps.a[p] = L.map_a[p];
        maps.b[p] = L.map_b[p];
        a.panel[p].n_refs = L.n_refs[p];
        a.panel[p].n_q = L.n_q[p];
        a.panel[p].n_rt = L.n_rt[p];
        a.panel[p].n_kb = L.kpad[p] / TC_BK;
        a.panel[p].sc = L.sched[p];
        a.panel[p].qconst = L.qconst[p];
        a.panel[p].gcut = L.gcut[p];
        a.panel[p].gcut_ld = L.gcut_ld[p];
        a.panel[p].n_pub = L.n_pub[p];
        a.panel[p].pub_rank = L.pub_rank[p];
        a.panel[p].pub_need = L.pub_need[p];
        a.panel[p].qspread = L.qspread[p];
        a.order[p] = L.order[p];
    }
    a.threshold = L.threshold;
    a.k = L.k;
    a.epi = L.epi;
    a.out = L.out;
    a.ld_out = L.ld_out;
    a.capacity = L.capacity;
    a.hit_q = L.hit_q;
    a.hit_r = L.hit_r;
    a.hit_score = L.hit_score;
    a.hit_count = L.hit_count;
    a.partial = L.partial;
    a.status = L.status;
    a.arrive = L.arrive;
    if (L.epi != EPI_TOPK) {
        if (L.cg2 || (L.pk && L.pair) || (!L.f4 && bn != 256)) return cudaErrorInvalidValue;
        return L.epi == EPI_HITS ? launch_single<MODE_HITS>(maps, a, L, s) : launch_single<MODE_SCORES>(maps, a, L, s);
    }
    // 16-slot lists when k allows (half the insert network, 32 fewer registers)
    const bool k16 = L.k <= 16;
    if (L.f4) {  // 224-reference tiles whatever bn says
        if (L.pk) {
            if (L.pair) return cudaErrorInvalidValue;
            return k16 ? launch_variant<TC_BN4, false, 16, true, true>(maps, a, L.n_groups, s)
                       : launch_variant<TC_BN4, false, 32, true, true>(maps, a, L.n_groups, s);
        }
        if (L.pair && L.cg2)
            return k16 ? launch_variant<TC_BN4, true, 16, false, true, true>(maps, a, L.n_groups, s)
                       : launch_variant<TC_BN4, true, 32, false, true, true>(maps, a, L.n_groups, s);
        if (L.pair) return k16 ? launch_variant<TC_BN4, true, 16, false, true>(maps, a, L.n_groups, s)
                               : launch_variant<TC_BN4, true, 32, false, true>(maps, a, L.n_groups, s);
        return k16 ? launch_variant<TC_BN4, false, 16, false, true>(maps, a, L.n_groups, s)
                   : launch_variant<TC_BN4, false, 32, false, true>(maps, a, L.n_groups, s);
    }
    if (L.pair && bn != 256) return cudaErrorInvalidValue;
    if (L.pk) {
        if (L.pair || bn != 256) return cudaErrorInvalidValue;
        return k16 ? launch_variant<256, false, 16, true>(maps, a, L.n_groups, s)
                   : launch_variant<256, false, 32, true>(maps, a, L.n_groups, s);
    }
    if (L.pair && L.cg2)
        return k16 ? launch_variant<256, true, 16, false, false, true>(maps, a, L.n_groups, s)
                   : launch_variant<256, true, 32, false, false, true>(maps, a, L.n_groups, s);
    if (L.pair) return k16 ? launch_variant<256, true, 16>(maps, a, L.n_groups, s)
                           : launch_variant<256, true, 32>(maps, a, L.n_groups, s);
    if (bn == 128) return k16 ? launch_variant<128, false, 16>(maps, a, L.n_groups, s)
                              : launch_variant<128, false, 32>(maps, a, L.n_groups, s);
    return k16 ? launch_variant<256, false, 16>(maps, a, L.n_groups, s)
               : launch_variant<256, false, 32>(maps, a, L.n_groups, s);
}

}  // namespace fastid
