// Few-query form of the FP4 comparison over packed rows: the per-query top-k
// of up to 64 queries, with the references streamed once.
//
// The tensor kernel (tensor.cu) keeps 128 queries as the MMA's M operand and
// expands each packed reference stage into shared memory; for one query tile
// the shared memory -- TMA writes, expansion reads and writes, and the tensor
// core reading queries and references back -- set its pace (48 queries x 20M
// references at N = 2048: 1.88 ms against 0.75 ms of HBM).  Here the roles
// are swapped:
//   M = 128 references, expanded from their packed rows in registers straight
//       into TMEM, where the MMA reads its A operand (tcgen05.mma kind::mxf4
//       with A in TMEM: eight e2m1 nibbles a 32-bit column, lane = row)
//   N = the queries (16 .. 64), encoded once and resident in shared memory
//       for the whole launch
//   D = 128 references x N queries in TMEM
// so the shared memory carries the packed bits once each way and the queries,
// and a 128-reference tile of 2048 loci costs 32 MMAs of 36 cycles (46 beside
// the expansion's TMEM stores; probe).  Above 64 queries an MMA takes longer
// and the accumulators crowd the operand stages out of TMEM: measured, the
// tensor kernel is then as fast or faster.
// Expansion is four logic operations for 32 loci: nibble position j of a
// packed word becomes e2m1 0.5, 1 or 2 by a mask alone for j = 0, 1, 2, and
// for j = 3 the bit is the sign of a 1 put beside it, so the element is
// 1 - 2 R.  The query operand holds the inverses -- a / 0.5, a, a / 2 and
// -a / 2 for the a of tensor.cu -- and the sum of a / 2 over the j = 3 loci
// goes into the query's constant, so every product is 0, +-0.5 or +-1 and
// D + constant is exact as there.
//
// Warps of a 672-thread CTA, one CTA an SM (persistent over a slice of
// reference tiles).  Every role waits far longer than it works, so each is
// doubled: even and odd tiles have their own epilogue warps, their own MMA
// issuer (an issuer spends ~250 cycles between a stage's MMAs and the next's,
// the MMAs themselves 370) and their own expanding warps, and the stages of
// an even and an odd tile alternate.  Each side has its own half of every
// ring, all of even length: a barrier's parity tells only the last two phases
// apart, so its phases have to follow one another for whoever waits.
//   0 .. 7    epilogue: a reference a thread, a query a column (two sets of
//             four, one warp a TMEM lane quadrant)
//   8 .. 15   expansion: two sets of four warps
//   16        TMA producer of packed stages (128 rows x 64 bytes)
//   17, 18    MMA issue (converged, see tc_ptx.cuh); 17 holds the TMEM
//   19, 20    merging: every other query each
//
// Top-k.  A score that beats its query's cut goes to the query's ring of
// FQ_QUEUE entries in shared memory; the merging warps take the entries out,
// sort them and merge them into the query's sorted list by warp shuffles, and
// lower the cut.  Nothing meets at a barrier: an epilogue warp waits only for
// room in a full ring.  (With queues merged by the epilogue warps between
// tiles, every tile's barrier cost as much as its filter.)  Cuts start at the
// k-th best of a sample of the references (seed kernel), and the slices publish
// their best scores, which bound the k-th of all of them together (see the
// merging warps), so that few candidates ever arrive.
//
// Measured (fastid_topk, 20M references, N = 2048, us; the tensor kernel over
// packed rows before -> this form): 1 query 1930 -> 1043, 48 mixtures 1990 ->
// 1157, 64 at k = 32 2400 -> 1404.  HBM is the floor at 754; the SM's issue
// slots set the pace (expansion ~2000 of ~3900 warp instructions a tile).
#include <algorithm>
#include <cstring>

#include "few.h"
#include "keys.cuh"
#include "tc_ptx.cuh"

namespace fastid {

namespace {

constexpr int FQ_M = 128;            // references a tile
constexpr int FQ_THREADS = 672;
constexpr int FQ_STAGE = FQ_M * 64;  // packed stage: 512 loci of 128 references
constexpr int FQ_MAX_STAGES = 16;
constexpr int FQ_MIN_STAGES = 4;
constexpr int FQ_A_STAGES = 4;       // TMEM operand stages of 64 columns, two a side
constexpr int FQ_ACC = 4;            // accumulators of up to 48 queries; 2 of 64
constexpr uint32_t FQ_A_COL = 192;   // operand columns, after 192 of accumulators
constexpr int FQ_N = 64;             // queries at most
constexpr uint32_t FQ_SF_COL = 448;  // unit scale factors, 64 columns
constexpr int FQ_QUEUE = 32;         // ring entries a query: one a lane when merged
constexpr int FQ_MERGE_MIN = 8;      // rings of this many entries are merged before shorter ones
constexpr int FQ_SLICES_MAX = 256;   // slices whose published scores a warp looks through
constexpr int FQ_SEED_WARPS = 32;    // seed kernel: one encodes, the others score FQ_SEED_ROWS references each
constexpr int FQ_SEED_ROWS = 8;
constexpr int FQ_SAMPLE_ROUND = (FQ_SEED_WARPS - 1) * FQ_SEED_ROWS;
constexpr int FQ_SAMPLE_MAX = 4 * FQ_SAMPLE_ROUND;

struct FewArgs {
    int64_t n_refs;
    int64_t n_rt;        // reference tiles
    int32_t n_q;         // queries
    int32_t slices;      // CTAs
    int32_t ncols;       // N of the MMA: queries rounded up to 16
    int32_t n_kb;        // 256-locus chunks
    int32_t stages;      // packed stages
    int32_t k;
    uint32_t threshold;  // clamped to <= N
    const float *qconst;
    int32_t *gcut;
    int32_t *pub;        // [query][slices]: each slice's pub_rank-th best score so far
    int32_t pub_rank, pub_need;  // the pub_need-th smallest of those bounds the k-th of all
    uint64_t *partial;   // [slot = CTA][k][128]
    uint32_t *status;
};

struct FewSmem {
    uint64_t full[FQ_MAX_STAGES];
    uint64_t empty[FQ_MAX_STAGES];
    uint64_t afull[FQ_A_STAGES];
    uint64_t aempty[FQ_A_STAGES];
    uint64_t tfull[FQ_ACC];
    uint64_t tempty[FQ_ACC];
    uint64_t bfull;
    uint64_t done;
    uint32_t tmem_base;
    int abort_flag;
    int finished;     // epilogue warps that are through
    int64_t tile[8];  // the tile each epilogue warp is at
};

// Shared memory after the 1024-byte aligned base: queries, packed stages,
// lists, rings, per-query cuts, constants and ring ends, control block.
__host__ __device__ inline uint32_t few_smem_bytes(int ncols, int n_kb, int stages, int k) {
    return 1024u + (uint32_t)ncols * 128u * n_kb + (uint32_t)stages * FQ_STAGE + (uint32_t)ncols * k * 8u +
           (uint32_t)ncols * FQ_QUEUE * 8u + 4u * FQ_N * 4u + 512u;
}
static_assert(sizeof(FewSmem) <= 512, "control block");

// A stage's MMAs -- eight, or four where FULL is false -- and the commit that
// frees its TMEM columns, in one block with one election: A at TMEM columns a,
// a + 8, ..., the queries' descriptors from b and b2 (the two 256-locus
// chunks) advancing 32 bytes of K each.  An MMA of 16 .. 64 queries takes ~40
// cycles and the pipe holds one or two, so what the issuing warp does between
// stages must not wait: the next stage's barrier and the next accumulator's
// are tested first in the block and the answers (ready, room) read last, when
// they have long arrived.  The answers are each lane's own: the warp votes on
// them before it branches, as it does on everything that other warps or CTAs
// change, because the two sides of such a branch meet at whole-warp
// instructions (elect.sync, votes, reductions).
template <bool FULL>
__device__ __forceinline__ void mma_few(uint32_t d, uint32_t a, uint64_t b, uint64_t b2, uint32_t idesc, uint32_t sfa,
                                        uint32_t sfb, uint32_t acc, uint32_t commit, uint32_t next, uint32_t next_par,
                                        uint32_t room_bar, uint32_t room_par, uint32_t &ready, uint32_t &room) {
#define FASTID_MMA_TS "@e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%2], "
#define FASTID_MMA_ARGS ", %11, [%12], [%13], "
#define FASTID_FEW_HEAD                                                                           \
    "{\n\t.reg .pred p, q, e, r, s;\n\t"                                                          \
    "mbarrier.test_wait.parity.shared::cta.b64 r, [%16], %17;\n\t"                                \
    "mbarrier.test_wait.parity.shared::cta.b64 s, [%18], %19;\n\t" FASTID_ELECT                   \
    "setp.ne.b32 p, %14, 0;\n\tsetp.ne.b32 q, %14, 0xFFFFFFFF;\n\t" FASTID_MMA_TS               \
    "[%3], %7" FASTID_MMA_ARGS "p;\n\t" FASTID_MMA_TS "[%4], %8" FASTID_MMA_ARGS "q;\n\t" FASTID_MMA_TS \
    "[%5], %9" FASTID_MMA_ARGS "q;\n\t" FASTID_MMA_TS "[%6], %10" FASTID_MMA_ARGS "q;\n\t"
#define FASTID_FEW_TAIL                                                                                        \
    "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%15];\n\t"                     \
    "selp.u32 %0, 1, 0, r;\n\tselp.u32 %1, 1, 0, s;\n\t}"
#define FASTID_FEW_IN                                                                                           \
    "r"(d), "r"(a), "r"(a + 8), "r"(a + 16), "r"(a + 24), "l"(b), "l"(b + 2u), "l"(b + 4u), "l"(b + 6u), "r"(idesc), \
        "r"(sfa), "r"(sfb), "r"(acc), "r"(commit), "r"(next), "r"(next_par), "r"(room_bar), "r"(room_par)
    if constexpr (FULL)
        asm volatile(FASTID_FEW_HEAD FASTID_MMA_TS "[%20], %24" FASTID_MMA_ARGS "q;\n\t" FASTID_MMA_TS
                     "[%21], %25" FASTID_MMA_ARGS "q;\n\t" FASTID_MMA_TS "[%22], %26" FASTID_MMA_ARGS
                     "q;\n\t" FASTID_MMA_TS "[%23], %27" FASTID_MMA_ARGS "q;\n\t" FASTID_FEW_TAIL
                     : "=&r"(ready), "=&r"(room)
                     : FASTID_FEW_IN, "r"(a + 32), "r"(a + 40), "r"(a + 48), "r"(a + 56), "l"(b2), "l"(b2 + 2u),
                       "l"(b2 + 4u), "l"(b2 + 6u)
                     : "memory");
    else
        asm volatile(FASTID_FEW_HEAD FASTID_FEW_TAIL
                     : "=&r"(ready), "=&r"(room)
                     : FASTID_FEW_IN
                     : "memory");
#undef FASTID_MMA_TS
#undef FASTID_MMA_ARGS
#undef FASTID_FEW_HEAD
#undef FASTID_FEW_TAIL
#undef FASTID_FEW_IN
}

// 32 lanes x 32 consecutive columns.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

// Puts a key at place `at` of a ring, once there is room for it (bounded: the
// merging warps empty full rings).
__device__ __noinline__ void ring_put(uint64_t *ring, uint32_t *tail, uint32_t at, uint64_t key,
                                      volatile int *abort_flag, uint32_t *status) {
    volatile uint32_t *vt = tail;
    if (at - *vt >= (uint32_t)FQ_QUEUE) {
        const uint64_t t0 = globaltimer();
        while (at - *vt >= (uint32_t)FQ_QUEUE) {
            if (*abort_flag) return;
            if (globaltimer() - t0 > WAIT_NS) {
                *abort_flag = 1;
                atomicOr(status, ST_TIMEOUT);
                atomicExch(status + 1, 30u);
                return;
            }
        }
    }
    *reinterpret_cast<volatile uint64_t *>(ring + (at & (FQ_QUEUE - 1))) = key;
}

__global__ void __launch_bounds__(FQ_THREADS, 1)
    few_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_r, const FewArgs A) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t *base = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
    const int ncols = A.ncols, n_kb = A.n_kb, k = A.k;
    const uint32_t n_st = (uint32_t)(A.n_kb + 1) >> 1;
    uint8_t *sB = base;
    uint8_t *sP = sB + ncols * 128 * n_kb;
    uint64_t *list = reinterpret_cast<uint64_t *>(sP + A.stages * FQ_STAGE);  // [query][k], ascending
    uint64_t *ring = list + ncols * k;                                // [query][FQ_QUEUE] keys, KEY_EMPTY: free
    float *cut = reinterpret_cast<float *>(ring + ncols * FQ_QUEUE);  // candidate: d < cut
    float *qc = cut + FQ_N;
    uint32_t *head = reinterpret_cast<uint32_t *>(qc + FQ_N);  // entries ever put in
    uint32_t *tail = head + FQ_N;                              // and taken out
    FewSmem *ctl = reinterpret_cast<FewSmem *>(tail + FQ_N);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *abort_flag = &ctl->abort_flag;
    const int64_t y = blockIdx.x;  // slice
    const int64_t t_lo = y * A.n_rt / A.slices, t_hi = (y + 1) * A.n_rt / A.slices;
    // Stages come in this order: those of a pair of tiles in turn (an odd last
    // tile's partner's places stay empty).
    const uint32_t n_acc = ncols <= 48 ? 4 : 2, d_col = ncols <= 48 ? 48 : 64;
    const uint32_t n_tiles = (uint32_t)(t_hi - t_lo);

    if (tid == 0) {
        for (int s = 0; s < A.stages; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);
            mbar_init(smem_u32(&ctl->empty[s]), 4);
        }
        for (int s = 0; s < FQ_A_STAGES; ++s) {
            mbar_init(smem_u32(&ctl->afull[s]), 4);
            mbar_init(smem_u32(&ctl->aempty[s]), 1);
        }
        for (int a = 0; a < FQ_ACC; ++a) {
            mbar_init(smem_u32(&ctl->tfull[a]), 1);
            mbar_init(smem_u32(&ctl->tempty[a]), 4);
        }
        mbar_init(smem_u32(&ctl->bfull), 1);
        mbar_init(smem_u32(&ctl->done), 2);
        ctl->abort_flag = 0;
        ctl->finished = 0;
        for (int w = 0; w < 8; ++w) ctl->tile[w] = t_lo;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 17) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&ctl->tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < ncols * (k + FQ_QUEUE); i += FQ_THREADS) list[i] = KEY_EMPTY;  // lists and rings
    if (tid < FQ_N) head[tid] = tail[tid] = 0u;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's TMEM lane quadrant
    if (warp < 4) {
#pragma unroll
        for (int c = 0; c < 64; c += 16) tmem_fill16(lanes + FQ_SF_COL + c, TC_SF_UNIT);
        // columns past ncols are read with the others and never written
        for (int c = 0; c < (int)FQ_A_COL; c += 16) tmem_fill16(lanes + c, 0u);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    pdl_wait();  // (everything up to here ran beside the seed kernel)
    const float INF = __int_as_float(0x7f800000);
    const float t1 = A.threshold == 0xFFFFFFFFu ? INF : (float)A.threshold + 1.0f;
    if (tid < FQ_N) {
        const bool valid = tid < A.n_q;
        const float cq = valid ? A.qconst[tid] : 0.f;
        const int32_t c = valid ? load_cut(A.gcut + tid) : NET_EMPTY;
        qc[tid] = cq;
        cut[tid] = !valid ? -INF : (c == NET_EMPTY ? t1 : fminf(t1, (float)(c + 1))) - cq;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp == 16) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            const uint32_t bf = smem_u32(&ctl->bfull);
            mbar_expect_tx(bf, (uint32_t)ncols * 128u * n_kb);
            for (int kb = 0; kb < n_kb; ++kb)
                tma_load_2d(smem_u32(sB) + kb * ncols * 128, &map_q, bf, kb * 128, 0);
            uint32_t stage = 0, phase = 0;
            uint32_t used = 0, filled = 0;  // stages filled, and the phase of each one's last fill
            bool ok = true;
            auto load = [&](uint32_t tt, uint32_t st) {
                ok = mbar_wait(smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag, A.status, 21);
                if (!ok) return;
                const uint32_t fb = smem_u32(&ctl->full[stage]);
                mbar_expect_tx(fb, FQ_STAGE);
                tma_load_2d(smem_u32(sP) + stage * FQ_STAGE, &map_r, fb, st * 8, (int32_t)((t_lo + tt) * FQ_M));
                used |= 1u << stage;
                filled = (filled & ~(1u << stage)) | (phase << stage);
            };
            auto next = [&]() {
                if (++stage == (uint32_t)A.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            };
            for (uint32_t tt = 0; tt < n_tiles && ok; tt += 2) {
                for (uint32_t st = 0; st < n_st && ok; ++st) {
                    load(tt, st);
                    next();
                    if (ok && tt + 1 < n_tiles) load(tt + 1, st);
                    next();
                }
            }
            // Drain: this CTA's copies have landed before it exits.
            mbar_drain(bf, 0, A.status, 22);
            for (int n = 0; n < A.stages; ++n)
                if ((used >> n) & 1u) mbar_drain(smem_u32(&ctl->full[n]), (filled >> n) & 1u, A.status, 22);
        }
    } else if (warp == 17 || warp == 18) {
        // ---------------- MMA issuers: even tiles, odd tiles ----------------
        const uint32_t first = (uint32_t)warp - 17u;
        const uint32_t idesc = idesc_mxf4(FQ_M, ncols);
        const uint64_t bd0 = sw128_desc(smem_u32(sB));
        const uint64_t b_step = (uint64_t)(ncols * 128) >> 4;
        const uint32_t sfa = tmem + FQ_SF_COL, sfb = sfa + 16;
        const uint32_t af0 = smem_u32(&ctl->afull[0]), ae0 = smem_u32(&ctl->aempty[0]);
        uint32_t acc = first, acc_phase = 0, as = first, aphase = 0;
        uint32_t ready = 0, room = 1;
        bool ok = warp_wait(smem_u32(&ctl->bfull), 0, abort_flag, A.status, 23);
        for (uint32_t tt = first; tt < n_tiles && ok; tt += 2) {
            if (!__all_sync(0xffffffffu, room)) {
                ok = warp_wait(smem_u32(&ctl->tempty[acc]), acc_phase ^ 1u, abort_flag, A.status, 24);
                if (!ok) break;
            }
            const uint32_t d = tmem + acc * d_col, tf = smem_u32(&ctl->tfull[acc]);
            if ((acc += 2) >= n_acc) {
                acc = first;
                acc_phase ^= 1u;
            }
            const uint32_t rb = smem_u32(&ctl->tempty[acc]);
            uint64_t b = bd0;
            for (uint32_t st = 0; st < n_st; ++st) {
                if (!__all_sync(0xffffffffu, ready)) {
                    ok = warp_wait(af0 + 8 * as, aphase, abort_flag, A.status, 25);
                    if (!ok) break;
                }
                tc_fence_after();  // the expanding warps' TMEM stores, and the epilogue's reads of the accumulator
                const uint32_t a = tmem + FQ_A_COL + as * 64, ab = ae0 + 8 * as;
                if ((as += 2) >= FQ_A_STAGES) {
                    as = first;
                    aphase ^= 1u;
                }
                if (2 * st + 1 < (uint32_t)n_kb)
                    mma_few<true>(d, a, b, b + b_step, idesc, sfa, sfb, st != 0, ab, af0 + 8 * as, aphase, rb,
                                  acc_phase ^ 1u, ready, room);
                else
                    mma_few<false>(d, a, b, b, idesc, sfa, sfb, st != 0, ab, af0 + 8 * as, aphase, rb,
                                   acc_phase ^ 1u, ready, room);
                b += 2 * b_step;
            }
            if (!ok) break;
            tc_commit(tf);
        }
        tc_commit(smem_u32(&ctl->done));
        mbar_drain(smem_u32(&ctl->done), 0, A.status, 26);
    } else if (warp >= 19) {
        // ---------------- merging: warp 19 even queries, warp 20 odd ones; lane l owns its l-th ----------------
        const int mine = 2 * lane + (warp == 19 ? 0 : 1), q0 = warp == 19 ? 0 : 1;
        const bool valid = mine < A.n_q;
        int32_t kth = NET_EMPTY;  // the list's k-th score
        uint32_t kth_r = 0u;      // and that entry's reference
        bool strict = true;       // the cut is below the k-th score, not at it
        int32_t shared = valid ? load_cut(A.gcut + mine) : NET_EMPTY;
        uint32_t least = FQ_MERGE_MIN;
        const int first_q = (int)y % A.n_q;
        int union_q = first_q;  // the query whose cut this slice bounds over all slices next
        for (bool last = false;;) {
            const bool ended = __all_sync(0xffffffffu, *reinterpret_cast<volatile int *>(&ctl->finished) == 8);
            __threadfence_block();  // entries put in before the warps were through are seen below
            int64_t at = t_hi;  // every reference below tile `at` has been filtered
            for (int w = 0; w < 8; ++w) at = min(at, *reinterpret_cast<volatile int64_t *>(&ctl->tile[w]));
            bool busy = false;
            const uint32_t waiting = valid ? *reinterpret_cast<volatile uint32_t *>(head + mine) -
                                                 *reinterpret_cast<volatile uint32_t *>(tail + mine)
                                           : 0u;
            uint32_t todo = __ballot_sync(0xffffffffu, waiting >= least);
            while (todo) {
                const int l = __ffs(todo) - 1, q = q0 + 2 * l;
                todo &= todo - 1u;
                // the entries written so far, in order of their places
                const uint32_t t0 = *reinterpret_cast<volatile uint32_t *>(tail + q);
                volatile uint64_t *slot = ring + q * FQ_QUEUE + ((t0 + lane) & (FQ_QUEUE - 1));
                uint64_t v = *slot;
                const uint32_t there = __ballot_sync(0xffffffffu, v != KEY_EMPTY);
                const int n = there == 0xffffffffu ? 32 : __ffs(~there) - 1;
                if (n == 0) continue;
                busy = true;
                if (lane < n)
                    *slot = KEY_EMPTY;
                else
                    v = KEY_EMPTY;
                __threadfence_block();
                __syncwarp();
                if (lane == 0) *reinterpret_cast<volatile uint32_t *>(tail + q) = t0 + n;
                v = warp_sort32(v, lane);
                v = warp_merge32(lane < k ? list[q * k + lane] : KEY_EMPTY, v, lane);
                if (lane < k) list[q * k + lane] = v;
                const uint64_t end = shfl64(v, k - 1), front = shfl64(v, A.pub_rank - 1);
                if (lane == l) {
                    if (front != KEY_EMPTY)
                        *reinterpret_cast<volatile int32_t *>(A.pub + (int64_t)q * A.slices + y) =
                            (int32_t)(front >> 32);
                    if (end != KEY_EMPTY) {
                        kth = (int32_t)(end >> 32);
                        kth_r = (uint32_t)end;
                        strict = false;
                        if (kth < shared) {
                            shared = kth;
                            atomicMin(A.gcut + q, kth);
                        }
                    }
                }
                __syncwarp();
            }
            // Cuts: at the shared one (ties kept), and at the k-th score --
            // below it once every reference up to the k-th entry's has been
            // filtered, when a tie can only come from a higher one.
            if (valid) {
                shared = min(shared, load_cut(A.gcut + mine));
                strict = strict || (int64_t)kth_r < at * FQ_M;
                float c = t1;
                if (shared != NET_EMPTY) c = fminf(c, (float)(shared + 1));
                if (kth != NET_EMPTY) c = fminf(c, (float)(strict ? kth : kth + 1));
                *reinterpret_cast<volatile float *>(cut + mine) = c - qc[mine];
            }
            if (__any_sync(0xffffffffu, last || *abort_flag != 0)) break;
            last = ended && !busy && least == 1u;  // one more look after the last entries
            least = busy && !ended ? FQ_MERGE_MIN : 1u;
            if (busy || ended) continue;
            // Idle: one query's cut over all slices.  pub_need slices have each
            // published a pub_rank-th best score, so the largest of the
            // pub_need smallest bounds the k-th best of their union -- which,
            // unlike any slice's own k-th, keeps up with all the references
            // compared so far on the whole GPU.  (48 queries x 20M: 1740 ->
            // 1500 us when this came in.)
            if (warp == 19 && A.slices <= FQ_SLICES_MAX) {
                int32_t v[FQ_SLICES_MAX / 32];
#pragma unroll
                for (int i = 0; i < FQ_SLICES_MAX / 32; ++i)
                    v[i] = 32 * i + lane < A.slices ? load_cut(A.pub + (int64_t)union_q * A.slices + 32 * i + lane)
                                                    : NET_EMPTY;
                const int32_t now = __shfl_sync(0xffffffffu, load_cut(A.gcut + union_q), 0);
                int32_t lo = 0, hi = now == NET_EMPTY ? FASTID_MAX_LOCI : now;
                auto at_most = [&](int32_t m) {
                    int n = 0;
#pragma unroll
                    for (int i = 0; i < FQ_SLICES_MAX / 32; ++i) n += v[i] <= m;
                    return (int)__reduce_add_sync(0xffffffffu, (uint32_t)n);
                };
                if (hi > 0 && at_most(hi - 1) >= A.pub_need) {
                    while (lo < hi) {  // the smallest score with pub_need slices at or below it
                        const int32_t mid = (lo + hi) >> 1;
                        if (at_most(mid) >= A.pub_need)
                            hi = mid;
                        else
                            lo = mid + 1;
                    }
                    if (lane == 0) atomicMin(A.gcut + union_q, lo);
                }
                union_q += A.slices;  // fewer slices than queries: several in turn
                if (union_q >= A.n_q) union_q = first_q;
            }
            __nanosleep(300);
        }
        __syncwarp();
        // The lists: slot = CTA, [k][128].
        for (int q = q0; q < A.n_q; q += 2)
            if (lane < k) A.partial[(y * k + lane) * TC_TILE_Q + q] = list[q * k + lane];
    } else if (warp >= 8) {
        // ---------------- expansion ----------------
        const uint32_t set = (uint32_t)(warp - 8) >> 2;   // the side: its tiles' stages are every other one
        const int row = (warp & 3) * 32 + lane;
        const uint32_t swz = (uint32_t)((row >> 1) & 3) << 4;  // TMA's 64-byte swizzle
        const uint32_t src = smem_u32(sP) + row * 64;
        uint32_t stage = set, as = set;
        uint32_t phase = 0, aphase = 0;
        uint32_t stored = 0u;  // afull barrier of the store in flight
        auto announce = [&]() {
            if (stored) {
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(stored);
                stored = 0u;
            }
        };
        const uint32_t mine = (n_tiles + 1 - set) / 2 * n_st;  // its tiles' stages
        uint32_t st = 0;
        for (uint32_t i = 0; i < mine; ++i) {
            const uint32_t fb = smem_u32(&ctl->full[stage]);
            if (!__all_sync(0xffffffffu, mbar_try_wait(fb, phase))) {
                announce();
                if (!warp_wait(fb, phase, abort_flag, A.status, 27)) break;
            }
            const uint32_t from = src + stage * FQ_STAGE;
            uint32_t w[16];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(w[4 * c]), "=r"(w[4 * c + 1]), "=r"(w[4 * c + 2]), "=r"(w[4 * c + 3])
                             : "r"(from + ((uint32_t)(c << 4) ^ swz))
                             : "memory");
            announce();
            if (!warp_wait(smem_u32(&ctl->aempty[as]), aphase ^ 1u, abort_flag, A.status, 28)) break;
            tc_fence_after();  // the MMAs that read this stage before
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t v[32];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t b = w[8 * half + j];
                    v[4 * j] = b & 0x11111111u;             // 0.5
                    v[4 * j + 1] = b & 0x22222222u;         // 1
                    v[4 * j + 2] = b & 0x44444444u;         // 2
                    v[4 * j + 3] = (b & 0x88888888u) | 0x22222222u;  // 1 - 2 R
                }
                if (half == 0 || 2 * st + 1 < (uint32_t)n_kb) tmem_st32(lanes + FQ_A_COL + as * 64 + half * 32, v);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->empty[stage]));
            stored = smem_u32(&ctl->afull[as]);
            if (++st == n_st) st = 0;
            if ((stage += 2) >= (uint32_t)A.stages) {
                stage -= A.stages;
                phase ^= 1u;
            }
            if ((as += 2) >= FQ_A_STAGES) {
                as -= FQ_A_STAGES;
                aphase ^= 1u;
            }
        }
        __syncwarp();
        announce();
    } else {
        // ---------------- epilogue ----------------
        const int row = (warp & 3) * 32 + lane;
        const uint32_t odd = (uint32_t)warp >> 2;
        uint32_t acc = odd, acc_phase = 0;
        for (int64_t t = t_lo + odd; t < t_hi; t += 2) {
            if (lane == 0) *reinterpret_cast<volatile int64_t *>(&ctl->tile[warp]) = t;
            if (!warp_wait(smem_u32(&ctl->tfull[acc]), acc_phase, abort_flag, A.status, 29)) break;
            tc_fence_after();
            const uint32_t taddr = lanes + acc * d_col;
            const int64_t r = t * FQ_M + row;
            const bool live = r < A.n_refs;
            for (int cb = 0; cb < ncols; cb += 32) {
                uint32_t v[32];
                tmem_ld32(taddr + cb, v);
                // any d < cut: the sign of d - cut (an infinite cut keeps its
                // sign, and D holds no NaN), ORed
                const float4 *c4 = reinterpret_cast<const float4 *>(cut + cb);
                uint32_t d[32], any = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 c = c4[j];
                    d[4 * j] = __float_as_uint(__uint_as_float(v[4 * j]) - c.x);
                    d[4 * j + 1] = __float_as_uint(__uint_as_float(v[4 * j + 1]) - c.y);
                    d[4 * j + 2] = __float_as_uint(__uint_as_float(v[4 * j + 2]) - c.z);
                    d[4 * j + 3] = __float_as_uint(__uint_as_float(v[4 * j + 3]) - c.w);
                    any |= d[4 * j] | d[4 * j + 1];
                    any |= d[4 * j + 2] | d[4 * j + 3];
                }
                if (!__any_sync(0xffffffffu, live && (int32_t)any < 0)) continue;
                // A short loop over the groups of four columns that some lane
                // needs, re-read from TMEM: unrolled over the 32 columns, the code was
                // fetched anew each time (2048 loci, 48 queries, k = 32: 3M
                // references 353 -> 301 us, 20M 1273 -> 1206).
                uint32_t m = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    m |= ((d[4 * j] | d[4 * j + 1] | d[4 * j + 2] | d[4 * j + 3]) >> 31) << j;
                m = __reduce_or_sync(0xffffffffu, live ? m : 0u);
#pragma unroll 1
                while (m != 0u) {
                    const int q0 = cb + 4 * (__ffs(m) - 1);
                    m &= m - 1u;
                    uint32_t w[4];
                    tmem_ld_group(taddr + q0, w);
                    const float4 c = *reinterpret_cast<const float4 *>(cut + q0);
                    const float cq[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float x = __uint_as_float(w[j]);
                        if (live && x < cq[j]) {
                            const int q = q0 + j;
                            const uint64_t key = make_key((uint32_t)(int32_t)(x + qc[q]), (uint32_t)r);
                            const uint32_t at = atomicAdd(&head[q], 1u);
                            ring_put(ring + q * FQ_QUEUE, tail + q, at, key, abort_flag, A.status);
                        }
                    }
                    __syncwarp();
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->tempty[acc]));
            if ((acc += 2) >= n_acc) {
                acc = odd;
                acc_phase ^= 1u;
            }
        }
        __threadfence_block();
        __syncwarp();
        if (lane == 0) {
            *reinterpret_cast<volatile int64_t *>(&ctl->tile[warp]) = t_hi;
            atomicAdd(&ctl->finished, 1);
        }
    }

    pdl_trigger();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 17)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// Query operand and starting cut, a block a row: warp 0 encodes the row (the
// inverses of the expansion, see the top) and its constant; the others score
// a strided sample of the references against the query, and the k-th smallest
// of those bounds every result entry of the query (there are k references no
// worse).  The kernel is a chain of latencies (1024 samples for every call
// and a block barrier in each bisection step: 16 us of a 38 us call), so a
// warp loads 8 references at once, few calls take a second round, one warp
// selects alone, and the compare kernel sets itself up meanwhile.
__global__ void __launch_bounds__(FQ_SEED_WARPS * 32)
    few_seed_kernel(const uint64_t *__restrict__ q, int64_t ld_q, int64_t n_q, int32_t n_words, int32_t n_loci,
                    const uint8_t *__restrict__ modes, int32_t kbytes, uint8_t *__restrict__ out,
                    float *__restrict__ qconst, const SharedCut cut, const uint64_t *__restrict__ refs, int64_t stride,
                    int sample, int k, int32_t *__restrict__ pub, int32_t slices) {
    pdl_trigger();
    __shared__ uint32_t sc[FQ_SAMPLE_MAX];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r = blockIdx.x;
    const bool valid = r < n_q;
    const uint64_t *qr = q + r * ld_q;
    const bool mis = valid && modes[r] == FASTID_MODE_MISMATCH;
    int32_t best = NET_EMPTY;
    if (warp == 0) {
        if (valid && cut.run_s) {
            const int64_t last = r * cut.k + cut.k - 1;
            if (cut.run_i[last] >= 0 && cut.run_s[last] <= (uint32_t)FASTID_MAX_LOCI) best = (int32_t)cut.run_s[last];
        }
        uint32_t pc = 0;
        int32_t a3 = 0;  // sum of a over the j = 3 loci
        for (int32_t c = lane; c < kbytes / 16; c += 32) {
            const int32_t l0 = c * 32;
            uint32_t bits = 0;
            if (valid && (l0 >> 6) < n_words) bits = (uint32_t)(qr[l0 >> 6] >> (l0 & 63));
            const int32_t live = n_loci - l0;
            const uint32_t in_n = !valid ? 0u : live >= 32 ? 0xFFFFFFFFu : live <= 0 ? 0u : ((1u << live) - 1u);
            bits &= in_n;
            pc += __popc(bits);
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t qb = (bits >> j) & 0x11111111u;  // Q at nibble n = locus 4n + j
                const uint32_t nb = (in_n >> j) & 0x11111111u;  // l < N
                // e2m1 of a = +1 and of a = -1: 2, 1, 0.5 times a, and -0.5 times
                const uint32_t plus = j == 0 ? 4u : j == 1 ? 2u : j == 2 ? 1u : 9u;
                w[j] = (nb & ~qb) * plus | (mis ? qb * (plus ^ 8u) : 0u);
                if (j == 3) a3 += __popc(nb & ~qb) - (mis ? __popc(qb) : 0);
            }
            reinterpret_cast<uint4 *>(out + r * (int64_t)kbytes)[c] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        pc = __reduce_add_sync(0xffffffffu, pc);
        a3 = __reduce_add_sync(0xffffffffu, a3);
        if (lane == 0) qconst[r] = (mis ? (float)pc : 0.f) + 0.5f * (float)a3;
        for (int i = lane; i < slices; i += 32) pub[r * slices + i] = NET_EMPTY;
    } else if (valid) {
        for (int i0 = (warp - 1) * FQ_SEED_ROWS; i0 < sample; i0 += FQ_SAMPLE_ROUND) {
            uint32_t pc[FQ_SEED_ROWS] = {};
            for (int32_t w = lane; w < n_words; w += 32) {
                uint64_t rw[FQ_SEED_ROWS];
                const uint64_t qw = qr[w];
#pragma unroll
                for (int u = 0; u < FQ_SEED_ROWS; ++u) rw[u] = i0 + u < sample ? refs[(i0 + u) * stride + w] : 0ull;
#pragma unroll
                for (int u = 0; u < FQ_SEED_ROWS; ++u) pc[u] += __popcll(mis ? rw[u] ^ qw : rw[u] & ~qw);
            }
#pragma unroll
            for (int u = 0; u < FQ_SEED_ROWS; ++u) {
                const uint32_t s = __reduce_add_sync(0xffffffffu, pc[u]);
                if (lane == 0 && i0 + u < sample) sc[i0 + u] = s;
            }
        }
    }
    __syncthreads();
    if (warp != 0) return;
    if (valid && sample >= k) {
        constexpr int V = FQ_SAMPLE_MAX / 32;
        uint32_t v[V];
#pragma unroll
        for (int u = 0; u < V; ++u) v[u] = u * 32 + lane < sample ? sc[u * 32 + lane] : 0xFFFFFFFFu;
        uint32_t lo = 0, hi = (uint32_t)n_loci;
        while (lo < hi) {  // the smallest value with k samples at or below it
            const uint32_t mid = (lo + hi) >> 1;
            uint32_t n = 0;
#pragma unroll
            for (int u = 0; u < V; ++u) n += v[u] <= mid;
            if (__reduce_add_sync(0xffffffffu, n) >= (uint32_t)k)
                hi = mid;
            else
                lo = mid + 1;
        }
        best = min(best, (int32_t)lo);
    }
    if (lane == 0) cut.out[r] = best;
}

constexpr uint32_t FQ_SMEM_MAX = 227u * 1024u;

}  // namespace

bool few_shape(int64_t n_q, int32_t n_loci, int32_t k, FewShape *S) {
    if (n_q < 1 || n_q > FQ_N) return false;
    S->ncols = (int32_t)((n_q + 15) / 16 * 16);
    S->n_kb = tensor_kbytes4(n_loci) / 128;
    const int64_t least = (int64_t)few_smem_bytes(S->ncols, S->n_kb, FQ_MIN_STAGES, k);
    if (least > FQ_SMEM_MAX) return false;
    S->stages = (int32_t)std::min<int64_t>(FQ_MAX_STAGES,
                                           FQ_MIN_STAGES + 2 * ((FQ_SMEM_MAX - least) / (2 * FQ_STAGE)));
    return true;
}

// The tensor kernel takes one query as it takes 128, and its lists fill faster;
// this form streams the rows faster, starts its cuts from a sample, and takes
// longer with every query and with k.  So up to 8 queries it is never the slower
// by more than 3 us, and with more it needs a database long enough to repay its
// lists, and rows wider than 256 bytes (N = 2048) one long enough to repay four
// rounds of samples (seed kernel).  Above k = 16 the tensor kernel's lists are
// the slower 32-slot ones.  Measured (fastid_topk, us, this form / the tensor
// kernel over packed rows; MiB of packed rows, N = 2048 unless named):
//   queries, k      0.5     24        61         122        244        366        659
//    8, 10        24/31    35/46    44/62      56/90      81/132     106/178    169/277
//   16, 1         26/22    37/33    43/50      56/78      82/122     109/166    171/266
//   16, 10        29/32    43/48    51/62      65/90      87/134     114/179    175/279
//   32, 1         32/23    45/33    52/52      63/80      84/123     111/168    173/268
//   32, 10        37/33    53/48    67/66      83/92      101/136    126/182    187/281
//   32, 32        51/54    62/77    91/98      117/128    150/172    166/223    225/329
//   48, 1         40/23    53/35    58/52      73/81      87/124     117/168    181/268
//   48, 10        45/33    64/48    83/65      101/93     123/137    144/182    207/281
//   48, 32        64/54    82/77    124/97     159/128    204/173    228/223    282/328
//   64, 1         46/24    60/35    65/54      76/80      101/124    137/168    212/269
//   64, 10        53/33    84/48    102/66     127/95     148/137    178/183    251/282
//   64, 32        78/54    107/77   159/98     205/128    246/175    270/224    334/329
//   16, 10, N = 8192       57/45               90/84                 (488: 165/212)
//   32, 32, N = 8192       68/68               115/109               (488: 187/242)
// and N = 200 and 512 as N = 2048 for as many bytes.  (With one line for every k,
// and none up to 32 queries, 32 queries of k = 1 took 36 us over 1000 references
// where the tensor kernel takes 23 and took 29 before its queues.)
bool few_pays(int64_t n_q, int32_t k, int64_t n_refs, int64_t row_bytes) {
    if (n_q <= 8) return true;
    // the shortest database, KiB of packed rows: up to 16, 32, 48, 64 queries; k up to 4, up to 16, above
    constexpr int64_t least[4][3] = {
        {32 << 10, 256, 0}, {48 << 10, 48 << 10, 256}, {112 << 10, 224 << 10, 384 << 10}, {224 << 10, 448 << 10, 640 << 10}};
    const int64_t wide = k <= 16 && row_bytes > 256 ? (row_bytes - 256) * 200 : 0;
    return n_refs * row_bytes >= (least[std::min<int64_t>((n_q - 1) / 16, 3)][k <= 4 ? 0 : k <= 16 ? 1 : 2] + wide) << 10;
}

cudaError_t launch_few_seed(const FewLaunch &L, const FewShape &S, cudaStream_t s) {
    // At most a sixteenth of the references.  With up to 8 queries the seeds
    // are on the call's critical path and one round is enough (one query over
    // 2M x 2048: 132.7 us with one round, 141.9 with four; over 200000 x 1024
    // the same); with more the first tiles' candidates cost more than the
    // rounds (48 queries, top 32 of 200000 x 1024: 151 us with one, 115 with
    // four, 97 with eight, but 16 queries over 50000 40.7, 41.5 and 45.8).
    const int rounds = L.n_q <= 8 ? 1 : FQ_SAMPLE_MAX / FQ_SAMPLE_ROUND;
    const int sample = (int)std::min<int64_t>(rounds * FQ_SAMPLE_ROUND, L.n_refs / 16);
    const int64_t stride = sample > 0 ? L.n_refs / sample * L.ld64 : 0;
    few_seed_kernel<<<(unsigned)S.ncols, FQ_SEED_WARPS * 32, 0, s>>>(
        L.q, L.ld_q, L.n_q, L.n_words, L.n_loci, L.modes, S.n_kb * 128, L.operand, L.qconst, L.cut, L.packed, stride,
        sample, L.k, L.pub, L.slices);
    return cudaGetLastError();
}

cudaError_t launch_few(const FewLaunch &L, const FewShape &S, cudaStream_t s) {
    CUtensorMap map_q, map_r;
    cudaError_t e = make_operand_map(&map_q, L.operand, S.ncols, S.n_kb * 128, S.ncols);
    if (e == cudaSuccess) e = make_packed_map(&map_r, L.packed, L.n_pad, L.ld64, 8, FQ_M, true);
    if (e != cudaSuccess) return e;
    FewArgs a;
    memset(&a, 0, sizeof a);
    a.n_refs = L.n_refs;
    a.n_rt = (L.n_refs + FQ_M - 1) / FQ_M;
    a.n_q = (int32_t)L.n_q;
    a.slices = L.slices;
    a.ncols = S.ncols;
    a.n_kb = S.n_kb;
    a.stages = S.stages;
    a.k = L.k;
    a.threshold = L.threshold;
    a.qconst = L.qconst;
    a.gcut = L.cut.out;
    a.pub = L.pub;
    a.pub_rank = (L.k + L.slices - 1) / L.slices;
    a.pub_need = (L.k + a.pub_rank - 1) / a.pub_rank;
    a.partial = L.partial;
    a.status = L.status;
    const uint32_t smem = few_smem_bytes(S.ncols, S.n_kb, S.stages, L.k);
    e = cudaFuncSetAttribute(few_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FQ_SMEM_MAX);
    if (e != cudaSuccess) return e;
    return launch_dependent(few_kernel, dim3((unsigned)L.slices), dim3(FQ_THREADS), smem, s, map_q, map_r, a);
}

}  // namespace fastid
