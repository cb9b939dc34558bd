// Reductions after a comparison launch: merge of per-segment top-k lists and
// the hit-list finish (count, overflow flag, sort by (q, r)).
#include <algorithm>

#include "common.cuh"
#include "keys.cuh"

namespace fastid {

namespace {

// Merge of one query's lists by W warps (a power of two, all in one block).
// A list is k ascending keys, one per lane; list i is load(i), KEY_EMPTY on
// lanes >= k.  Each warp folds every W-th list, MERGE_AHEAD of them loaded
// before the first is used -- a lone warp that loaded and folded one list
// after another was bound by that chain (0.73 us a list: 111 us for one
// query's 149 lists, 249 us for 304) -- and a list whose smallest key cannot
// enter is passed over.  The warps' results then meet in shared memory, in
// log2(W) rounds.  Warp 0 of the query returns the 32 smallest keys.
constexpr int MERGE_AHEAD = 8;
constexpr int MERGE_MAX_WARPS = 16;

template <class Load>
__device__ __forceinline__ uint64_t merge_lists(int n, int W, int k, int lane, uint64_t (*sm)[32], Load load) {
    const int warp = threadIdx.x >> 5, w = warp & (W - 1);
    uint64_t acc = KEY_EMPTY;
    for (int i = w; i < n; i += MERGE_AHEAD * W) {
        uint64_t v[MERGE_AHEAD];
#pragma unroll
        for (int u = 0; u < MERGE_AHEAD; ++u) v[u] = i + u * W < n ? load(i + u * W) : KEY_EMPTY;
#pragma unroll
        for (int u = 0; u < MERGE_AHEAD; ++u)
            if (shfl64(v[u], 0) < shfl64(acc, k - 1)) acc = warp_merge32(acc, v[u], lane);
    }
    // (a round writes rows [h, 2h) of the query's W and reads them back; the
    // next one writes lower rows, so one barrier a round is enough)
    for (int h = W >> 1; h > 0; h >>= 1) {
        if (w >= h && w < 2 * h) sm[warp][lane] = acc;
        __syncthreads();
        if (w < h) acc = warp_merge32(acc, sm[warp + h][lane], lane);
    }
    return acc;
}

// CTA whose unit range contains unit u.
__device__ int64_t cta_of(const Partition &P, int64_t u) {
    int64_t c = (u * P.grid) / P.n_units;
    while (c + 1 < P.grid && part_begin(P, c + 1) <= u) ++c;
    while (c > 0 && part_begin(P, c) > u) --c;
    return c;
}

// Plain launches, W warps per query: merge the sorted k-lists of every segment
// that covered the query's tile.  Segment lists are laid out [slot][tile_q][k]
// with slot = cta * max_seg + (segment index within the CTA).
__global__ void topk_merge_kernel(const uint64_t *__restrict__ partial, Partition P, int64_t n_q, int32_t k, int W,
                                  uint32_t *__restrict__ out_scores, int64_t *__restrict__ out_idx) {
    __shared__ uint64_t sm[MERGE_MAX_WARPS][32];
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int64_t q = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) / W;
    int64_t ql = 0, c_lo = 0, c_hi = -1, seg_lo = 0;
    if (q < n_q) {
        const int64_t qt = q / P.tile_q;
        ql = q - qt * P.tile_q;
        c_lo = cta_of(P, qt * P.n_rt);
        c_hi = cta_of(P, qt * P.n_rt + P.n_rt - 1);
        seg_lo = qt - part_begin(P, c_lo) / P.n_rt;
    }
    // (only the first CTA can have had an earlier tile: every other one starts inside this tile, segment 0)
    const uint64_t acc = merge_lists((int)(c_hi - c_lo + 1), W, k, lane, sm, [&](int i) {
        const int64_t slot = (c_lo + i) * P.max_seg + (i == 0 ? seg_lo : 0);
        return lane < k ? partial[(slot * P.tile_q + ql) * k + lane] : KEY_EMPTY;
    });
    if (q < n_q && (warp & (W - 1)) == 0 && lane < k) {
        out_scores[q * k + lane] = acc == KEY_EMPTY ? 0xFFFFFFFFu : (uint32_t)(acc >> 32);
        out_idx[q * k + lane] = acc == KEY_EMPTY ? -1ll : (int64_t)(uint32_t)acc;
    }
}

// Tensor launches: W warps per query; its tile's lists sit in one slot of
// every reference slice's group of its tile group (see TcSched).  Slot
// layout [slot][k][128].
struct MergeSched {
    int32_t n_panels;
    int32_t pair;
    int32_t k;
    TcSched sc[TC_MAXP];
    int64_t n_slots;   // slots in partial (checked by debug builds)
    uint32_t *status;  // the context's status word
    // accumulate: merge into the output lists instead of overwriting them,
    // this launch's reference indices taken + ref_offset
    int32_t accumulate;
    int64_t ref_offset;
    int64_t qspread;  // single-call jobs: output j is input query j (see spread_query_to_row)
};

// Debug builds (FASTID_DEBUG) check every slot a merge reads against the
// slot count; a slot out of range records ST_DEVICE with detail code 1 and is
// read as empty.  Release builds take the schedule's word for it.
__device__ __forceinline__ bool merge_slot_ok(const MergeSched &M, int64_t slot) {
#ifdef FASTID_DEBUG
    if (slot < 0 || slot >= M.n_slots) {
        if ((threadIdx.x & 31) == 0) {
            atomicOr(M.status, ST_DEVICE);
            atomicExch(M.status + 1, 1u);
        }
        return false;
    }
#else
    (void)M;
    (void)slot;
#endif
    return true;
}

__global__ void topk_merge_sched_kernel(const uint64_t *__restrict__ partial, const MergeSched M,
                                        const MergeJob *__restrict__ jobs, int64_t n_jobs, int W,
                                        uint32_t *__restrict__ out_s, int64_t *__restrict__ out_i) {
    __shared__ uint64_t sm[MERGE_MAX_WARPS][32];
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int64_t j = ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) / W;
    const int k = M.k;
    MergeJob jb;
    if (j >= n_jobs) {  // an idle warp of the last block: no lists, but the block's barriers
        jb.out_s = nullptr;
        jb.out_i = nullptr;
        jb.panel = 0;
        jb.q = 0;
    } else if (jobs) {
        jb = jobs[j];
    } else {
        jb.out_s = out_s + j * k;
        jb.out_i = out_i + j * k;
        jb.panel = 0;
        jb.q = (int32_t)spread_query_to_row(j, M.qspread);  // its operand row
    }
    const TcSched &sc = M.sc[jb.panel];
    const int64_t qt = jb.q / TC_TILE_Q, ql = jb.q - qt * TC_TILE_Q;
    const int64_t qq = M.pair ? qt >> 1 : qt;
    const int64_t rank = M.pair ? qt & 1 : 0;
    const int64_t x = qq / sc.tpx, li = qq - x * sc.tpx;
    const int64_t cpg = M.pair ? 2 : 1;
    // lists 0 .. b - 1: the slices' groups; list b: the tail group holding
    // this query tile, if there is a tail (see TcSched)
    const int n = j < n_jobs ? sc.b + (sc.t_groups > 0 ? 1 : 0) : 0;
    uint64_t acc = merge_lists(n, W, k, lane, sm, [&](int i) {
        int64_t slot;
        if (i < sc.b) {
            slot = (int64_t)sc.slot0 + ((x * sc.b + i) * cpg + rank) * sc.tpx + li;
        } else {
            const int64_t t = qq / sc.t_tpx, lt = qq - t * sc.t_tpx;
            slot = (int64_t)sc.slot0 + (int64_t)sc.a * sc.b * cpg * sc.tpx + (t * cpg + rank) * sc.t_tpx + lt;
        }
        return lane < k && merge_slot_ok(M, slot) ? partial[(slot * k + lane) * TC_TILE_Q + ql] : KEY_EMPTY;
    });
    if (j >= n_jobs || (warp & (W - 1)) != 0) return;
    if (M.accumulate) {
        // keys are (score << 32) | r: the offset moves r, never the score (r + offset < 2^32)
        if (acc != KEY_EMPTY) acc += (uint64_t)M.ref_offset;
        uint64_t run = KEY_EMPTY;
        if (lane < k) {
            const int64_t ri = jb.out_i[lane];
            if (ri >= 0) run = make_key(jb.out_s[lane], (uint32_t)ri);
        }
        acc = warp_merge32(acc, run, lane);
    }
    if (lane < k) {
        jb.out_s[lane] = acc == KEY_EMPTY ? 0xFFFFFFFFu : (uint32_t)(acc >> 32);
        jb.out_i[lane] = acc == KEY_EMPTY ? -1ll : (int64_t)(uint32_t)acc;
    }
}

// Streamed reference blocks: fold one block's lists (reference indices
// relative to the block, offset added here) into the running lists, one warp
// per query.  Both lists are ascending (score, reference) keys; a bitonic
// merge keeps the k smallest.
__global__ void topk_fold_kernel(uint32_t *__restrict__ run_s, int64_t *__restrict__ run_i,
                                 const uint32_t *__restrict__ blk_s, const int64_t *__restrict__ blk_i,
                                 int64_t offset, int64_t n_q, int32_t k) {
    const int lane = threadIdx.x & 31;
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= n_q) return;
    uint64_t a = KEY_EMPTY, b = KEY_EMPTY;
    if (lane < k) {
        const int64_t ia = run_i[q * k + lane];
        const int64_t ib = blk_i[q * k + lane];
        if (ia >= 0) a = make_key(run_s[q * k + lane], (uint32_t)ia);
        if (ib >= 0) b = make_key(blk_s[q * k + lane], (uint32_t)(ib + offset));
    }
    const uint64_t v = warp_merge32(a, b, lane);
    if (lane < k) {
        run_s[q * k + lane] = v == KEY_EMPTY ? 0xFFFFFFFFu : (uint32_t)(v >> 32);
        run_i[q * k + lane] = v == KEY_EMPTY ? -1ll : (int64_t)(uint32_t)v;
    }
}

// Streamed reference blocks, hit lists: after block b's hits are appended,
// snaps[b] = the count; the hits appended by block b, positions
// [snaps[b - 1], min(snaps[b], capacity)), get the block's first reference
// index added.
__global__ void hits_snap_kernel(const unsigned long long *__restrict__ count, unsigned long long *__restrict__ snap) {
    *snap = *count;
}

__global__ void hits_offset_kernel(const unsigned long long *__restrict__ snaps, int64_t b, int64_t capacity,
                                   int64_t *__restrict__ hit_r, int64_t r0) {
    const unsigned long long lo = b > 0 ? snaps[b - 1] : 0ull;
    const unsigned long long hi = min(snaps[b], (unsigned long long)capacity);
    for (unsigned long long i = lo + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < hi;
         i += (unsigned long long)gridDim.x * blockDim.x)
        hit_r[i] += r0;
}

// ---- hit list finish ----------------------------------------------------
// The list is sorted by (q, r) with a least-significant-digit radix sort on
// the key q << r_bits | r, in an even number of passes so that it leaves the
// caller's buffers for the scratch arrays and ends in them.  A block takes
// 2^rs_shift consecutive elements (at least RS_TILE, at most RS_BLOCKS
// blocks); table[p][block][digit] holds each block's digit counts for pass p,
// counted by a kernel of its own for the first pass and by the previous
// pass's scatter (which knows every element's place in the next order) for
// the others, so that a pass is one launch.  Everything is sized on the device
// by the live count.  (A bitonic sort over the buffer's capacity took 57
// launches and ~240 us for 60,000 hits in a buffer of 2^20, 1 ms in one of
// 2^21, whatever the count; the count kernel and four passes take ~53 us, half
// of it the global atomics of the next counts: a kernel of its own for those
// would cost as much.)
// Up to RS_FEW hits the count kernel's first block sorts them itself, each
// hit's place being the number of hits before it, and the passes have nothing
// to do: their latencies alone (19 us for two hits, where the bitonic sort of a
// small buffer took 3) were a third of a small call.
constexpr int RS_BITS = 8;
constexpr int RS_DIGITS = 1 << RS_BITS;
constexpr int RS_THREADS = 1024;
constexpr int RS_ITEMS = 4;  // elements a thread
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_GROUPS = RS_THREADS / RS_DIGITS;
constexpr int RS_FEW = 512;
constexpr int RS_BLOCKS = 256;  // about what fits the GPU at once (two a SM); every block reads every block's counts

__device__ __forceinline__ int64_t hits_live(const unsigned long long *count, int64_t capacity) {
    const unsigned long long c = *count;
    return (int64_t)(c < (unsigned long long)capacity ? c : (unsigned long long)capacity);
}

// log2 of a block's elements
__device__ __forceinline__ int rs_shift(int64_t n) {
    int sh = 12;
    while (((n + ((int64_t)1 << sh) - 1) >> sh) > RS_BLOCKS) ++sh;
    return sh;
}
static_assert(RS_TILE == 1 << 12, "rs_shift starts at one tile");

// The true count to the caller, the overflow condition, and the first pass's
// digit counts -- or the sorted list, where the hits are few.
__global__ void __launch_bounds__(RS_THREADS) hits_count_kernel(const unsigned long long *__restrict__ count,
                                                                int64_t capacity, int64_t *__restrict__ count_out,
                                                                uint32_t *__restrict__ status,
                                                                int64_t *__restrict__ hq, int64_t *__restrict__ hr,
                                                                uint32_t *__restrict__ hs, int r_bits,
                                                                uint32_t *__restrict__ table) {
    pdl_trigger();
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long c = *count;
        *count_out = (int64_t)c;
        if (c > (unsigned long long)capacity) atomicOr(status, ST_OVERFLOW);
    }
    const int64_t n = hits_live(count, capacity);
    const int sh = rs_shift(n);
    const int64_t b0 = (int64_t)blockIdx.x << sh;
    if (b0 >= n) return;
    if (n <= RS_FEW) {  // (one block)
        __shared__ uint64_t keys[RS_FEW];
        const int i = threadIdx.x, live = (int)n;
        uint64_t key = 0;
        uint32_t score = 0;
        if (i < live) {
            key = ((uint64_t)hq[i] << r_bits) | (uint64_t)hr[i];
            score = hs[i];
            keys[i] = key;
        }
        __syncthreads();
        if (i >= live) return;
        int at = 0;
#pragma unroll 8
        for (int j = 0; j < live; ++j) at += keys[j] < key || (keys[j] == key && j < i);
        hq[at] = (int64_t)(key >> r_bits);
        hr[at] = (int64_t)(key & ((1ull << r_bits) - 1ull));
        hs[at] = score;
        return;
    }
    __shared__ uint32_t cnt[RS_DIGITS];
    if (threadIdx.x < RS_DIGITS) cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t i = b0 + threadIdx.x; i < min(n, b0 + ((int64_t)1 << sh)); i += RS_THREADS) {
        const uint64_t key = ((uint64_t)hq[i] << r_bits) | (uint64_t)hr[i];
        atomicAdd(&cnt[key & (RS_DIGITS - 1)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < RS_DIGITS) table[(int64_t)blockIdx.x * RS_DIGITS + threadIdx.x] = cnt[threadIdx.x];
}

// One pass: digit (key >> shift) & 255.  FIRST reads the caller's (q, r,
// score) triples, LAST writes them; passes between use keys and scores.
// table: this pass's counts; next: the next pass's (zero before), unused
// when LAST.
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(RS_THREADS)
    hits_scatter_kernel(const unsigned long long *__restrict__ count, int64_t capacity, int r_bits, int shift,
                        const uint32_t *__restrict__ table, uint32_t *__restrict__ next,
                        const uint64_t *__restrict__ src_k, const int64_t *__restrict__ src_r,
                        const uint32_t *__restrict__ src_v, uint64_t *__restrict__ dst_k, int64_t *__restrict__ dst_r,
                        uint32_t *__restrict__ dst_v) {
    pdl_trigger();
    pdl_wait();
    const int64_t n = hits_live(count, capacity);
    if (n <= RS_FEW) return;  // sorted already
    const int sh = rs_shift(n);
    const int64_t b0 = (int64_t)blockIdx.x << sh, b1 = min(n, b0 + ((int64_t)1 << sh));
    if (b0 >= n) return;
    __shared__ uint16_t cnt[RS_WARPS][RS_DIGITS];  // of the tile, then each (warp, digit)'s first place in it
    __shared__ uint64_t part[2][RS_GROUPS][RS_DIGITS];
    __shared__ uint64_t place[RS_DIGITS];  // where this block's next element of a digit goes
    __shared__ uint64_t wsum[RS_DIGITS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {  // digit counts of every block, and of the blocks before this one
        const int nb = (int)((n + ((int64_t)1 << sh) - 1) >> sh), d = tid % RS_DIGITS, g = tid / RS_DIGITS;
        uint64_t tot = 0, pre = 0;
#pragma unroll 8
        for (int b = g; b < nb; b += RS_GROUPS) {
            const uint32_t c = table[(int64_t)b * RS_DIGITS + d];
            tot += c;
            pre += b < (int)blockIdx.x ? c : 0u;
        }
        part[0][g][d] = tot;
        part[1][g][d] = pre;
    }
    __syncthreads();
    uint64_t before = 0, incl = 0;
    if (tid < RS_DIGITS) {  // smaller digits anywhere, then this digit in earlier blocks
        uint64_t t = 0;
        for (int i = 0; i < RS_GROUPS; ++i) t += part[0][i][tid], before += part[1][i][tid];
        incl = t;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t x = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += x;
        }
        if (lane == 31) wsum[warp] = incl;
        before += incl - t;
    }
    __syncthreads();
    if (tid < RS_DIGITS) {
        for (int w = 0; w < warp; ++w) before += wsum[w];
        place[tid] = before;
    }
    for (int64_t t0 = b0; t0 < b1; t0 += RS_TILE) {
        // Elements in order: warp w takes 32 RS_ITEMS consecutive ones, 32 at a time.
        uint64_t key[RS_ITEMS];
        uint32_t val[RS_ITEMS], rank[RS_ITEMS];
        const int64_t i0 = t0 + warp * (32 * RS_ITEMS) + lane;
#pragma unroll
        for (int it = 0; it < RS_ITEMS; ++it) {
            const int64_t i = i0 + it * 32;
            key[it] = 0;
            val[it] = 0;
            if (i < b1) {
                key[it] = FIRST ? ((src_k[i] << r_bits) | (uint64_t)src_r[i]) : src_k[i];
                val[it] = src_v[i];
            }
        }
        for (int i = lane; i < RS_DIGITS; i += 32) cnt[warp][i] = 0;
        __syncwarp();
        // Rank within the warp: among equal digits, earlier elements first.
#pragma unroll
        for (int it = 0; it < RS_ITEMS; ++it) {
            const bool live = i0 + it * 32 < b1;
            const uint32_t dg = live ? (uint32_t)(key[it] >> shift) & (RS_DIGITS - 1) : RS_DIGITS;
            const uint32_t peers = __match_any_sync(0xffffffffu, dg);
            const uint32_t ahead = __popc(peers & ((1u << lane) - 1u));
            const uint32_t seen = live ? cnt[warp][dg] : 0u;
            __syncwarp();
            if (live && ahead == 0) cnt[warp][dg] = (uint16_t)(seen + __popc(peers));
            __syncwarp();
            rank[it] = seen + ahead;
        }
        __syncthreads();
        uint32_t in_tile = 0;  // this digit's elements in the tile
        if (tid < RS_DIGITS) {
#pragma unroll 8
            for (int w = 0; w < RS_WARPS; ++w) {
                const uint32_t c = cnt[w][tid];
                cnt[w][tid] = (uint16_t)in_tile;
                in_tile += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < RS_ITEMS; ++it) {
            if (i0 + it * 32 >= b1) break;
            const uint32_t dg = (uint32_t)(key[it] >> shift) & (RS_DIGITS - 1);
            const uint64_t pos = place[dg] + cnt[warp][dg] + rank[it];
            if (LAST) {
                dst_k[pos] = key[it] >> r_bits;
                dst_r[pos] = (int64_t)(key[it] & ((1ull << r_bits) - 1ull));
            } else {
                dst_k[pos] = key[it];
                atomicAdd(&next[(int64_t)(pos >> sh) * RS_DIGITS +
                                ((uint32_t)(key[it] >> (shift + RS_BITS)) & (RS_DIGITS - 1))],
                          1u);
            }
            dst_v[pos] = val[it];
        }
        __syncthreads();
        if (tid < RS_DIGITS) place[tid] += in_tile;
    }
}

int bits_for(int64_t n) {  // bits of n - 1
    int b = 0;
    while (b < 62 && (1ll << b) < n) ++b;
    return b;
}

int64_t hits_blocks(int64_t capacity) { return std::min<int64_t>(RS_BLOCKS, (capacity + RS_TILE - 1) / RS_TILE); }

}  // namespace

int hits_passes(int64_t n_q, int64_t n_refs) {
    const int bits = bits_for(n_q) + bits_for(n_refs);
    return std::max(2, 2 * ((bits + 2 * RS_BITS - 1) / (2 * RS_BITS)));
}

HitsLayout hits_layout(int64_t capacity, int passes) {
    HitsLayout L;
    L.table = 256;  // the counter's line first
    L.zero_bytes = L.table + (size_t)passes * hits_blocks(capacity) * RS_DIGITS * sizeof(uint32_t);
    L.keys = (L.zero_bytes + 255) & ~size_t(255);
    L.vals = L.keys + ((size_t)capacity * sizeof(uint64_t) + 255 & ~size_t(255));
    L.bytes = L.vals + (size_t)capacity * sizeof(uint32_t);
    return L;
}

// Warps per query for n_q queries of up to n lists: about MERGE_AHEAD lists a
// warp, so that one round of loads covers them, but no more warps than about
// two waves of the GPU's (152 SMs x 64): past that more warps a query only
// add shared-memory rounds (7165 queries of a 4-panel plan, up to 76 lists:
// 52 us with 16 warps each; one warp a query took 33 us).  One query of 149
// lists: 111 -> 8.9 us; 48 of 152: 119 -> 8.8; 32 of 304 (plain): 249 -> 11.7;
// 2048 of 10: 11.5 -> 10.5.
static int merge_warps(int64_t n_q, int64_t n_lists) {
    int W = 1;
    while (W < MERGE_MAX_WARPS && (int64_t)W * MERGE_AHEAD < n_lists && 2 * W * n_q <= 16384) W <<= 1;
    return W;
}

// Blocks of 8 warps, or of W where a query takes more.
static int merge_block_warps(int W) { return W > 8 ? W : 8; }

cudaError_t launch_topk_merge(const uint64_t *partial, const Partition &part, int64_t n_q, int32_t k,
                              uint32_t *out_scores, int64_t *out_idx, cudaStream_t s) {
    if (n_q == 0) return cudaSuccess;
    const int64_t n_qt = part.n_qt;
    const int W = merge_warps(n_q, (part.grid + n_qt - 1) / n_qt + 1), per = merge_block_warps(W) / W;
    return launch_dependent(topk_merge_kernel, dim3((unsigned)((n_q + per - 1) / per)), dim3(per * W * 32), 0, s, partial,
                            part, n_q, k, W, out_scores, out_idx);
}

cudaError_t launch_merge_sched(const uint64_t *partial, const TcLaunch &L, const MergeJob *jobs, int64_t n_jobs,
                               uint32_t *out_scores, int64_t *out_idx, cudaStream_t s, bool accumulate,
                               int64_t ref_offset) {
    if (n_jobs == 0) return cudaSuccess;
    MergeSched M;
    M.accumulate = accumulate ? 1 : 0;
    M.ref_offset = ref_offset;
    M.n_panels = L.n_panels;
    M.pair = L.pair;
    M.k = L.k;
    for (int p = 0; p < TC_MAXP; ++p) M.sc[p] = L.sched[p];
    M.n_slots = L.n_slots;
    M.status = L.status;
    M.qspread = L.qspread[0];
    int64_t n_lists = 1;
    for (int p = 0; p < L.n_panels; ++p)
        n_lists = std::max<int64_t>(n_lists, L.sched[p].b + (L.sched[p].t_groups > 0 ? 1 : 0));
    const int W = merge_warps(n_jobs, n_lists), per = merge_block_warps(W) / W;
    const dim3 grid((unsigned)((n_jobs + per - 1) / per)), block(per * W * 32);
    return launch_dependent(topk_merge_sched_kernel, grid, block, 0, s, partial, M, jobs, n_jobs, W, out_scores, out_idx);
}

cudaError_t launch_topk_fold(uint32_t *run_s, int64_t *run_i, const uint32_t *blk_s, const int64_t *blk_i,
                             int64_t offset, int64_t n_q, int32_t k, cudaStream_t s) {
    if (n_q == 0) return cudaSuccess;
    const int wpb = 8;
    topk_fold_kernel<<<(unsigned)((n_q + wpb - 1) / wpb), wpb * 32, 0, s>>>(run_s, run_i, blk_s, blk_i, offset,
                                                                             n_q, k);
    return cudaGetLastError();
}

cudaError_t launch_hits_block_offset(const unsigned long long *count, unsigned long long *snaps, int64_t b,
                                     int64_t capacity, int64_t *hit_r, int64_t r0, int grid, cudaStream_t s) {
    hits_snap_kernel<<<1, 1, 0, s>>>(count, snaps + b);
    if (r0 != 0 && capacity > 0) hits_offset_kernel<<<grid, 256, 0, s>>>(snaps, b, capacity, hit_r, r0);
    return cudaGetLastError();
}

cudaError_t launch_hits_finish(void *aux, int64_t capacity, int64_t n_q, int64_t n_refs, int64_t *hit_q,
                               int64_t *hit_r, uint32_t *hit_score, int64_t *count_out, uint32_t *status,
                               cudaStream_t s) {
    const int passes = hits_passes(n_q, n_refs), r_bits = bits_for(n_refs);
    const HitsLayout L = hits_layout(capacity, passes);
    uint8_t *base = static_cast<uint8_t *>(aux);
    const unsigned long long *count = reinterpret_cast<unsigned long long *>(base);
    const int64_t nb = hits_blocks(capacity);
    uint32_t *table = reinterpret_cast<uint32_t *>(base + L.table);
    uint64_t *tk = reinterpret_cast<uint64_t *>(base + L.keys);
    uint32_t *tv = reinterpret_cast<uint32_t *>(base + L.vals);
    const unsigned grid = (unsigned)std::max<int64_t>(1, nb);
    const dim3 blocks(grid), threads(RS_THREADS);
    cudaError_t e = launch_dependent(hits_count_kernel, blocks, threads, 0, s, count, capacity, count_out, status, hit_q,
                                     hit_r, hit_score, r_bits, table);
    if (capacity == 0) return e;
    uint64_t *hk = reinterpret_cast<uint64_t *>(hit_q);
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        const uint32_t *now = table + (int64_t)p * nb * RS_DIGITS;
        uint32_t *next = p + 1 < passes ? table + (int64_t)(p + 1) * nb * RS_DIGITS : nullptr;
        const int shift = p * RS_BITS;
        int64_t *none = nullptr;
        if (p == 0)
            e = launch_dependent(hits_scatter_kernel<true, false>, blocks, threads, 0, s, count, capacity, r_bits, shift,
                                 now, next, hk, hit_r, hit_score, tk, none, tv);
        else if (p + 1 == passes)
            e = launch_dependent(hits_scatter_kernel<false, true>, blocks, threads, 0, s, count, capacity, r_bits, shift,
                                 now, next, tk, none, tv, hk, hit_r, hit_score);
        else if (p & 1)
            e = launch_dependent(hits_scatter_kernel<false, false>, blocks, threads, 0, s, count, capacity, r_bits,
                                 shift, now, next, tk, none, tv, hk, none, hit_score);
        else
            e = launch_dependent(hits_scatter_kernel<false, false>, blocks, threads, 0, s, count, capacity, r_bits,
                                 shift, now, next, hk, none, hit_score, tk, none, tv);
    }
    return e;
}

}  // namespace fastid
