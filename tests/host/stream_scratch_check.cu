// Host check of a streamed call's scratch: what it sets aside before it starts
// (stream_scratch_bytes) covers the scratch of every block's comparison
// (tensor_scratch_bytes), whose sizes follow from each block's own schedule.
// The walk over the blocks is restated here.  No GPU call is made.  Exit status
// 0 = all pass.
#include <algorithm>
#include <cstdio>

#include "internal.h"

using namespace fastid;

int main() {
    fastid_ctx ctx;
    ctx.grid_tensor = 152;
    int bad = 0, cases = 0;
    for (int pairs : {0, 10, 76})
        for (int32_t n_loci : {64, 512, 2048, 16384, 65536})
            for (int64_t n_q : {129, 200, 512, 2048, 30000, 200000})
                for (int32_t k : {0, 1, 10, 16, 32})
                    for (int64_t block : {1ll, 255ll, 256ll, 2049ll, 70000ll, 1ll << 20, 1ll << 22})
                        for (int64_t n_refs : {1ll, 300ll, 2048ll, 1000003ll, 20000000ll}) {
                            if (n_refs / block > 2000) continue;
                            ctx.pair_clusters = pairs;
                            fastid_refdb db;
                            db.n_loci = n_loci;
                            db.n_words64 = (n_loci + 63) / 64;
                            db.ld64 = (db.n_words64 + 7) / 8 * 8;
                            db.kpad = tensor_kpad(n_loci);
                            db.kbytes4 = tensor_kbytes4(n_loci);
                            const int64_t most = std::min(block, n_refs);
                            const size_t got = stream_scratch_bytes(&ctx, db, n_refs, most, n_q, k, OP_FP4);
                            size_t need = 0;
                            int64_t r0 = 0, next = std::max<int64_t>(std::min<int64_t>(most, ROW_ALIGN), most / 8);
                            int64_t seen = -1;
                            while (r0 < n_refs) {
                                db.n_refs = std::min(next, n_refs - r0);
                                next = std::min(most, 2 * next);
                                r0 += db.n_refs;
                                db.n_pad = (db.n_refs + ROW_ALIGN - 1) / ROW_ALIGN * ROW_ALIGN;
                                if (db.n_refs != seen) need = std::max(need, tensor_scratch_bytes(&ctx, &db, n_q, k, OP_FP4));
                                seen = db.n_refs;
                            }
                            ++cases;
                            if (need == 0 || got < need || got > need) {
                                printf("N %d n_q %lld k %d block %lld n_refs %lld: %zu for %zu\n", n_loci, (long long)n_q, k,
                                       (long long)block, (long long)n_refs, got, need);
                                ++bad;
                            }
                        }
    printf("cases %d bad %d\n", cases, bad);
    return bad != 0;
}
