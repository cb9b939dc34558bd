// What tests set in a context that the C ABI does not offer; compiled against
// the library's internal header and called with a context's handle.
#include "few.h"
#include "internal.h"

extern "C" {

// Most bytes that a streamed call's FP4 block operands may take (negative: the
// library's own rule).
void hook_fp4_block_bytes(fastid_ctx *ctx, int64_t bytes) { ctx->fp4_block_bytes = bytes; }

// Top-k calls over packed rows: 0 the library's rule, 1 the few-query form
// wherever it fits, -1 never.
void hook_few_rule(fastid_ctx *ctx, int32_t rule) { ctx->few_rule = rule; }

// Packed stages of the few-query form for such a call; 0: it does not fit.
int32_t hook_few_stages(int64_t n_q, int32_t n_loci, int32_t k) {
    fastid::FewShape S;
    return fastid::few_shape(n_q, n_loci, k, &S) ? S.stages : 0;
}

// The library's rule for it: k deep, over n_refs packed rows of row_bytes.
int32_t hook_few_pays(int64_t n_q, int32_t k, int64_t n_refs, int64_t row_bytes) {
    return fastid::few_pays(n_q, k, n_refs, row_bytes);
}

// Whether a plain launch's CTAs take every place of a GPU that holds `places`
// of them.
int32_t hook_plain_fills(int32_t places, int32_t tile_q, int64_t n_q, int64_t n_refs) {
    const int64_t n_rt = (n_refs + fastid::ROW_ALIGN - 1) / fastid::ROW_ALIGN * (fastid::ROW_ALIGN / fastid::PL_TR);
    const fastid::Partition p = fastid::make_partition(tile_q, n_q, n_rt, places);
    return p.fills;
}

// Row bytes of an FP4 operand.
int32_t hook_kbytes4(int32_t n_loci) { return fastid::tensor_kbytes4(n_loci); }
}
