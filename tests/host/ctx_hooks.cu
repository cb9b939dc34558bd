// What tests set in a context that the C ABI does not offer; compiled against
// the library's internal header and called with a context's handle.
#include "internal.h"

extern "C" {

// Most bytes that a streamed call's FP4 block operands may take (negative: the
// library's own rule).
void hook_fp4_block_bytes(fastid_ctx *ctx, int64_t bytes) { ctx->fp4_block_bytes = bytes; }

// Row bytes of an FP4 operand.
int32_t hook_kbytes4(int32_t n_loci) { return fastid::tensor_kbytes4(n_loci); }
}
