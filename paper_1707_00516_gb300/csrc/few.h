// Few-query form (few.cu): host interface.
#pragma once

#include "common.cuh"

namespace fastid {

// Shape of a call: the MMA's columns (queries rounded up to 16), chunks of 256
// loci, packed stages in flight.
struct FewShape {
    int32_t ncols, n_kb, stages;
};

// Whether the form takes the call: at most 64 queries, which with their lists
// and at least four packed stages fit an SM's shared memory.
bool few_shape(int64_t n_q, int32_t n_loci, int32_t k, FewShape *S);

// Whether it is the faster for a call that it fits: k deep, over n_refs packed
// rows of row_bytes.
bool few_pays(int64_t n_q, int32_t k, int64_t n_refs, int64_t row_bytes);

struct FewLaunch {
    const uint64_t *q;  // packed queries
    int64_t ld_q, n_q;
    int32_t n_words, n_loci;
    const uint8_t *modes;
    uint8_t *operand;    // [ncols][n_kb * 128]
    float *qconst;       // [ncols]
    SharedCut cut;       // out: [ncols]
    const uint64_t *packed;
    int64_t n_pad, ld64, n_refs;
    int32_t k;
    uint32_t threshold;
    int32_t slices;      // CTAs
    int32_t *pub;        // [ncols][slices]
    uint64_t *partial;   // [slices][k][128]
    uint32_t *status;
};

// The query operand, constants and starting cuts; then the compare kernel.
cudaError_t launch_few_seed(const FewLaunch &L, const FewShape &S, cudaStream_t s);
cudaError_t launch_few(const FewLaunch &L, const FewShape &S, cudaStream_t s);

}  // namespace fastid
