// Kernel 1's sort by buckets (bucket.cu).
#pragma once

#include "internal.h"

namespace gb {

// Bits of the first and the second digit (0: one digit only).
struct BucketPlan {
    int p0, p1;
};

// Whether m tuples of 2^scale vertices can be built by buckets, and how: fewer
// than 2^32 directed entries, and what two digits of at most 10 bits leave of a
// key fits 32 bits (SCALE 26 and less; with weights 64 bits, SCALE 24 and less).
bool bucket_plan(int64_t m, int scale, bool weighted, BucketPlan *out);

// The CSR (and, with w, the weights) of the tuples into g, and its auxiliary
// arrays.  Synchronises the stream.
gb_status bucket_build(const int64_t *edges, const float *w, int64_t m, int scale, const BucketPlan &plan, gb_graph *g,
                       cudaStream_t s);

// Whether the rows of nnz entries can be ordered by weight by buckets (fewer than 2^32).
bool bucket_order_fits(int64_t nnz);
// (column, weight) of every entry of g into wadj, each row by ascending weight
// (ties by column).  The caller synchronises the stream.
gb_status bucket_weight_order(const gb_graph *g, uint2 *wadj, cudaStream_t s);

}  // namespace gb
