// The exact scan of many queries by tensor cores and comparison of what is left (frog_exact_filter.cu).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace froghost {

struct FilterArgs {
    const int32_t* sorted_attr;
    const int32_t* rank2id;
    const float* vectors;
    int n, d, d_pad;
    const float* queries;
    const int32_t* lo;
    const int32_t* hi;
    int nq, k;
    int32_t* out_ids;
    float* out_dists;
    // scratch, in this order (filter_scratch)
    float* rounded;          // nq x d_pad: the queries in tf32
    int2* slab;              // per query: first and last rank
    float* norm;             // squared
    uint32_t* off;           // where its values, then its masks, begin in `store`
    float* tau;              // no answer is farther
    uint32_t* tile_norm;     // per 128 rows: the largest squared norm (bits); infinite where a rough distance is not finite
    uint32_t* store;
    size_t words;            // of `store`
};

// Scratch bytes of a call: what it cannot do without (the rest is used as far as it goes) and what covers every case.
struct FilterRoom {
    size_t least, most;
};
FilterRoom filter_room(size_t n, size_t nq, int k, int d_pad);
void filter_scratch(char* mem, size_t bytes, FilterArgs* A);
cudaError_t filter_launch(const FilterArgs& A, int sm_count, cudaStream_t s);

}  // namespace froghost
