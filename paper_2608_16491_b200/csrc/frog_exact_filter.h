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
    int* first;              // per round: its first query; then the number of queries
    uint32_t* store;
    int rounds;
    unsigned long long step; // a round's share of the words of all queries, laid end to end
};

// Scratch for nq queries of any width in one round.
size_t filter_bytes(size_t n, size_t nq, int k, int d_pad);
// How so many bytes serve: a call goes in parts of `queries` (0: not at all), a part in rounds, of which as many do
// something as the widths ask for; per_round: queries of the widest slabs in a round.
struct FilterFit {
    size_t queries, parts, rounds, per_round, step;
};
FilterFit filter_fit(size_t n, size_t nq, size_t bytes, int k, int d_pad);
void filter_scratch(char* mem, FilterArgs* A);
cudaError_t filter_launch(const FilterArgs& A, int sm_count, cudaStream_t s);

}  // namespace froghost
