// frog_exact_search: exact filtered kNN (paper Def. 2) by scanning each query's contiguous rank
// slab (Sec. 4).  Ordering: (squared distance, original object id) ascending, the total order of Def. 2's
// tie rule (objects with equal attributes are ranked by id, so this differs from rank order only between
// equidistant objects with different attributes).
//
// A CTA scans a piece of the rows for a GROUP of queries and keeps the k nearest of each:
//   * a team of 8 lanes holds two rows in registers and computes their distances to every query of the group
//     (queries in shared memory), so a row is fetched once per group;
//   * a distance that beats the query's bound goes to the query's buffer; one warp per query merges the
//     buffer into the query's pool when it fills (a few times per piece) and lowers the bound.  The bound is
//     shared by all pieces of a query through global memory: whatever exceeds the k-th best of ANY piece
//     cannot be an answer;
//   * the last CTA to finish a group merges the pieces' lists.
// Many queries on all but small indexes are filtered first (frog_exact_filter.cu).
// Few queries are not grouped: all rows are cut into equal pieces, one query each (one launch for fewer than
// EXACT_PLAN_MIN, else a planning kernel finds the slabs first).  Otherwise queries are ordered by (width, position),
// grouped by eight, and the groups' rows are cut into pieces of equal size (two small kernels).  The form with one CTA
// per query and no scratch remains for small indexes, for captured streams, for rows too long for eight queries in
// shared memory, and for the case that scratch cannot be had.  exact_form says where the lines lie.
#include <algorithm>

#include "frog_device.cuh"
#include "frog_exact_filter.h"
#include "frog_internal.h"

using namespace frogdev;

namespace {

constexpr int EXACT_WARPS = 8;
constexpr int EXACT_GROUP = 8;           // queries per group = warps per CTA (one merges each query's buffer)
constexpr int EXACT_SPLIT_MAX = 200;     // queries that the split form can cut between
constexpr size_t EXACT_GROW_BYTES = (size_t)16 << 20;   // see exact_scratch
constexpr int EXACT_PLAN_MIN = 17;       // from here on a planning kernel finds the slabs (100,000 x 96, 16 queries: 49 us without)
constexpr int EXACT_STEP = 8 * EXACT_WARPS;    // rows per step of a CTA: two per team
constexpr int EXACT_BUF = 256;           // keys buffered per query; merged from 64 on, two steps add at most 128
constexpr int EXACT_BINS = 33 * 32;      // (width class, position) bins that queries are ordered by

struct ExactArgs {
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
    // scratch (see exact_scratch); unused by the form with one CTA per query
    int2* ranges;
    int32_t* order;
    int4* jobs;                      // (group, first row, end row, unused)
    int2* groups;                    // (first piece, pieces)
    unsigned int* counters;          // [0] pieces of this call, [1] next piece: set per call; [2..] bins, zero between calls
    unsigned int* done;              // finished pieces per group (or query); zero between calls
    unsigned long long* bound;       // per query: k-th best key of any piece; all ones between calls
    uint64_t* part;                  // per piece and query of the group: k keys
    int max_pieces, min_rows;
};

template <int EPL, int G>
struct ExactSmem {
    uint64_t* pool;      // G x 32 EPL
    uint64_t* buf;       // G x EXACT_BUF
    uint64_t* tau;       // G: keys above it are not wanted
    int* cnt;            // G: keys in buf
    int* l;              // G: first rank
    int* r;              // G: last rank
    int* id;             // G: query number, -1 = none
    int* misc;           // 8
    float4* q;           // G x d_pad floats
    static constexpr size_t FIXED = (size_t)G * (32 * EPL + EXACT_BUF + 1) * 8 + (size_t)G * 16 + 32;
    static __host__ __device__ size_t bytes(int d_pad) { return (FIXED + 15) / 16 * 16 + (size_t)G * d_pad * 4; }
    __device__ __forceinline__ explicit ExactSmem(unsigned char* base) {
        pool = reinterpret_cast<uint64_t*>(base);
        buf = pool + G * 32 * EPL;
        tau = buf + G * EXACT_BUF;
        cnt = reinterpret_cast<int*>(tau + G);
        l = cnt + G;
        r = l + G;
        id = r + G;
        misc = id + G;
        q = reinterpret_cast<float4*>(base + (FIXED + 15) / 16 * 16);
    }
};

// merge query `g`'s buffer into its pool (one warp) and lower its bound
template <int EPL, int G>
__device__ __forceinline__ void exact_flush(const ExactArgs& A, const ExactSmem<EPL, G>& S, int g, int lane) {
    uint64_t* const pool = S.pool + g * 32 * EPL;
    const int n = S.cnt[g];
    for (int off = 0; off < n; off += 32)
        merge_ranked<EPL>(pool, S.buf + g * EXACT_BUF + off, min(32, n - off), A.k, lane);
    uint64_t kth = pool[A.k - 1];
    if (S.id[g] >= 0) {
        unsigned long long seen = 0;
        if (lane == 0) {
            if (n > 0 && kth != KEY_EMPTY) atomicMin(A.bound + S.id[g], (unsigned long long)kth);
            seen = __ldcg(A.bound + S.id[g]);
        }
        seen = __shfl_sync(FULL, seen, 0);
        kth = min(kth, (uint64_t)seen);
    }
    __syncwarp();
    if (lane == 0) {
        S.tau[g] = kth;
        S.cnt[g] = 0;
    }
}

// squares of a row's chunk against a query's, four groups of four elements
template <bool FULL_CHUNK>
__device__ __forceinline__ float exact_chunk(float acc, const float4 (&x)[4], const float4* q, int left) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (FULL_CHUNK || 8 * c < left) {
            const float4 v = q[8 * c];
            float t;
            t = x[c].x - v.x; acc = fmaf(t, t, acc);
            t = x[c].y - v.y; acc = fmaf(t, t, acc);
            t = x[c].z - v.z; acc = fmaf(t, t, acc);
            t = x[c].w - v.w; acc = fmaf(t, t, acc);
        }
    }
    return acc;
}

// exact_scan for a single query: four rows per team, 16 per warp in flight (bounded by row bytes).
template <int EPL>
__device__ __forceinline__ void exact_scan_one(const ExactArgs& A, const ExactSmem<EPL, 1>& S, int row0, int row1) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int team = lane >> 3, sub = lane & 7;
    const int groups = A.d_pad >> 2;
    for (int b = row0; b < row1; b += 2 * EXACT_STEP) {
        const int base = b + warp * 16, end = min(base + 16, row1);
        if (base < row1) {                                   // warp-uniform
            const float4* row = reinterpret_cast<const float4*>(A.vectors + (size_t)(base + team) * (size_t)A.d_pad) + sub;
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int g0 = 0; g0 < groups; g0 += 32) {
                float4 x[4][4];
                const int left = groups - g0 - sub;          // groups of the row from this lane's first on
                const float4* qv = S.q + g0 + sub;
                if (g0 + 32 <= groups && end == base + 16) {
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) x[r][c] = __ldg(row + (size_t)r * groups * 4 + g0 + 8 * c);
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[r] = exact_chunk<true>(acc[r], x[r], qv, left);
                } else {
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            x[r][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (base + 4 * r + team < row1 && 8 * c < left) x[r][c] = __ldg(row + (size_t)r * groups * 4 + g0 + 8 * c);
                        }
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[r] = exact_chunk<false>(acc[r], x[r], qv, left);
                }
            }
            // the butterfly 4, 2, 1 over the team, every lane handing on the sums it does not keep: half of the
            // rows after partner distance 4, one row after 2
            const bool up4 = (sub & 4) != 0, up2 = (sub & 2) != 0;
            float s1[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float give = up4 ? acc[r] : acc[r + 2], keep = up4 ? acc[r + 2] : acc[r];
                s1[r] = keep + __shfl_xor_sync(FULL, give, 4);
            }
            const float give = up2 ? s1[0] : s1[1], keep = up2 ? s1[1] : s1[0];
            float d = keep + __shfl_xor_sync(FULL, give, 2);
            d = d + __shfl_xor_sync(FULL, d, 1);
            const int mine = base + 4 * ((up4 ? 2 : 0) + (up2 ? 1 : 0)) + team;
            if ((sub & 1) == 0 && mine < row1 && __float_as_uint(d) <= (uint32_t)(S.tau[0] >> 32)) {
                const uint64_t key = make_key(d, (uint32_t)__ldg(A.rank2id + mine), 1u);
                if (key < S.tau[0]) S.buf[atomicAdd(&S.cnt[0], 1)] = key;
            }
        }
        __syncthreads();
        const bool full = S.cnt[0] >= 64;
        __syncthreads();
        if (full) {
            if (warp == 0) exact_flush<EPL, 1>(A, S, 0, lane);
            __syncthreads();
        }
    }
    if (warp == 0) exact_flush<EPL, 1>(A, S, 0, lane);
    __syncthreads();
}

// merge what may be among the k best of the pieces' lists into a single query's pool (one warp); eight loads per
// lane are in flight at once
template <int EPL>
__device__ __forceinline__ void exact_gather(const ExactArgs& A, const ExactSmem<EPL, 1>& S, int first, int pieces, int lane) {
    const unsigned long long* const lists = reinterpret_cast<const unsigned long long*>(A.part) + (size_t)first * A.k;
    uint64_t* const pool = S.pool;
    uint64_t* const buf = S.buf;
    const unsigned int n = (unsigned int)pieces * (unsigned int)A.k;
    uint64_t tau = (uint64_t)__ldcg(A.bound + S.id[0]);
    int c = 0;
    for (unsigned int off = 0; off < n; off += 256) {
        uint64_t key[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const unsigned int x = off + 32 * i + lane;
            key[i] = KEY_EMPTY;
            if (x < n) key[i] = (uint64_t)__ldcg(lists + x);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t M = __ballot_sync(FULL, key[i] != KEY_EMPTY && key[i] <= tau);
            if ((M >> lane) & 1u) buf[c + __popc(M & ((1u << lane) - 1u))] = key[i];
            c += __popc(M);
            __syncwarp();
            if (c >= 32) {
                for (int x = 0; x < c; x += 32) merge_ranked<EPL>(pool, buf + x, min(32, c - x), A.k, lane);
                tau = min(tau, pool[A.k - 1]);
                c = 0;
                __syncwarp();
            }
        }
    }
    if (c > 0) merge_ranked<EPL>(pool, buf, c, A.k, lane);
    __syncwarp();
}

// The rows [row0, row1) of the group whose slabs and queries are in S; the pools hold the result.
// Bounded by fp32 issue where rows are shared (8 queries) and by row bytes where they are not.
template <int EPL, int G>
__device__ __forceinline__ void exact_scan(const ExactArgs& A, const ExactSmem<EPL, G>& S, int row0, int row1) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int team = lane >> 3, sub = lane & 7;
    const int groups = A.d_pad >> 2;
    for (int b = row0; b < row1;) {
        // rows that no query wants are jumped over
        int next = row1;
        bool any = false;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            any = any || (S.l[g] < b + 2 * EXACT_STEP && S.r[g] >= b);
            if (S.l[g] >= b && S.l[g] <= S.r[g]) next = min(next, S.l[g]);
        }
        if (!any) { b = next; continue; }
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const int base = b + half * EXACT_STEP + warp * 8;
            unsigned int cover = 0;                          // queries that want one of the 8 rows
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (S.l[g] < min(base + 8, row1) && S.r[g] >= base) cover |= 1u << g;
            if (base >= row1 || cover == 0) continue;
            const int rowA = base + team, rowB = rowA + 4;
            const bool vA = rowA < row1, vB = rowB < row1;
            const float4* pA = reinterpret_cast<const float4*>(A.vectors + (size_t)rowA * (size_t)A.d_pad);
            const float4* pB = reinterpret_cast<const float4*>(A.vectors + (size_t)rowB * (size_t)A.d_pad);
            float acc[2][G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[0][g] = acc[1][g] = 0.f;
#pragma unroll 1
            for (int g0 = 0; g0 < groups; g0 += 32) {
                float4 xa[4], xb[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int i = g0 + 8 * c + sub;
                    xa[c] = xb[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (vA && i < groups) xa[c] = __ldg(pA + i);
                    if (vB && i < groups) xb[c] = __ldg(pB + i);
                }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if ((cover >> g) & 1u) {
                        const float4* qv = S.q + g * groups;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int i = g0 + 8 * c + sub;
                            if (i < groups) {
                                const float4 q = qv[i];
                                float t;
                                t = xa[c].x - q.x; acc[0][g] = fmaf(t, t, acc[0][g]);
                                t = xb[c].x - q.x; acc[1][g] = fmaf(t, t, acc[1][g]);
                                t = xa[c].y - q.y; acc[0][g] = fmaf(t, t, acc[0][g]);
                                t = xb[c].y - q.y; acc[1][g] = fmaf(t, t, acc[1][g]);
                                t = xa[c].z - q.z; acc[0][g] = fmaf(t, t, acc[0][g]);
                                t = xb[c].z - q.z; acc[1][g] = fmaf(t, t, acc[1][g]);
                                t = xa[c].w - q.w; acc[0][g] = fmaf(t, t, acc[0][g]);
                                t = xb[c].w - q.w; acc[1][g] = fmaf(t, t, acc[1][g]);
                            }
                        }
                    }
                }
            }
            // the butterfly 4, 2, 1 over the team, every lane handing on the sums it does not keep: after
            // partner distance 4 a lane has one row, after 2 half of the queries, after 1 a quarter
            const bool up4 = (sub & 4) != 0;
            float s1[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const float give = up4 ? acc[0][g] : acc[1][g], keep = up4 ? acc[1][g] : acc[0][g];
                s1[g] = keep + __shfl_xor_sync(FULL, give, 4);
            }
            const int row = up4 ? rowB : rowA;
            constexpr int NK = G / 4;
            float fin[NK];
            int g_lo = 0;
            const bool emits = row < row1;
            {
                const bool up2 = (sub & 2) != 0, up1 = (sub & 1) != 0;
                float s2[G / 2];
#pragma unroll
                for (int g = 0; g < G / 2; ++g) {
                    const float give = up2 ? s1[g] : s1[g + G / 2], keep = up2 ? s1[g + G / 2] : s1[g];
                    s2[g] = keep + __shfl_xor_sync(FULL, give, 2);
                }
#pragma unroll
                for (int g = 0; g < G / 4; ++g) {
                    const float give = up1 ? s2[g] : s2[g + G / 4], keep = up1 ? s2[g + G / 4] : s2[g];
                    fin[g] = keep + __shfl_xor_sync(FULL, give, 1);
                }
                g_lo = (up2 ? G / 2 : 0) + (up1 ? G / 4 : 0);
            }
#pragma unroll
            for (int x = 0; x < NK; ++x) {
                const int g = g_lo + x;
                const uint64_t tau = S.tau[g];
                if (emits && row >= S.l[g] && row <= S.r[g] && __float_as_uint(fin[x]) <= (uint32_t)(tau >> 32)) {
                    const uint64_t key = make_key(fin[x], (uint32_t)__ldg(A.rank2id + row), 1u);
                    if (key < tau) S.buf[g * EXACT_BUF + atomicAdd(&S.cnt[g], 1)] = key;
                }
            }
        }
        b += 2 * EXACT_STEP;
        __syncthreads();
        bool full = false;
#pragma unroll
        for (int g = 0; g < G; ++g) full = full || S.cnt[g] >= 64;
        __syncthreads();
        if (full) {
            if (warp < G) exact_flush<EPL, G>(A, S, warp, lane);
            __syncthreads();
        }
    }
    if (warp < G) exact_flush<EPL, G>(A, S, warp, lane);
    __syncthreads();
}

template <int EPL>
__device__ __forceinline__ void exact_output(const ExactArgs& A, const uint64_t* pool, int q, int lane) {
    for (int j = lane; j < A.k; j += 32) {
        const uint64_t key = pool[j];
        int32_t oid = -1;
        float dist = __int_as_float(0x7F800000);
        if (key != KEY_EMPTY) {
            oid = (int32_t)key_rank(key);
            dist = __fsqrt_rn(key_dist2(key));
        }
        A.out_ids[(size_t)q * A.k + j] = oid;
        A.out_dists[(size_t)q * A.k + j] = dist;
    }
}

// One piece: queries S.id[] with slabs S.l/S.r, rows [row0, row1), `pieces` pieces from `first` on belong to
// the group, whose count of finished pieces is *done.
template <int EPL, int G>
__device__ __forceinline__ void exact_piece(const ExactArgs& A, const ExactSmem<EPL, G>& S, int row0, int row1, int piece,
                                            int first, int pieces, unsigned int* done) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    for (int g = 0; g < G; ++g) {
        float* qf = reinterpret_cast<float*>(S.q) + (size_t)g * A.d_pad;
        const float* src = A.queries + (size_t)max(S.id[g], 0) * A.d;
        for (int i = threadIdx.x; i < A.d_pad; i += EXACT_WARPS * 32) qf[i] = i < A.d && S.id[g] >= 0 ? __ldg(src + i) : 0.f;
    }
    for (int i = threadIdx.x; i < G * 32 * EPL; i += EXACT_WARPS * 32) S.pool[i] = KEY_EMPTY;
    if (threadIdx.x < G) {
        S.cnt[threadIdx.x] = 0;
        S.tau[threadIdx.x] = S.id[threadIdx.x] >= 0 ? (uint64_t)__ldcg(A.bound + S.id[threadIdx.x]) : KEY_EMPTY;
    }
    __syncthreads();
    if constexpr (G == 1) exact_scan_one<EPL>(A, S, row0, row1);
    else exact_scan<EPL, G>(A, S, row0, row1);
    if (pieces > 1) {
        if (warp < G) {
            const uint64_t tau = S.tau[warp];              // keys above it lose to another piece's
            uint64_t* out = A.part + ((size_t)piece * G + warp) * A.k;
            for (int j = lane; j < A.k; j += 32) {
                const uint64_t key = S.pool[warp * 32 * EPL + j];
                __stcg(reinterpret_cast<unsigned long long*>(out + j), (unsigned long long)(key <= tau ? key : KEY_EMPTY));
            }
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) S.misc[0] = atomicAdd(done, 1u) == (unsigned int)pieces - 1u;
        __syncthreads();
        if (!S.misc[0]) return;
        __threadfence();
        if constexpr (G == 1) {
            // (this piece's own list is read back too: the merge drops what the pool holds)
            if (warp == 0) exact_gather<EPL>(A, S, first, pieces, lane);
        } else if (warp < G && S.id[warp] >= 0) {
            uint64_t* const pool = S.pool + warp * 32 * EPL;
            uint64_t* const buf = S.buf + warp * EXACT_BUF;
            uint64_t tau = min((uint64_t)__ldcg(A.bound + S.id[warp]), pool[A.k - 1]);
            int c = 0;
            for (int p = first; p < first + pieces; ++p) {
                if (p == piece) continue;
                const unsigned long long* in =
                    reinterpret_cast<const unsigned long long*>(A.part) + ((size_t)p * G + warp) * A.k;
                for (int off = 0; off < A.k; off += 32) {
                    const uint64_t key = off + lane < A.k ? (uint64_t)__ldcg(in + off + lane) : KEY_EMPTY;
                    const uint32_t M = __ballot_sync(FULL, key != KEY_EMPTY && key <= tau);
                    if ((M >> lane) & 1u) buf[c + __popc(M & ((1u << lane) - 1u))] = key;
                    c += __popc(M);
                    __syncwarp();
                    if (c >= 32) {
                        for (int x = 0; x < c; x += 32) merge_ranked<EPL>(pool, buf + x, min(32, c - x), A.k, lane);
                        tau = min(tau, pool[A.k - 1]);
                        c = 0;
                        __syncwarp();
                    }
                    if (M != FULL) break;                   // the list is ascending
                }
            }
            if (c > 0) merge_ranked<EPL>(pool, buf, c, A.k, lane);
            __syncwarp();
        }
        __syncthreads();
        if (threadIdx.x == 0) *done = 0u;                   // leave the scratch as it was found
        if (threadIdx.x < G && S.id[threadIdx.x] >= 0) A.bound[S.id[threadIdx.x]] = ~0ull;
    } else if (threadIdx.x < G && S.id[threadIdx.x] >= 0) {
        A.bound[S.id[threadIdx.x]] = ~0ull;
    }
    if (warp < G && S.id[warp] >= 0) exact_output<EPL>(A, S.pool + warp * 32 * EPL, S.id[warp], lane);
    __syncthreads();
}

// One CTA per query, no scratch: each warp streams batches of 16 rows and keeps a list of its own, warp 0 merges
// the lists.  32 warps per SM and no barrier in the loop: the better form for many short slabs (see exact_form).
template <int EPL>
__global__ void __launch_bounds__(EXACT_WARPS * 32)
frog_exact_kernel(const ExactArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int POOL = 32 * EPL;
    const int lane = lane_id();
    const int warp = threadIdx.x >> 5;
    const int q = blockIdx.x;
    float4* qs = reinterpret_cast<float4*>(smem_raw);
    uint64_t* pools = reinterpret_cast<uint64_t*>(smem_raw + (size_t)A.d_pad * 4);
    uint64_t* pool = pools + (size_t)warp * POOL;

    {
        float* qf = reinterpret_cast<float*>(qs);
        const float* src = A.queries + (size_t)q * A.d;
        for (int i = threadIdx.x; i < A.d_pad; i += blockDim.x) qf[i] = i < A.d ? __ldg(src + i) : 0.f;
        for (int i = lane; i < POOL; i += 32) pool[i] = KEY_EMPTY;
    }
    const int32_t lo = __ldg(A.lo + q), hi = __ldg(A.hi + q);
    int l_q, r_q;
    warp_rank_interval(A.sorted_attr, A.n, lo, hi, lane, l_q, r_q);
    const int w = (lo > hi) ? 0 : (r_q - l_q + 1);
    __syncthreads();

    for (int b0 = warp * 16; b0 < w; b0 += EXACT_WARPS * 16) {
        const int cnt = min(16, w - b0);
        const uint32_t rank = (uint32_t)(l_q + b0 + (lane & 15));
        float d2 = batch_dist2<4>(A.vectors, A.d_pad, qs, rank, cnt, lane);
        uint64_t key = KEY_EMPTY;
        if (lane < cnt) key = make_key(d2, (uint32_t)__ldg(A.rank2id + rank), 1u);   // keyed by object id
        // (merge_batch itself rejects candidates not better than the current k-th best)
        merge_batch<EPL>(pool, key, A.k, lane);
    }
    __syncthreads();
    if (warp == 0) {
        for (int ow = 1; ow < EXACT_WARPS; ++ow) {
            const uint64_t* other = pools + (size_t)ow * POOL;
            for (int j0 = 0; j0 < A.k; j0 += 32) {
                uint64_t key = (j0 + lane < A.k) ? other[j0 + lane] : KEY_EMPTY;
                merge_batch<EPL>(pool, key, A.k, lane);
            }
        }
        __syncwarp();
        for (int j = lane; j < A.k; j += 32) {
            uint64_t key = pool[j];
            int32_t oid = -1;
            float dist = __int_as_float(0x7F800000);
            if (key != KEY_EMPTY) {
                oid = (int32_t)key_rank(key);
                dist = __fsqrt_rn(key_dist2(key));
            }
            A.out_ids[(size_t)q * A.k + j] = oid;
            A.out_dists[(size_t)q * A.k + j] = dist;
        }
    }
}

// what the two kernels that do not group keep behind the scan's shared memory
struct FewExtra {
    int2 slab[EXACT_PLAN_MIN];
};
struct SplitExtra {
    unsigned long long rows;
    int first[EXACT_SPLIT_MAX + 1];                          // first piece of each query
    int warp_sum[EXACT_WARPS];
};

// Fewer than EXACT_PLAN_MIN queries: all rows cut into equal pieces, at most one per CTA.
template <int EPL>
__global__ void __launch_bounds__(EXACT_WARPS * 32, 2)
frog_exact_few_kernel(const ExactArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int2* const slab = reinterpret_cast<FewExtra*>(smem_raw + ExactSmem<EPL, 1>::bytes(A.d_pad))->slab;
    const ExactSmem<EPL, 1> S(smem_raw);
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    for (int q = warp; q < A.nq; q += EXACT_WARPS) {
        const int32_t lo = __ldg(A.lo + q), hi = __ldg(A.hi + q);
        int l_q, r_q;
        warp_rank_interval(A.sorted_attr, A.n, lo, hi, lane, l_q, r_q);
        if (lane == 0) slab[q] = make_int2(l_q, max(0, lo > hi ? 0 : r_q - l_q + 1));
    }
    __syncthreads();
    long long rows = 0;
    for (int q = 0; q < A.nq; ++q) rows += slab[q].y;
    // the pieces of a query but its last are full, so nq extra ones at most
    const int share = max((int)gridDim.x - A.nq, 1);
    int size = (int)max((rows + share - 1) / share, (long long)A.min_rows);
    size = (size + EXACT_STEP - 1) / EXACT_STEP * EXACT_STEP;
    int first = 0;
    for (int q = 0; q < A.nq; ++q) {
        const int pieces = max(1, (int)(((long long)slab[q].y + size - 1) / size));
        const int p = (int)blockIdx.x - first;
        if (p >= 0 && p < pieces) {
            if (threadIdx.x == 0) {
                S.l[0] = slab[q].x;
                S.r[0] = slab[q].x + slab[q].y - 1;
                S.id[0] = q;
            }
            const int row0 = slab[q].x + p * size, row1 = min(row0 + size, slab[q].x + slab[q].y);
            __syncthreads();
            exact_piece<EPL, 1>(A, S, row0, row1, (int)blockIdx.x, first, pieces, A.done + q);
            return;
        }
        first += pieces;
    }
}

// Up to EXACT_SPLIT_MAX queries: all rows cut into pieces of equal size, about two per CTA, which evens out their
// ends.  Every CTA works out the cut for itself from the slabs that the planning kernel found.
template <int EPL>
__global__ void __launch_bounds__(EXACT_WARPS * 32, 2)
frog_exact_split_kernel(const ExactArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitExtra& X = *reinterpret_cast<SplitExtra*>(smem_raw + ExactSmem<EPL, 1>::bytes(A.d_pad));
    unsigned long long& rows = X.rows;
    int *const first = X.first, *const warp_sum = X.warp_sum;
    const ExactSmem<EPL, 1> S(smem_raw);
    const int lane = lane_id(), warp = threadIdx.x >> 5, t = threadIdx.x;
    if (t == 0) rows = 0;
    __syncthreads();
    auto slab_of = [&](int q) {                              // first rank, rows
        const int2 lr = A.ranges[q];
        return make_int2(lr.x, max(0, lr.y - lr.x + 1));
    };
    unsigned long long mine = 0;
    for (int q = t; q < A.nq; q += EXACT_WARPS * 32) mine += (unsigned long long)slab_of(q).y;
    if (mine) atomicAdd(&rows, mine);
    __syncthreads();
    const long long share = 2 * (long long)gridDim.x;
    long long size = max(((long long)rows + share - 1) / share, (long long)A.min_rows);
    size = (size + EXACT_STEP - 1) / EXACT_STEP * EXACT_STEP;
    int before = 0;
    for (int q0 = 0; q0 < A.nq; q0 += EXACT_WARPS * 32) {
        const int q = q0 + t;
        const int np = q < A.nq ? max(1, (int)((slab_of(q).y + size - 1) / size)) : 0;
        int x = np;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        int add = before;
        for (int w = 0; w < EXACT_WARPS; ++w) {
            if (w < warp) add += warp_sum[w];
            before += warp_sum[w];
        }
        if (q < A.nq) first[q] = add + x - np;
        __syncthreads();
    }
    if (t == 0) first[A.nq] = before;
    __syncthreads();
    for (int piece = blockIdx.x; piece < first[A.nq]; piece += gridDim.x) {
        int q = 0, end = A.nq;                               // the last query whose first piece is not beyond this one
        while (end - q > 1) {
            const int mid = (q + end) >> 1;
            if (first[mid] <= piece) q = mid; else end = mid;
        }
        const int2 sl = slab_of(q);
        if (t == 0) {
            S.l[0] = sl.x;
            S.r[0] = sl.x + sl.y - 1;
            S.id[0] = q;
        }
        const int p = piece - first[q];
        const int row0 = sl.x + (int)(p * size), row1 = (int)min((long long)row0 + size, (long long)sl.x + sl.y);
        __syncthreads();
        exact_piece<EPL, 1>(A, S, row0, row1, piece, first[q], first[q + 1] - first[q], A.done + q);
        __syncthreads();
    }
}

// The pieces that frog_exact_cut_kernel listed, for groups of eight queries.
template <int EPL>
__global__ void __launch_bounds__(EXACT_WARPS * 32, 2)
frog_exact_group_kernel(const ExactArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ExactSmem<EPL, EXACT_GROUP> S(smem_raw);
    for (;;) {
        if (threadIdx.x == 0) S.misc[1] = (int)atomicAdd(A.counters + 1, 1u);
        __syncthreads();
        const int piece = S.misc[1];
        if (piece >= (int)__ldcg(A.counters)) break;
        const int4 job = A.jobs[piece];
        const int2 gp = A.groups[job.x];
        if (threadIdx.x < EXACT_GROUP) {
            const int i = job.x * EXACT_GROUP + threadIdx.x;
            const int q = i < A.nq ? A.order[i] : -1;
            const int2 lr = q >= 0 ? A.ranges[q] : make_int2(1, 0);
            S.id[threadIdx.x] = q;
            S.l[threadIdx.x] = lr.x;
            S.r[threadIdx.x] = lr.y;
        }
        __syncthreads();
        exact_piece<EPL, EXACT_GROUP>(A, S, job.y, job.z, piece, gp.x, gp.y, A.done + job.x);
        __syncthreads();
    }
}

// bin of a query: widest first, then by position, so that the queries of a group share rows
__device__ __forceinline__ int exact_bin(const int2& lr, int n) {
    const int w = lr.y - lr.x + 1;
    return (w <= 0 ? 32 : __clz(w)) * 32 + (w <= 0 ? 0 : (int)((long long)lr.x * 32 / n));
}

// slabs of the queries and the histogram of their bins (one warp per query)
__global__ void __launch_bounds__(256)
frog_exact_plan_kernel(const ExactArgs A) {
    const unsigned int q = blockIdx.x * 8u + (threadIdx.x >> 5);
    const int lane = lane_id();
    if (q >= (unsigned int)A.nq) return;
    const int32_t lo = __ldg(A.lo + q), hi = __ldg(A.hi + q);
    int l_q, r_q;
    warp_rank_interval(A.sorted_attr, A.n, lo, hi, lane, l_q, r_q);
    if (lane == 0) {
        const int2 lr = lo > hi || r_q < l_q ? make_int2(1, 0) : make_int2(l_q, r_q);
        A.ranges[q] = lr;
        if (A.jobs) atomicAdd(A.counters + 2 + exact_bin(lr, A.n), 1u);
    }
}

// rows that a group's slabs cover (l ascending), and the row where `skip` of them lie below
__device__ __forceinline__ int exact_covered(const int2* s, int cnt) {
    int total = 0, end = 0;
    for (int i = 0; i < cnt; ++i) {
        if (s[i].y < s[i].x) continue;
        total += max(0, s[i].y + 1 - max(s[i].x, end));
        end = max(end, s[i].y + 1);
    }
    return total;
}
__device__ __forceinline__ int exact_cut(const int2* s, int cnt, int skip) {
    int end = 0;
    for (int i = 0; i < cnt; ++i) {
        if (s[i].y < s[i].x) continue;
        const int from = max(s[i].x, end), len = max(0, s[i].y + 1 - from);
        if (skip < len) return from + skip;
        skip -= len;
        end = max(end, s[i].y + 1);
    }
    return end;
}

// order of the queries, and the groups' rows cut into pieces of equal size (one CTA)
__global__ void __launch_bounds__(1024)
frog_exact_cut_kernel(const ExactArgs A) {
    __shared__ unsigned int start[2048];
    __shared__ unsigned int warp_sum[32];
    __shared__ unsigned long long rows;
    __shared__ unsigned int pieces;
    const int t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    if (t == 0) { rows = 0; pieces = 0; }
    // exclusive scan of the bins, two per thread
    const unsigned int a = 2 * t < EXACT_BINS ? A.counters[2 + 2 * t] : 0u;
    const unsigned int b = 2 * t + 1 < EXACT_BINS ? A.counters[3 + 2 * t] : 0u;
    unsigned int x = a + b;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned int s = warp_sum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int y = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s += y;
        }
        warp_sum[lane] = s;
    }
    __syncthreads();
    const unsigned int before = (warp ? warp_sum[warp - 1] : 0u) + x - a - b;
    start[2 * t] = before;
    start[2 * t + 1] = before + a;
    if (2 * t < EXACT_BINS) A.counters[2 + 2 * t] = 0u;          // leave the bins empty
    if (2 * t + 1 < EXACT_BINS) A.counters[3 + 2 * t] = 0u;
    __syncthreads();
    for (int q = t; q < A.nq; q += 1024) A.order[atomicAdd(&start[exact_bin(A.ranges[q], A.n)], 1u)] = q;
    __syncthreads();
    const int groups = (A.nq + EXACT_GROUP - 1) / EXACT_GROUP;
    auto slabs = [&](int g, int2* s) -> int {
        const int cnt = min(EXACT_GROUP, A.nq - g * EXACT_GROUP);
        for (int i = 0; i < cnt; ++i) {
            const int2 lr = A.ranges[A.order[g * EXACT_GROUP + i]];
            int j = i;
            for (; j > 0 && s[j - 1].x > lr.x; --j) s[j] = s[j - 1];
            s[j] = lr;
        }
        return cnt;
    };
    for (int g = t; g < groups; g += 1024) {
        int2 s[EXACT_GROUP];
        const int c = exact_covered(s, slabs(g, s));
        A.groups[g] = make_int2(c, 0);
        atomicAdd(&rows, (unsigned long long)c);
    }
    __syncthreads();
    // a group of several pieces has at most twice its rows' share of them, so max_pieces is never exceeded
    const long long want = ((long long)rows * 2 + A.max_pieces - 1) / A.max_pieces;
    long long size = want > A.min_rows ? want : A.min_rows;
    size = (size + 2 * EXACT_STEP - 1) / (2 * EXACT_STEP) * (2 * EXACT_STEP);
    // groups of several pieces first: their piece numbers address the partial lists
    for (int pass = 0; pass < 2; ++pass) {
        for (int g = t; g < groups; g += 1024) {
            const int2 have = A.groups[g];
            const int c = have.x, np = max(1, (int)(((long long)c + size - 1) / size));
            if ((np > 1) != (pass == 0) || (pass == 1 && have.y != 0)) continue;
            int2 s[EXACT_GROUP];
            const int cnt = slabs(g, s);
            const unsigned int first = atomicAdd(&pieces, (unsigned int)np);
            int from = exact_cut(s, cnt, 0);
            for (int p = 0; p < np; ++p) {
                const int to = p + 1 < np ? exact_cut(s, cnt, (int)((long long)(p + 1) * size)) : exact_cut(s, cnt, c);
                A.jobs[first + p] = make_int4(g, from, to, 0);
                from = to;
            }
            A.groups[g] = make_int2((int)first, np);
        }
        __syncthreads();
    }
    if (t == 0) {
        A.counters[0] = pieces;
        A.counters[1] = 0u;
    }
}

typedef void (*exact_fn)(const ExactArgs);

template <template <int> class K>
exact_fn exact_pick(int k) {
    return k <= 32 ? K<1>::fn() : k <= 64 ? K<2>::fn() : k <= 128 ? K<4>::fn() : k <= 256 ? K<8>::fn() : K<16>::fn();
}
template <int EPL> struct OnePerQuery { static exact_fn fn() { return frog_exact_kernel<EPL>; } };
template <int EPL> struct Few { static exact_fn fn() { return frog_exact_few_kernel<EPL>; } };
template <int EPL> struct Split { static exact_fn fn() { return frog_exact_split_kernel<EPL>; } };
template <int EPL> struct Grouped { static exact_fn fn() { return frog_exact_group_kernel<EPL>; } };

template <int G>
size_t exact_smem(int k, int d_pad) {
    return k <= 32 ? ExactSmem<1, G>::bytes(d_pad) : k <= 64 ? ExactSmem<2, G>::bytes(d_pad)
         : k <= 128 ? ExactSmem<4, G>::bytes(d_pad) : k <= 256 ? ExactSmem<8, G>::bytes(d_pad) : ExactSmem<16, G>::bytes(d_pad);
}

// Which form scans.  Two things decide that the host can know, as the slabs' widths are on the device: whether a CTA
// per query leaves the GPU idle (few queries), and whether the whole index is so short that cutting it costs more
// than it saves.  us, one CTA per query / split by query / grouped, k = 10, slabs of all rows | log-uniform down to 1/16:
//                     40 queries                  100                          200                          1,000
//   1,000 x 96     48/53/84 | 46/52/99        48/77/85 | 46/58/97         49/104/90 | 46/80/95         89/-/100 | 65/-/99
//   2,000 x 96     63/78/86 | 60/56/96        62/90/87 | 59/77/99         64/123/89 | 60/95/101       120/-/139 | 87/-/116
//   5,000 x 96     98/73/90 | 95/56/99        99/117/92 | 94/83/101      103/174/95 | 93/116/105      218/-/271 | 151/-/160
//   20,000 x 96   276/128/111 | 248/96/123   278/220/155 | 269/140/129   293/371/235 | 272/192/164    679/-/678 | 421/-/401
//   2,000 x 768   137/90/189 | 130/63/176    138/117/190 | 131/93/182    151/175/192 | 140/126/189    359/-/343 | 215/-/201
//   100,000 x 128      - | 1234/172/280           - | 1284/272/336            - | 1282/446/472             - | 2015/-/1182
// Long result lists favour pieces (k = 100, second column: 2,000 x 96, 1,000 queries 207/-/121, 5,000 x 96, 100
// 162/134/122).  Over 3,400 combinations (300 to 1,000,000 objects, 32 to 2,000 dimensions, 1-2,000 queries, k = 10 to
// 512, three mixes of widths) the rule takes 0.51 of the time of one CTA per query in the mean and is slower by more
// than a tenth in 1 %; the best form of each would take 0.48.
// More queries than a line that depends on rows and k, on 4,000 rows or more, are filtered (frog_exact_filter.cu): six
// launches and two passes of products, which take 50-110 us in any case and hardly grow with the queries.  us, the
// form of the lines above / filtered, log-uniform widths down to 2^-10 | all rows:
//                      40 queries, k = 10      100, k = 10           400, k = 10            2,000, k = 100
//   3,000 x 96      34/55 | 58/48         50/55 | 54/48          54/60 | 66/53        120/123 | 369/136
//   5,000 x 128     33/56 | 51/52         74/58 | 84/51          82/62 | 104/60       149/118 | 488/157
//   20,000 x 50     51/54 | 100/50        68/54 | 188/54         240/59 | 282/88      370/145 | 1,137/288
//   5,000 x 768     43/110 | 76/100       69/112 | 165/104       179/123 | 321/135    321/248 | 1,303/417
//   20,000 x 768    72/121 | 212/117      120/120 | 464/137      283/128 | 1,071/294  953/411 | 4,521/1,451
//   100,000 x 128   90/100 | 253/105      149/107 | 555/129      411/128 | 1,190/259  1,163/294 | 5,075/873
//   400,000 x 96    155/207 | 1,200/251   352/246 | 2,926/302    1,032/327 | 3,497/663  3,802/808 | 16,761/2,978
// Slabs of fewer than 10 k rows are not filtered.  Where no slab is wider, all that the form does is to scan each with one CTA,
// which up to EXACT_SPLIT_MAX queries still beats the form that splits them and after that loses to the grouped one; us, the
// same columns:
//                          100, k = 512          200                  400                  2,000
//   5,119 x 32           189/187 | 362/194    166/188 | 198/195    172/190 | 266/202    232/270 | 716/740
//   5,119 x 128          186/203 | 375/207    284/205 | 369/215    182/205 | 281/232    245/293 | 794/861
//   4,096 x 200          148/210 | 379/218    281/215 | 393/231    186/217 | 270/252    236/313 | 811/957
//   5,119 x 768          208/400 | 422/410    299/406 | 525/456    279/414 | 471/520    410/590 | 1,663/2,024
//   8,000 x 128          322/222 | 406/101         -               227/236 | 385/114    344/342 | 1,055/366
//   100,000 x 128            - | 1,051/167        -                    - | 1,890/325    - | 6,428/1,255
//   400,000 x 96             - | 3,577/383        -                    - | 4,872/750    - | 19,502/3,306
//   64,000 x 128         582/249 | 839/140         -               560/269 | 1,388/263  1,264/533 | 4,506/1,087
enum class ExactForm { OnePerQuery, Few, Split, Grouped, Filter };
int filter_line(size_t n, size_t row_bytes, int k) {
    if (n < 4000 || row_bytes > 16384) return 0x7FFFFFFF;
    if (row_bytes > 1024) return n >= 16000 ? 128 : 400;
    return n < 16000 ? 100 : k <= 32 ? 80 : n < 64000 ? 40 : EXACT_PLAN_MIN;
}
ExactForm exact_form(size_t n, size_t row_bytes, int nq, int k, bool filter) {
    const size_t bytes = n * row_bytes;
    if (filter && nq >= filter_line(n, row_bytes, k) && (n >= (size_t)10 * k || nq <= EXACT_SPLIT_MAX)) return ExactForm::Filter;
    if (nq < EXACT_PLAN_MIN) return k <= 32 && bytes <= 500000 ? ExactForm::OnePerQuery : ExactForm::Few;
    const double work = (double)n * (double)(row_bytes + 384) * (k > 128 ? 3.0 : k > 64 ? 1.4 : 1.0);
    if (nq <= EXACT_SPLIT_MAX && nq * (n < 8000 ? 45e3 : 100e3) <= work) return ExactForm::Split;
    if (k > 128) return ExactForm::Grouped;
    if (n < 3000) return k > 32 && nq >= (k > 64 ? 600 : 1400) ? ExactForm::Grouped : ExactForm::OnePerQuery;
    return k > 32 || bytes > 4500000 || (n >= 8000 && nq <= 300) ? ExactForm::Grouped : ExactForm::OnePerQuery;
}

// A set for a scan on stream s: the one it used last, an idle one, a new one, or null when all are busy with other
// streams' scans (the caller does without: a wait for another stream is not made here).  Called with exact_mu held.
FrogExactSet* exact_set(frog_index* ix, cudaStream_t s) {
    unsigned long long id = 0;
    if (cudaStreamGetId(s, &id) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    for (int i = 0; i < ix->n_exact; ++i)
        if (ix->exact[i].used && ix->exact[i].stream_id == id) return &ix->exact[i];
    for (int i = 0; i < ix->n_exact; ++i) {
        FrogExactSet& set = ix->exact[i];
        if (!set.used || cudaEventQuery(set.done) == cudaSuccess) return &set;
        cudaGetLastError();
    }
    if (ix->n_exact == FROG_EXACT_SETS) return nullptr;
    FrogExactSet& set = ix->exact[ix->n_exact];
    if (cudaEventCreateWithFlags(&set.done, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    ++ix->n_exact;
    return &set;
}

// How a call's rows are cut, and what that takes of scratch.  A piece holds at least `min_rows` rows of its query or
// group, or all of them, so that small indexes and small batches need little; only groups (queries, where they are not
// grouped) of several pieces have partial lists.
struct ExactCut {
    size_t groups;             // groups of queries, or queries
    size_t pieces;             // with partial lists, at most
    size_t lists;              // their keys
    int max_pieces, min_rows;
};
ExactCut exact_cut_of(size_t n, size_t nq, int k, int grid, bool few) {
    ExactCut c;
    c.min_rows = few ? 256 : 512;
    c.groups = few ? nq : (nq + EXACT_GROUP - 1) / EXACT_GROUP;
    // enough pieces to even out their ends; fewer for long result lists, whose partial lists they multiply
    const size_t most = few ? 2 * (size_t)grid + nq : (size_t)grid * (k <= 128 ? 16 : 8);
    c.max_pieces = (int)most;
    c.pieces = std::min(most, c.groups * ((n + c.min_rows - 1) / c.min_rows));
    c.lists = c.pieces * (few ? 1 : EXACT_GROUP) * k;
    return c;
}

// Scratch of one call.  At rest the bins, `done` and `bound` are as exact_scratch sets them: the kernels see to it.
struct ExactScratch {
    char* bound;               // u64 per query
    char* counters;            // EXACT_BINS + 2
    char* done;                // int per group
    char* ranges;              // int2 per query
    char* order;               // int per query
    char* groups;              // int2 per group
    char* jobs;                // int4 per piece
    char* part;                // keys of the pieces' lists
};
size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
size_t exact_rest_bytes(size_t queries) { return up256(queries * 8) + up256((EXACT_BINS + 2) * 4) + up256(queries * 4); }
size_t exact_bytes(size_t nq, const ExactCut& c, bool few) {
    const size_t grouping = few ? 0 : up256(nq * 4) + up256(c.groups * 8) + up256((c.pieces + c.groups) * 16);
    return up256(nq * 8) + grouping + up256(c.lists * 8);
}
bool exact_small(const frog_index* ix) { return (size_t)ix->info.n * ix->info.d_pad * 4 <= EXACT_GROW_BYTES; }
// make sure the set has `bytes` beside what `nq` queries keep between calls; `refused`: this call has been told to do without
bool exact_room(frog_index* ix, FrogExactSet* set, size_t nq, size_t bytes, bool* refused) {
    if (!set->mem || nq > set->queries || bytes > set->bytes) {
        // Growing takes 0.5-3 ms.  A first scan of 2,000 queries, k = 100, without scratch / with growth: 20,000 x 96 (7.7 MB)
        // 1,370/1,600 us, 201 queries 490/920; 100,000 x 128 (51 MB) 2,740/1,950.  So on small indexes a scan that would
        // need more does without, whichever forms it asks for, and only a second one grows.
        if (*refused || (!ix->exact_asked && exact_small(ix))) {
            ix->exact_asked = *refused = true;
            return false;
        }
        const size_t new_queries = std::max(nq, set->queries), new_bytes = std::max(bytes, set->bytes);
        char* mem = nullptr;
        // (the set's last scan may still be running: on this stream, as a set is taken idle from another)
        if (cudaMalloc(&mem, exact_rest_bytes(new_queries) + new_bytes) != cudaSuccess ||
            (set->used && cudaEventSynchronize(set->done) != cudaSuccess)) {
            cudaGetLastError();
            cudaFree(mem);
            return false;                                  // the set stays as it is
        }
        cudaFree(set->mem);
        set->mem = mem;
        set->queries = new_queries;
        set->bytes = new_bytes;
        set->clean = false;
    }
    return true;
}
bool exact_scratch(frog_index* ix, FrogExactSet* set, cudaStream_t s, size_t nq, const ExactCut& c, bool few,
                   bool* refused, ExactScratch* out) {
    if (!exact_room(ix, set, nq, exact_bytes(nq, c, few), refused)) return false;
    out->bound = set->mem;
    out->counters = out->bound + up256(set->queries * 8);
    out->done = out->counters + up256((EXACT_BINS + 2) * 4);
    out->ranges = set->mem + exact_rest_bytes(set->queries);
    out->order = out->ranges + up256(nq * 8);
    out->groups = out->order + (few ? 0 : up256(nq * 4));
    out->jobs = out->groups + (few ? 0 : up256(c.groups * 8));
    out->part = out->jobs + (few ? 0 : up256((c.pieces + c.groups) * 16));
    if (!set->clean) {
        if (cudaMemsetAsync(out->bound, 0xFF, out->counters - out->bound, s) != cudaSuccess ||
            cudaMemsetAsync(out->counters, 0, out->ranges - out->counters, s) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

}  // namespace

extern "C" int frog_exact_search(const frog_index_t* index, const float* queries, const int32_t* lo,
                                 const int32_t* hi, int nq, int k, int32_t* out_ids, float* out_dists,
                                 void* stream) {
    if (!index || nq < 0 || k < 1 || k > FROG_MAX_BEAM_WIDTH) return FROG_ERR_INVALID_ARG;
    if (nq == 0) return FROG_OK;
    if (!queries || !lo || !hi || !out_ids || !out_dists) return FROG_ERR_INVALID_ARG;
    FROG_CUDA_TRY(cudaSetDevice(index->info.device));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ExactArgs A{};
    A.sorted_attr = index->d_sorted_attr;
    A.rank2id = index->d_rank2id;
    A.vectors = index->d_vectors;
    A.n = (int)index->info.n;
    A.d = index->info.d;
    A.d_pad = index->info.d_pad;
    A.queries = queries;
    A.lo = lo;
    A.hi = hi;
    A.nq = nq;
    A.k = k;
    A.out_ids = out_ids;
    A.out_dists = out_dists;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    FROG_CUDA_TRY(cudaStreamIsCapturing(s, &capture));
    ExactForm form = exact_form((size_t)index->info.n, (size_t)A.d_pad * 4, nq, k, capture == cudaStreamCaptureStatusNone);
    bool refused = false;
    if (form == ExactForm::Filter) {
        // Scratch of the sets' part that has no state at rest, for slabs of any width, as these are on the device, up to the
        // larger of 64 MB and half of the index.  A batch for which that may not be enough goes in rounds, where these are
        // few or each is large (one that has nothing to do takes 15-25 us, and the grouped form 27 us for 1,000 queries of
        // 50 rows); where scratch cannot be had, the other forms.  Batches over all rows, us, by the forms below / filtered
        // with one CTA for a query that there was no room for / in rounds: 2,000 queries, k = 10, on 100,000 x 128
        // 4,990 / 3,980 / 803, 400,000 x 96 17,200 / 15,300 / 2,650; 100 on 4,000,000 x 32 23,100 / 55,900 / 1,760.
        frog_index* mix = const_cast<frog_index*>(index);
        std::lock_guard<std::mutex> lock(mix->exact_mu);
        const size_t n = (size_t)index->info.n;
        const size_t want = std::min(froghost::filter_bytes(n, (size_t)nq, k, A.d_pad),
                                     std::max((size_t)index->info.device_bytes / 2, (size_t)64 << 20));
        FrogExactSet* set = nullptr;
        froghost::FilterFit fit{};
        {
            const froghost::NoCaptureOfOurs relaxed;
            set = exact_set(mix, s);
            if (set && set->mem) fit = froghost::filter_fit(n, (size_t)nq, set->bytes, k, A.d_pad);
            if (set && set->bytes < want) {
                // (what takes the batch in four rounds will do for the first call of its kind)
                if (fit.queries && fit.parts * fit.rounds <= 4 && !mix->exact_asked) {
                    mix->exact_asked = true;
                    refused = exact_small(mix);
                } else if (exact_room(mix, set, 0, want, &refused)) {
                    fit = froghost::filter_fit(n, (size_t)nq, set->bytes, k, A.d_pad);
                }
            }
        }
        if (fit.queries && fit.per_round >= (size_t)filter_line(n, (size_t)A.d_pad * 4, k) &&
            (fit.parts * fit.rounds <= 4 || (fit.per_round >= 512 && fit.parts <= 64))) {
            froghost::FilterArgs F{};
            F.sorted_attr = A.sorted_attr;
            F.rank2id = A.rank2id;
            F.vectors = A.vectors;
            F.n = A.n;
            F.d = A.d;
            F.d_pad = A.d_pad;
            F.k = k;
            F.rounds = (int)fit.rounds;
            F.step = fit.step;
            for (size_t p = 0; p < fit.parts; ++p) {
                const size_t q0 = (size_t)nq * p / fit.parts, q1 = (size_t)nq * (p + 1) / fit.parts;
                F.queries = queries + q0 * A.d;
                F.lo = lo + q0;
                F.hi = hi + q0;
                F.nq = (int)(q1 - q0);
                F.out_ids = out_ids + q0 * k;
                F.out_dists = out_dists + q0 * k;
                froghost::filter_scratch(set->mem + exact_rest_bytes(set->queries), &F);
                FROG_CUDA_TRY(froghost::filter_launch(F, index->sm_count, s));
            }
            FROG_CUDA_TRY(cudaEventRecord(set->done, s));
            FROG_CUDA_TRY(cudaStreamGetId(s, &set->stream_id));
            set->used = true;
            return FROG_OK;
        }
        form = exact_form((size_t)index->info.n, (size_t)A.d_pad * 4, nq, k, false);
    }
    const bool few = form != ExactForm::Grouped;
    const size_t smem = !few ? exact_smem<EXACT_GROUP>(k, A.d_pad)
                             : exact_smem<1>(k, A.d_pad) + (form == ExactForm::Few ? sizeof(FewExtra) : sizeof(SplitExtra));
    // (the planning kernels count queries in ints with some room)
    if (capture == cudaStreamCaptureStatusNone && form != ExactForm::OnePerQuery && smem <= froghost::MAX_SMEM &&
        nq <= 1 << 30) {
        const exact_fn fn = form == ExactForm::Few ? exact_pick<Few>(k) : few ? exact_pick<Split>(k) : exact_pick<Grouped>(k);
        FROG_CUDA_TRY(froghost::allow_smem(fn));
        int per_sm = 0;
        FROG_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)fn, EXACT_WARPS * 32, smem));
        const int grid = std::max(per_sm, 1) * index->sm_count;
        const ExactCut cut = exact_cut_of((size_t)index->info.n, (size_t)nq, k, grid, few);
        frog_index* mix = const_cast<frog_index*>(index);      // the scratch sets are the index's only mutable part
        std::lock_guard<std::mutex> lock(mix->exact_mu);
        FrogExactSet* set = nullptr;
        ExactScratch X;
        {
            const froghost::NoCaptureOfOurs relaxed;
            set = exact_set(mix, s);
            if (set && !exact_scratch(mix, set, s, (size_t)nq, cut, few, &refused, &X)) set = nullptr;
        }
        if (set) {
            A.ranges = reinterpret_cast<int2*>(X.ranges);
            A.order = reinterpret_cast<int32_t*>(X.order);
            A.jobs = few ? nullptr : reinterpret_cast<int4*>(X.jobs);        // null: no histogram
            A.groups = reinterpret_cast<int2*>(X.groups);
            A.counters = reinterpret_cast<unsigned int*>(X.counters);
            A.done = reinterpret_cast<unsigned int*>(X.done);
            A.bound = reinterpret_cast<unsigned long long*>(X.bound);
            A.part = reinterpret_cast<uint64_t*>(X.part);
            A.max_pieces = cut.max_pieces;
            A.min_rows = cut.min_rows;
            set->clean = false;                            // until the launches are under way
            if (form != ExactForm::Few) frog_exact_plan_kernel<<<(nq - 1) / 8 + 1, 256, 0, s>>>(A);
            if (!few) frog_exact_cut_kernel<<<1, 1024, 0, s>>>(A);
            fn<<<grid, EXACT_WARPS * 32, smem, s>>>(A);
            FROG_CUDA_TRY(cudaGetLastError());
            set->clean = true;
            FROG_CUDA_TRY(cudaEventRecord(set->done, s));
            FROG_CUDA_TRY(cudaStreamGetId(s, &set->stream_id));
            set->used = true;
            return FROG_OK;
        }
    }
    const int pool_slots = k <= 32 ? 32 : k <= 64 ? 64 : k <= 128 ? 128 : k <= 256 ? 256 : 512;
    const size_t smem1 = (size_t)A.d_pad * 4 + (size_t)EXACT_WARPS * pool_slots * 8;
    const exact_fn one = exact_pick<OnePerQuery>(k);
    FROG_CUDA_TRY(froghost::allow_smem(one));
    one<<<nq, EXACT_WARPS * 32, smem1, s>>>(A);
    FROG_CUDA_TRY(cudaGetLastError());
    return FROG_OK;
}

// Scratch for one stream's scans of up to 2,048 queries with k up to 128 (39 MB at most), but no more than half of the
// index, so that a first scan has nothing to allocate as a rule.  Not having it is no error.
void froghost::reserve_exact(frog_index* ix) {
    const ExactCut cut = exact_cut_of((size_t)ix->info.n, 2048, 128, 2 * ix->sm_count, false);
    const size_t bytes = std::min(exact_bytes(2048, cut, false), (size_t)ix->info.device_bytes / 2);
    FrogExactSet& set = ix->exact[0];
    if (cudaEventCreateWithFlags(&set.done, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    ix->n_exact = 1;
    if (cudaMalloc(&set.mem, exact_rest_bytes(2048) + bytes) != cudaSuccess) {
        cudaGetLastError();
        set.mem = nullptr;
        return;
    }
    set.queries = 2048;
    set.bytes = bytes;
}
