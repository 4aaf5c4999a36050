// The exact scan of many queries: tensor cores rule rows out, what is left is compared in fp32.
//
// A row's distance to a query enters the answer only if it is among the k smallest, and of the rows of a slab all but a
// few can be told apart from those with a rough distance.  |x|^2 + |q|^2 - 2 x.q with x.q from tf32 matrix
// instructions is such a distance, for 128 rows and 128 queries at a time, and its error is bounded (row_error):
//   * bounds: for every query and every 8 (wide slabs: 32) rows the smallest upper bound of a distance.  The k-th
//     smallest of these belongs to k different rows, so no answer lies beyond it;
//   * masks: the same products again, one bit per row and query: the lower bound does not exceed that;
//   * the rows whose bit is set, a little more than k, are compared as frog_exact.cu compares all: fp32, in the fixed
//     order.  Ids and distances are therefore those of a scan of all rows, bit for bit.
// Products are computed twice, the second time only for tiles that a bound of the first says may hold an answer, because
// storing them would take 4 bytes per row and query.  2,000 queries, k = 100, on 100,000 x 128, log-uniform widths:
// 1,290 us by groups of eight in fp32, 294 filtered (k = 10: 222); one launch at a time under the profiler 10 planning, 116
// first pass, 17 bounds, 89 second pass, 81 comparison.  The passes are bound by issue and the latency of fragment loads (24
// for 16 matrix instructions) and of their epilogues, the matrix unit is active for a quarter of the time: tiles are as deep
// as a vector, 32 to 768.  Hence mma.sync, whose accumulators are where the epilogue needs them.
#include <algorithm>

#include "frog_device.cuh"
#include "frog_exact_filter.h"
#include "frog_internal.h"

using namespace frogdev;
using froghost::FilterArgs;

namespace {

constexpr int TILE = 128;                // rows, and queries, of a tile of products
constexpr int SEG = 2048;                // queries listed at a time
constexpr int THREADS = 256;             // 4 x 2 warps of 32 rows x 64 queries

// KC: elements of a row per pipeline stage, 64 in all.  Short rows have few stages, so more of them in flight count
// (100,000 x 32: 201 us with two stages of 32, 172 with four of 16), long ones pay for each stage's barrier (20,000 x
// 768: 277 and 299).
template <int KC>
struct FilterSmem {
    static constexpr int KP = KC + 4;    // stride of a row's part: fragment loads without bank conflicts
    static constexpr int STAGES = 64 / KC;
    float a[STAGES][TILE * KP];
    float b[STAGES][TILE * KP];
    int list[SEG];                       // queries whose slab meets the tile
    float row_norm[TILE];
    // of the batch's queries: first rank and how many follow it, blocks of 32 rows (0: no query), values per block
    uint32_t l[TILE], span[TILE], blocks[TILE];
    int per[TILE];
    float norm[TILE], root[TILE], tau[TILE];     // half the squared norm with its part of the bound, norm, half the bound of the answers
    uint32_t off[TILE];
    int count;
};

__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t y;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// 16 bytes to shared memory, zeros unless `on`
__device__ __forceinline__ void copy16(void* dst, const void* src, bool on) {
    const int bytes = on ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}

// Values of a query per 32 rows in the first pass: one where its slab is so wide that they are still many more than k
__device__ __forceinline__ int values_per_block(int w, int k) { return w >= 128 * k ? 1 : 4; }
// Narrower slabs have hardly k values to choose from: their rows are all compared
__device__ __forceinline__ bool filtered(int w, int k) { return w >= max(10 * k, 128); }

// slabs of the queries, their norms, and the queries themselves rounded to tf32 (one warp per query)
__global__ void __launch_bounds__(256)
filter_plan_kernel(const FilterArgs A) {
    const unsigned int q = blockIdx.x * 8u + (threadIdx.x >> 5);
    const int lane = lane_id();
    if (q >= (unsigned int)A.nq) return;
    const int32_t lo = __ldg(A.lo + q), hi = __ldg(A.hi + q);
    int l_q, r_q;
    warp_rank_interval(A.sorted_attr, A.n, lo, hi, lane, l_q, r_q);
    float s = 0.f;
    for (int i = lane; i < A.d_pad; i += 32) {
        const float x = i < A.d ? __ldg(A.queries + (size_t)q * A.d + i) : 0.f;
        s = fmaf(x, x, s);
        A.rounded[(size_t)q * A.d_pad + i] = __uint_as_float(to_tf32(x));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    if (lane == 0) {
        A.slab[q] = lo > hi || r_q < l_q ? make_int2(1, 0) : make_int2(l_q, r_q);
        A.norm[q] = s;
    }
}

// Where each query's values lie (one CTA); BOT: the query is not filtered.  The store holds the values of some queries at a
// time, as the widths, which are on the device, allow: a round takes those whose values, laid end to end, begin in its
// share of A.step.
__global__ void __launch_bounds__(1024)
filter_offsets_kernel(const FilterArgs A) {
    __shared__ unsigned long long warp_sum[32];
    __shared__ unsigned long long base;
    const int t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    if (t == 0) base = 0;
    for (int i = t; i * TILE < A.n; i += 1024) A.tile_norm[i] = 0u;
    __syncthreads();
    for (int q0 = 0; q0 < A.nq; q0 += 1024) {
        const int q = q0 + t;
        unsigned long long need = 0;                             // 32-bit words: the values, then the masks
        if (q < A.nq) {
            const int2 s = A.slab[q];
            const int w = s.y - s.x + 1;
            if (filtered(w, A.k))
                need = (unsigned long long)((s.y >> 5) - (s.x >> 5) + 1) * (values_per_block(w, A.k) + 1);
        }
        unsigned long long x = need;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        unsigned long long at = base + x - need;
        for (int w = 0; w < warp; ++w) at += warp_sum[w];
        if (q < A.nq) {
            const unsigned long long round = at / A.step, next = q + 1 < A.nq ? (at + need) / A.step : (unsigned long long)A.rounds;
            A.off[q] = need != 0 ? (uint32_t)(at - round * A.step) : BOT;
            if (q == 0) A.first[0] = 0;
            for (unsigned long long r = round + 1; r <= next; ++r) A.first[r] = q + 1;
        }
        __syncthreads();
        if (t == 1023) base = at + need;
        __syncthreads();
    }
}

// Bound of the error of a rough distance, and of what separates the fp32 distance of the scan from the true one.
// With u = 2^-11 the rounding of an operand: |x~.q~ - x.q| <= (2u + u^2) |x| |q|; the sums of d products, of the norms
// and of the scan are within d 2^-22 of their magnitude each (twice what rounding to nearest gives); the last two terms
// cover what underflows.  (x and q are the norms, c1 x q + own(x) + own(q) the bound.)  How the sums inside an instruction are
// rounded is not documented; measured against 64 bits (gaussian, positive, byte, decaying, like and mixed operands, 1 to 4,096
// elements, 64,000 products each) they take .09 of their part of c1 at most, and the whole error .99 of c1, where all operands
// are 1 + 2^-11.
// The epilogue computes HALF of a bound, which two finite norms cannot take beyond the range of fp32: it is infinite only
// where x.q is below -2^128, and then so is the distance.  A norm that is not finite makes it not a number, and the
// comparison with it false, which rules nothing out.
struct RowError {
    float c1, c2;
    __device__ __forceinline__ explicit RowError(int d) : c1(0.00197f + d * 0x1p-20f), c2(0x1p-19f + d * 0x1p-21f) {}
    __device__ __forceinline__ float own(float nx, float x) const { return c2 * nx + (1e-30f * x + 1e-34f); }
    __device__ __forceinline__ float operator()(float nx, float x, float nq, float q) const {
        return c1 * x * q + (own(nx, x) + own(nq, q));
    }
};

// PASS 0: bounds, PASS 1: masks.  One CTA per 128 rows and per share of the queries: those whose number is blockIdx.y
// modulo gridDim.y (the order in which a CTA lists its queries is not that of another).
__device__ __forceinline__ int2 round_queries(const FilterArgs& A, int round) {      // first and end
    return A.rounds == 1 ? make_int2(0, A.nq) : make_int2(__ldg(A.first + round), __ldg(A.first + round + 1));
}
template <int PASS, int KC>
__global__ void __launch_bounds__(THREADS, 2)
filter_tile_kernel(const FilterArgs A, int round) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FilterSmem<KC>& S = *reinterpret_cast<FilterSmem<KC>*>(smem_raw);
    constexpr int KP = FilterSmem<KC>::KP, STAGES = FilterSmem<KC>::STAGES;
    const int t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    const int wm = warp >> 1, wn = warp & 1;                     // this warp's rows and queries of the tile
    const int g = lane >> 2, p = lane & 3;                       // fragment coordinates
    const int row0 = blockIdx.x * TILE, row_end = min(row0 + TILE, A.n);
    const int chunks = (A.d_pad + KC - 1) / KC;
    const RowError error(A.d);
    const float tile_norm = PASS == 1 ? __uint_as_float(A.tile_norm[blockIdx.x]) : 0.f, tile_sqrt = __fsqrt_rn(tile_norm);
    bool have_norms = false;

    const int2 queries = round_queries(A, round);
    for (int q0 = queries.x; q0 < queries.y; q0 += SEG) {
        __syncthreads();
        if (t == 0) S.count = 0;
        __syncthreads();
        constexpr int EACH = SEG / THREADS;                      // queries per thread, in flight together
        int2 slabs[EACH];
        uint32_t offs[EACH];
#pragma unroll
        for (int x = 0; x < EACH; ++x) {
            const int q = q0 + x * THREADS + t;
            const bool mine = q < queries.y && q % gridDim.y == blockIdx.y;
            offs[x] = mine ? A.off[q] : BOT;
            slabs[x] = mine ? A.slab[q] : make_int2(1, 0);
        }
#pragma unroll 1
        for (int i = 0; i < EACH; ++i) {
            const int q = q0 + i * THREADS + t;
            int2 s = slabs[0];
            uint32_t off = offs[0];
#pragma unroll
            for (int x = 1; x < EACH; ++x)
                if (x == i) { s = slabs[x]; off = offs[x]; }
            bool hit = false;
            if (off != BOT) {
                hit = s.x < row_end && s.y >= row0;
                if (PASS == 1 && hit) {
                    // The second pass is for tiles with a row that may be an answer: a value of the first is a lower bound
                    // too, less twice the error.  (The infinite ones say nothing.)  The masks of the others are zero.
                    const int w = s.y - s.x + 1, per = values_per_block(w, A.k), all = (s.y >> 5) - (s.x >> 5) + 1;
                    const int from = max((row0 >> 5) - (s.x >> 5), 0), to = min(((row0 + TILE) >> 5) - (s.x >> 5), all);
                    const float nq = A.norm[q], tau = A.tau[q], e = 2.f * error(tile_norm, tile_sqrt, nq, __fsqrt_rn(nq));
                    uint32_t* const v = A.store + off;
                    hit = false;
                    for (int x = from * per; x < to * per; ++x) {
                        const float least = __uint_as_float(v[x]);
                        hit = hit || !(least - e > tau) || !(least < __int_as_float(0x7F800000));
                    }
                    if (!hit)
                        for (int x = from; x < to; ++x) v[all * per + x] = 0u;
                }
            }
            const uint32_t M = __ballot_sync(FULL, hit);
            int at = 0;
            if (lane == 0 && M) at = atomicAdd(&S.count, __popc(M));
            at = __shfl_sync(FULL, at, 0);
            if (hit) S.list[at + __popc(M & ((1u << lane) - 1u))] = q;
        }
        __syncthreads();
        const int count = S.count;
        for (int b0 = 0; b0 < count; b0 += TILE) {
            const int nb = min(TILE, count - b0);
            __syncthreads();                                     // the batch before is done with the tables
            if (t < TILE) {
                const int q = S.list[b0 + min(t, nb - 1)];
                const int2 s = A.slab[q];
                const float n = A.norm[q], root = __fsqrt_rn(n), own = error.own(n, root);
                const uint32_t blocks = (uint32_t)((s.y >> 5) - (s.x >> 5) + 1);
                const int per = values_per_block(s.y - s.x + 1, A.k);
                S.l[t] = t < nb ? (uint32_t)s.x : 0x80000000u;           // no row lies in the slab of none
                S.span[t] = t < nb ? (uint32_t)(s.y - s.x) : 0u;
                S.blocks[t] = t < nb ? blocks : 0u;
                S.per[t] = per;
                S.norm[t] = PASS == 0 ? 0.5f * n + 0.5f * own : 0.5f * n - 0.5f * own;
                S.root[t] = root;
                if (PASS == 1) S.tau[t] = 0.5f * A.tau[q];
                S.off[t] = A.off[q] + (PASS == 1 ? blocks * per : 0u);
            }
            float acc[2][8][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int x = 0; x < 8; ++x)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[m][x][c] = 0.f;
            auto fetch = [&](int chunk) {
                const int st = chunk % STAGES;
#pragma unroll
                for (int x = 0; x < TILE * (KC / 4) / THREADS; ++x) {
                    const int i = x * THREADS + t, r = i / (KC / 4), c = (i % (KC / 4)) * 4;
                    const bool in = chunk * KC + c < A.d_pad;
                    const bool ra = in && row0 + r < A.n, rb = in && r < nb;
                    copy16(&S.a[st][r * KP + c], A.vectors + (ra ? (size_t)(row0 + r) * A.d_pad + chunk * KC + c : 0), ra);
                    copy16(&S.b[st][r * KP + c], A.rounded + (rb ? (size_t)S.list[b0 + r] * A.d_pad + chunk * KC + c : 0), rb);
                }
            };
#pragma unroll
            for (int x = 0; x < STAGES - 1; ++x) {
                if (x < chunks) fetch(x);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            float part = 0.f;                                    // of the norm of row t / 2
            for (int chunk = 0; chunk < chunks; ++chunk) {
                asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
                __syncthreads();
                if (chunk + STAGES - 1 < chunks) fetch(chunk + STAGES - 1);
                asm volatile("cp.async.commit_group;" ::: "memory");
                const float* const a = S.a[chunk % STAGES];
                const float* const b = S.b[chunk % STAGES];
                if (!have_norms) {
                    const float4* const x = reinterpret_cast<const float4*>(a + (t >> 1) * KP + (t & 1) * (KC / 2));
#pragma unroll
                    for (int c = 0; c < KC / 8; ++c) {
                        const float4 v = x[c];
                        part = fmaf(v.x, v.x, part);
                        part = fmaf(v.y, v.y, part);
                        part = fmaf(v.z, v.z, part);
                        part = fmaf(v.w, v.w, part);
                    }
                }
                if (wn * 64 < nb) {
#pragma unroll
                    for (int k0 = 0; k0 < KC; k0 += 8) {
                        uint32_t fa[2][4];
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            const float* const x = a + (wm * 32 + m * 16 + g) * KP + k0 + p;
                            fa[m][0] = to_tf32(x[0]);
                            fa[m][1] = to_tf32(x[8 * KP]);
                            fa[m][2] = to_tf32(x[4]);
                            fa[m][3] = to_tf32(x[8 * KP + 4]);
                        }
#pragma unroll
                        for (int x = 0; x < 8; ++x) {
                            const float* const y = b + (wn * 64 + x * 8 + g) * KP + k0 + p;
                            const uint32_t b0f = __float_as_uint(y[0]), b1f = __float_as_uint(y[4]);
                            mma_tf32(acc[0][x], fa[0], b0f, b1f);
                            mma_tf32(acc[1][x], fa[1], b0f, b1f);
                        }
                    }
                }
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            if (!have_norms) {
                part += __shfl_xor_sync(FULL, part, 1);
                if ((t & 1) == 0) S.row_norm[t >> 1] = part;
                have_norms = true;
                if (PASS == 0) {
                    const uint32_t most = __reduce_max_sync(FULL, __float_as_uint(part));
                    if (lane == 0) atomicMax(A.tile_norm + blockIdx.x, most);
                }
                __syncthreads();
            }
            if (wn * 64 < nb) {
                // this thread's rows are base + g + 8 j, its queries 8 x + 2 p and the next one
                const int base = row0 + wm * 32;
                float finite = 0.f;                                  // or not a number
                // half a bound is (|x|^2 +- own(x) + |q|^2 +- own(q) +- c1 |x| |q|) / 2 - x.q
                float nx[4], sx[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float n = S.row_norm[wm * 32 + g + 8 * j], s = __fsqrt_rn(n), own = error.own(n, s);
                    nx[j] = PASS == 0 ? 0.5f * n + 0.5f * own : 0.5f * n - 0.5f * own;
                    sx[j] = PASS == 0 ? 0.5f * error.c1 * s : -0.5f * error.c1 * s;
                }
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    uint32_t bits[2][4];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int i = wn * 64 + x * 8 + 2 * p + c;
                        const uint32_t l = S.l[i], span = S.span[i], at = (uint32_t)(base + g) - l;
                        const float nq = S.norm[i], sq = S.root[i], tau = S.tau[i];
                        float least = __int_as_float(0x7F800000);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float bound = fmaf(sx[j], sq, (nx[j] + nq) - acc[j >> 1][x][(j & 1) * 2 + c]);
                            const bool in = at + 8u * j <= span;
                            if (PASS == 0) {
                                if (in && bound < least) least = bound;
                                finite = fmaf(bound, 0.f, finite);
                            } else {
                                bits[c][j] = __ballot_sync(FULL, in && !(bound > tau));
                            }
                        }
                        if (PASS == 0) {
                            least = least > 0.f ? 2.f * least : 0.f;
                            least = fminf(least, __shfl_xor_sync(FULL, least, 4));
                            const float wide = fminf(least, __shfl_xor_sync(FULL, least, 8));
                            const float all = fminf(wide, __shfl_xor_sync(FULL, wide, 16));
                            const uint32_t block = (uint32_t)(base >> 5) - (l >> 5);
                            if (block < S.blocks[i]) {
                                const int per = S.per[i];
                                if (per == 4 && (g & 1) == 0) A.store[S.off[i] + 4 * block + (g >> 1)] = __float_as_uint(least);
                                if (per == 1 && g == 0) A.store[S.off[i] + block] = __float_as_uint(all);
                            }
                        }
                    }
                    if (PASS == 1 && lane < 8) {
                        // query 8 x + lane: lanes 4 g + lane / 2 of the ballots of its parity; bit 4 g + j is row g + 8 j
                        uint32_t word = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            word |= ((((lane & 1) ? bits[1][j] : bits[0][j]) >> (lane >> 1)) & 0x11111111u) << j;
                        const int i = wn * 64 + x * 8 + lane;
                        const uint32_t block = (uint32_t)(base >> 5) - (S.l[i] >> 5);
                        if (block < S.blocks[i]) A.store[S.off[i] + block] = word;
                    }
                }
                if (PASS == 0 && !(finite == 0.f)) atomicMax(A.tile_norm + blockIdx.x, 0x7F800000u);
            }
        }
    }
}

// Per query: an upper bound, within 2^-14, of the k-th smallest of its values.  Two passes over the values, eleven bits
// of the (non-negative) numbers each.
__global__ void __launch_bounds__(256)
filter_bound_kernel(const FilterArgs A, int round) {
    __shared__ unsigned int bins[2048];
    __shared__ unsigned int warp_sum[8];
    __shared__ unsigned int found[2];                            // the bin that holds the k-th, values below it
    const int2 queries = round_queries(A, round);
    const int q = queries.x + blockIdx.x, t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    const uint32_t off = q < queries.y ? A.off[q] : BOT;
    if (off == BOT) return;
    const int2 s = A.slab[q];
    const int nv = ((s.y >> 5) - (s.x >> 5) + 1) * values_per_block(s.y - s.x + 1, A.k);
    unsigned int want = (unsigned int)A.k, prefix = 0;
    for (int pass = 0; pass < 2; ++pass) {
        for (int i = t; i < 2048; i += 256) bins[i] = 0u;
        if (t == 0) found[0] = 0x7F8u;
        __syncthreads();
        for (int i = t; i < nv; i += 256) {
            const uint32_t v = A.store[off + i];
            if (pass == 0) atomicAdd(&bins[v >> 20], 1u);
            else if ((v >> 20) == prefix) atomicAdd(&bins[(v >> 9) & 0x7FFu], 1u);
        }
        __syncthreads();
        unsigned int mine = 0;
        for (int i = 0; i < 8; ++i) mine += bins[8 * t + i];
        unsigned int x = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int y = __shfl_up_sync(FULL, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[warp] = x;
        __syncthreads();
        unsigned int below = x - mine;
        for (int w = 0; w < warp; ++w) below += warp_sum[w];
        if (below < want && below + mine >= want) {
            int i = 8 * t;
            while (below + bins[i] < want) below += bins[i++];
            found[0] = (unsigned int)i;
            found[1] = below;
        }
        __syncthreads();
        if (pass == 0) {
            prefix = found[0];
            if (prefix >= 0x7F8u) break;                         // fewer than k finite values
            want -= found[1];
            __syncthreads();
        }
    }
    if (t == 0) A.tau[q] = prefix >= 0x7F8u ? __int_as_float(0x7F800000) : __uint_as_float(prefix << 20 | found[0] << 9 | 0x1FFu);
}

// The rows that are left, one CTA of four warps per query, so that those of 2,000 queries are resident together; four
// rows per team in flight, as a step is a round trip.
constexpr int REFINE_WARPS = 4, REFINE_BUF = 192, REFINE_STEP = REFINE_WARPS * 16;
constexpr int REFINE_MORE = 512;         // rows listed before they are compared; as many as 128 masks give come on top
constexpr int REFINE_LIST = REFINE_MORE + REFINE_WARPS * 32 * 32;
template <int EPL>
struct RefineSmem {
    uint64_t pool[32 * EPL];
    uint64_t buf[REFINE_BUF];            // merged from 128 on, a step adds at most 64
    uint64_t bound;                      // keys from here on are not wanted
    int list[REFINE_LIST];               // rows to compare
    int count, kept;                     // entries of list, of buf
};

template <int EPL>
__global__ void __launch_bounds__(REFINE_WARPS * 32)
filter_refine_kernel(const FilterArgs A, int round) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RefineSmem<EPL>& S = *reinterpret_cast<RefineSmem<EPL>*>(smem_raw);
    const float4* const qs = reinterpret_cast<const float4*>(smem_raw + (sizeof(RefineSmem<EPL>) + 15) / 16 * 16);
    const int2 queries = round_queries(A, round);
    const int q = queries.x + blockIdx.x, t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    if (q >= queries.y) return;
    const int team = t >> 3, sub = lane & 7, groups = A.d_pad >> 2;
    const int2 slab = A.slab[q];
    const int w = slab.y - slab.x + 1;
    const uint32_t off = A.off[q];
    {
        float* qf = reinterpret_cast<float*>(smem_raw + (sizeof(RefineSmem<EPL>) + 15) / 16 * 16);
        for (int i = t; i < A.d_pad; i += REFINE_WARPS * 32) qf[i] = i < A.d ? __ldg(A.queries + (size_t)q * A.d + i) : 0.f;
        for (int i = t; i < 32 * EPL; i += REFINE_WARPS * 32) S.pool[i] = KEY_EMPTY;
        if (t == 0) {
            S.kept = 0;
            S.bound = KEY_EMPTY;
            if (off != BOT && A.tau[q] < __int_as_float(0x7F800000)) S.bound = (uint64_t)__float_as_uint(A.tau[q]) << 32 | 0xFFFFFFFFu;
        }
    }
    auto flush = [&]() {                                         // warp 0
        for (int x = 0; x < S.kept; x += 32) merge_ranked<EPL>(S.pool, S.buf + x, min(32, S.kept - x), A.k, lane);
        __syncwarp();
        if (lane == 0) {
            S.bound = min(S.bound, S.pool[A.k - 1]);
            S.kept = 0;
        }
    };
    // rows list[0..n), or first + [0..n)
    auto compare = [&](int n, int first, bool listed) {
        for (int j0 = 0; j0 < n; j0 += REFINE_STEP) {
            int row[4];
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            const float4* src[4];
            bool on[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int j = j0 + r * (REFINE_WARPS * 4) + team;
                on[r] = j < n;
                row[r] = on[r] ? (listed ? S.list[j] : first + j) : 0;
                src[r] = reinterpret_cast<const float4*>(A.vectors + (size_t)row[r] * (size_t)A.d_pad) + sub;
            }
#pragma unroll 1
            for (int g0 = 0; g0 < groups; g0 += 32) {
                float4 x[4][4];
                const int left = groups - g0 - sub;
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        x[r][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (on[r] && 8 * c < left) x[r][c] = __ldg(src[r] + g0 + 8 * c);
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (8 * c < left) {
                        const float4 v = qs[g0 + sub + 8 * c];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            float u;
                            u = x[r][c].x - v.x; acc[r] = fmaf(u, u, acc[r]);
                            u = x[r][c].y - v.y; acc[r] = fmaf(u, u, acc[r]);
                            u = x[r][c].z - v.z; acc[r] = fmaf(u, u, acc[r]);
                            u = x[r][c].w - v.w; acc[r] = fmaf(u, u, acc[r]);
                        }
                    }
                }
            }
            // the butterfly 4, 2, 1 over the team, every lane handing on the sums it does not keep
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
            const int mine = up4 ? (up2 ? row[3] : row[2]) : (up2 ? row[1] : row[0]);
            const bool have = up4 ? (up2 ? on[3] : on[2]) : (up2 ? on[1] : on[0]);
            if ((sub & 1) == 0 && have && __float_as_uint(d) <= (uint32_t)(S.bound >> 32)) {
                const uint64_t key = make_key(d, (uint32_t)__ldg(A.rank2id + mine), 1u);
                if (key < S.bound) S.buf[atomicAdd(&S.kept, 1)] = key;
            }
            __syncthreads();
            const bool full = S.kept >= REFINE_BUF - REFINE_STEP;
            __syncthreads();
            if (full) {
                if (warp == 0) flush();
                __syncthreads();
            }
        }
    };
    __syncthreads();
    if (off == BOT) {
        compare(w, slab.x, false);
    } else {
        const int blocks = (slab.y >> 5) - (slab.x >> 5) + 1, block0 = slab.x >> 5;
        const uint32_t* const mask = A.store + off + (uint32_t)(blocks * values_per_block(w, A.k));
        constexpr int MASKS = REFINE_WARPS * 32;
        if (t == 0) S.count = 0;
        __syncthreads();
        for (int m0 = 0; m0 < blocks; m0 += 4 * MASKS) {
            uint32_t word[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) word[x] = m0 + x * MASKS + t < blocks ? __ldcg(mask + m0 + x * MASKS + t) : 0u;
#pragma unroll 1
            for (int x = 0; x < 4 && m0 + x * MASKS < blocks; ++x) {
                uint32_t m = x == 0 ? word[0] : x == 1 ? word[1] : x == 2 ? word[2] : word[3];
                int sum = __popc(m);
                const int own = sum;
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, sum, o);
                    if (lane >= o) sum += y;
                }
                int at = 0;
                if (lane == 31 && sum) at = atomicAdd(&S.count, sum);
                at = __shfl_sync(FULL, at, 31) + sum - own;
                for (; m; m &= m - 1) {                          // bit 4 g + j: row g + 8 j of the mask's 32
                    const int bit = __ffs(m) - 1;
                    S.list[at++] = (block0 + m0 + x * MASKS + t) * 32 + (bit >> 2) + 8 * (bit & 3);
                }
                __syncthreads();
                const int n = S.count;
                if (n > REFINE_MORE || m0 + (x + 1) * MASKS >= blocks) {
                    compare(n, 0, true);
                    __syncthreads();
                    if (t == 0) S.count = 0;
                }
                __syncthreads();
            }
        }
    }
    __syncthreads();
    if (warp == 0) flush();
    __syncthreads();
    for (int j = t; j < A.k; j += REFINE_WARPS * 32) {
        const uint64_t key = S.pool[j];
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

}  // namespace
namespace froghost {

namespace {
size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }
typedef void (*filter_fn)(const FilterArgs, int);
size_t refine_smem(int k, int d_pad, filter_fn* fn) {
    const size_t q = (size_t)d_pad * 4;
    if (k <= 32) { *fn = filter_refine_kernel<1>; return up16(sizeof(RefineSmem<1>)) + q; }
    if (k <= 64) { *fn = filter_refine_kernel<2>; return up16(sizeof(RefineSmem<2>)) + q; }
    if (k <= 128) { *fn = filter_refine_kernel<4>; return up16(sizeof(RefineSmem<4>)) + q; }
    if (k <= 256) { *fn = filter_refine_kernel<8>; return up16(sizeof(RefineSmem<8>)) + q; }
    *fn = filter_refine_kernel<16>;
    return up16(sizeof(RefineSmem<16>)) + q;
}
// of a part (the CTAs of its queries, 0.9 ns each, are launched in a round that has nothing to do too)
constexpr size_t MOST_ROUNDS = 1000, MOST_QUERIES = 16384;
// words of the slab that has most
size_t most_words(size_t n, int k) { return std::max(2 * (n / 32 + 2), 5 * (std::min(n, (size_t)128 * k) / 32 + 2)); }
// the arrays of FilterArgs
size_t query_bytes(int d_pad) { return (size_t)d_pad * 4 + 8 + 4 + 4 + 4; }
size_t fixed_bytes(size_t n) { return (n / TILE + 1) * 4 + (MOST_ROUNDS + 1) * 4; }
}  // namespace

size_t filter_bytes(size_t n, size_t nq, int k, int d_pad) {
    return fixed_bytes(n) + std::min(nq, MOST_QUERIES) * (query_bytes(d_pad) + 4 * most_words(n, k));
}

FilterFit filter_fit(size_t n, size_t nq, size_t bytes, int k, int d_pad) {
    FilterFit f{};
    if (bytes < 2 * fixed_bytes(n)) return f;
    f.queries = std::min(nq, MOST_QUERIES);
    if (filter_bytes(n, nq, k, d_pad) > bytes) f.queries = std::min(f.queries, bytes / 4 / query_bytes(d_pad));
    if (f.queries == 0) return f;
    f.parts = (nq + f.queries - 1) / f.queries;
    const size_t each = most_words(n, k);
    // (offsets are 32-bit)
    const size_t words = std::min<size_t>((bytes - fixed_bytes(n) - f.queries * query_bytes(d_pad)) / 4, 0xFFFFFFF0u);
    if (f.queries * each <= words) {
        f.step = words + 1;
        f.rounds = 1;
        f.per_round = f.queries;
    } else if (words > each) {
        f.step = words - each;
        f.rounds = (f.queries - 1) * each / f.step + 1;
        f.per_round = f.step / each;
        if (f.rounds > MOST_ROUNDS) f.queries = 0;
    } else {
        f.queries = 0;
    }
    return f;
}

void filter_scratch(char* mem, FilterArgs* A) {
    const size_t nq = (size_t)A->nq;
    A->rounded = reinterpret_cast<float*>(mem);
    A->slab = reinterpret_cast<int2*>(mem + nq * A->d_pad * 4);
    A->norm = reinterpret_cast<float*>(A->slab + nq);
    A->off = reinterpret_cast<uint32_t*>(A->norm + nq);
    A->tau = reinterpret_cast<float*>(A->off + nq);
    A->tile_norm = reinterpret_cast<uint32_t*>(A->tau + nq);
    A->first = reinterpret_cast<int*>(A->tile_norm + A->n / TILE + 1);
    A->store = reinterpret_cast<uint32_t*>(A->first + MOST_ROUNDS + 1);
}

cudaError_t filter_launch(const FilterArgs& A, int sm_count, cudaStream_t s) {
    filter_fn refine;
    const size_t smem = refine_smem(A.k, A.d_pad, &refine);
    const bool deep = A.d_pad >= 384;
    const filter_fn bounds = deep ? filter_tile_kernel<0, 32> : filter_tile_kernel<0, 16>;
    const filter_fn masks = deep ? filter_tile_kernel<1, 32> : filter_tile_kernel<1, 16>;
    const size_t tile_smem = deep ? sizeof(FilterSmem<32>) : sizeof(FilterSmem<16>);
    cudaError_t e;
    if ((e = allow_smem(refine)) != cudaSuccess || (e = allow_smem(bounds)) != cudaSuccess || (e = allow_smem(masks)) != cudaSuccess)
        return e;
    const int tiles = (A.n - 1) / TILE + 1;
    // two CTAs per SM; several share a tile's queries where there are fewer tiles than that
    const int parts = std::max(1, std::min((A.nq - 1) / TILE + 1, 2 * sm_count / tiles));
    const dim3 grid((unsigned)tiles, (unsigned)parts);
    filter_plan_kernel<<<(A.nq - 1) / 8 + 1, 256, 0, s>>>(A);
    filter_offsets_kernel<<<1, 1024, 0, s>>>(A);
    for (int r = 0; r < A.rounds; ++r) {
        bounds<<<grid, THREADS, tile_smem, s>>>(A, r);
        filter_bound_kernel<<<A.nq, 256, 0, s>>>(A, r);
        masks<<<grid, THREADS, tile_smem, s>>>(A, r);
        refine<<<A.nq, REFINE_WARPS * 32, smem, s>>>(A, r);
    }
    return cudaGetLastError();
}

}  // namespace froghost
