// GPU index builder: the construction of paper Sec. 6 with one warp per object and all objects
// of a layer in flight together (Sec. 6.2.1).  Per layer, bottom-up:
//   candidates   leaf: distances to every other object of the leaf, nearest 64 kept;
//                inner layer: the object's m nearest of its own child segment + the m best of a
//                greedy search (Alg. 1, pool ef_c, patience rule of Sec. 6.2.2) in the sibling's
//                temporary graph;
//   forward row  RNG selection of the candidates in vector-distance order;
//   reverse      the sources of an object's incoming forward edges join its candidates (nearest
//                64 of the union are kept);
//   final        nearest list (m), temporary graph row (RNG selection, vector order) and the
//                layer's ENC row (same selection in ascending fusion distance, Eq. 3).
// The selection needs d(c, p) between candidates: the <= 64 candidate rows of an object are staged
// in shared memory by bulk copies.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <numeric>
#include <vector>

#include <sys/stat.h>
#include <unistd.h>

#include <thrust/execution_policy.h>
#include <thrust/scan.h>

#include "frog_build_gpu.h"
#include "frog_device.cuh"
#include "frog_internal.h"

using namespace frogdev;

namespace {

constexpr int CAND = 64;                 // candidate slots per object
constexpr int BWARPS = 2;                // warps per CTA of the candidate / search / pool kernels
constexpr int STAGE8 = 8 * STAGE_CHUNK;  // stage buffer of staged_dist2<8>

__device__ __forceinline__ void segment_of(int n, int h, int x, int& L, int& R) {
    L = 0;
    R = n - 1;
    for (int depth = 0; depth < h; ++depth) {
        const int mid = L + ((R - L) >> 1);
        if (x <= mid) R = mid; else L = mid + 1;
    }
}

struct BuildArgs {
    const float* V;          // n x d_pad, rank order
    int n, d_pad, H, m, ef_c, patience;
    double beta, gamma, inv_span;
    uint64_t* c1;            // n x CAND keys (d2 bits << 32 | rank << 1 | 1), ascending, KEY_EMPTY tail
    uint64_t* c2;
    uint32_t* ann_cur; float* pd_cur; uint32_t* pg_cur;
    uint32_t* ann_nxt; float* pd_nxt; uint32_t* pg_nxt;
    uint32_t* fwd;           // forward graph rows of the layer under construction
    uint32_t* enc;           // n x H x m
    uint32_t* rev_cnt;       // n + 1
    uint32_t* rev_off;       // n + 1
    uint32_t* rev_cur;       // n
    uint32_t* rev_src;       // n x m
    int h;                   // layer under construction
    int fusion_nearest;      // ENCs = the m fusion-nearest candidates (no RNG rule on them)
    int wait_limit;          // polls a wait on a bulk copy may take before giving up
    int skip_copies;         // test hook: expect the bytes but issue no copy, so that every wait runs out
    uint32_t* fail;          // set to 1 when a wait gave up: the build is not valid
};

// bounded wait on the bulk copies of a pass; records a give-up in *fail
__device__ __forceinline__ void wait_copies(const BuildArgs& A, uint64_t* bar, uint32_t phase) {
    if (!mbar_wait_limit(bar, phase, A.wait_limit)) *A.fail = 1u;
}

// shared-memory slice of one warp in the candidate / search / pool kernels
struct BWarp {
    float4* q;
    uint64_t* pool;      // CAND keys
    uint64_t* spool;     // search pool (sibling search only)
    uint64_t* keys;      // keys of one expansion (sibling search only): the second half of `pool`, empty until its end
    uint32_t* cand;
    uint64_t* bar;
    float4* stage;       // (sibling search: its table of evaluated ranks)
};
constexpr int SEEN_BITS = 10;
static_assert((4 << SEEN_BITS) == STAGE8, "the table takes the place of the stage buffer");
__host__ __device__ inline size_t bwarp_bytes(int d_pad, int spool_slots) {
    return (size_t)d_pad * 4 + CAND * 8 + (size_t)spool_slots * 8 + 32 * 4 + 16 + STAGE8;
}
__device__ __forceinline__ BWarp bwarp_carve(unsigned char* base, int d_pad, int spool_slots) {
    BWarp W;
    W.q = reinterpret_cast<float4*>(base);
    W.pool = reinterpret_cast<uint64_t*>(base + (size_t)d_pad * 4);
    W.spool = W.pool + CAND;
    W.keys = W.pool + 32;                       // the m <= 32 nearest of the own child lie before it
    W.cand = reinterpret_cast<uint32_t*>(W.spool + spool_slots);
    W.bar = reinterpret_cast<uint64_t*>(W.cand + 32);
    W.stage = reinterpret_cast<float4*>(W.bar + 2);
    return W;
}

__device__ __forceinline__ void load_query(const BuildArgs& A, const BWarp& W, int u, int lane) {
    const float4* src = reinterpret_cast<const float4*>(A.V + (size_t)u * A.d_pad);
    for (int i = lane; i < (A.d_pad >> 2); i += 32) W.q[i] = __ldg(src + i);
}

// distances of the ns (<= 32, pairwise distinct) ranks in W.cand to the query, as keys
__device__ __forceinline__ uint64_t cand_keys(const BuildArgs& A, const BWarp& W, int ns, uint32_t flag,
                                              uint32_t& phase, int lane) {
    const uint32_t id = lane < ns ? W.cand[lane] : 0u;
    float d2 = 0.f;
    bool ok = true;
    if (ns > 0) d2 = staged_dist2<8>(A.V, A.d_pad, W.q, W.stage, W.bar, phase, ok, id, ns, lane, A.wait_limit, !A.skip_copies);
    if (!ok) *A.fail = 1u;
    return lane < ns ? make_key(d2, id, flag) : KEY_EMPTY;
}

// ---- leaf layer: nearest CAND of the leaf -----------------------------------------------------
__global__ void __launch_bounds__(BWARPS * 32)
leaf_cand_kernel(const BuildArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const BWarp W = bwarp_carve(smem_raw + bwarp_bytes(A.d_pad, 0) * warp, A.d_pad, 0);
    if (lane == 0) mbar_init(W.bar, 1u);
    __syncwarp();
    uint32_t phase = 0;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int nwarps = gridDim.x * BWARPS;
    for (int u = blockIdx.x * BWARPS + warp; u < A.n; u += nwarps) {
        int L, R;
        segment_of(A.n, A.H - 1, u, L, R);
        load_query(A, W, u, lane);
        W.pool[lane] = KEY_EMPTY;
        W.pool[lane + 32] = KEY_EMPTY;
        __syncwarp();
        for (int b0 = L; b0 <= R; b0 += 32) {
            const int v = b0 + lane;
            const bool keep = v <= R && v != u;
            const uint32_t M = __ballot_sync(FULL, keep);
            if (keep) W.cand[__popc(M & lt_mask)] = (uint32_t)v;
            __syncwarp();
            const uint64_t key = cand_keys(A, W, __popc(M), 1u, phase, lane);
            merge_batch<2>(W.pool, key, CAND, lane);
            __syncwarp();
        }
        A.c1[(size_t)u * CAND + lane] = W.pool[lane];
        A.c1[(size_t)u * CAND + lane + 32] = W.pool[lane + 32];
        __syncwarp();
    }
}

// first pool entry after `from` that is neither expanded nor empty (0xFFFF: none)
template <int EPL>
__device__ __forceinline__ uint32_t next_open(const uint64_t* pool, int from, int lane) {
    for (int e = from >> 5; e < EPL; ++e) {
        const uint32_t lo = reinterpret_cast<const uint32_t*>(pool + lane + 32 * e)[0];     // flag bit; empty keys have it set
        const uint32_t M = __ballot_sync(FULL, !(lo & 1u));
        if (M) return (uint32_t)(32 * e + __ffs(M) - 1);
    }
    return 0xFFFFu;
}

// ---- inner layer: own nearest list + greedy search in the sibling's graph (Alg. 1) ---------------
// One warp per object, SM full of warps: bounded by instruction issue (65 % of the slots).  Rows are read into
// registers (eight in flight per warp), only keys that a full pool does not reject are merged, by rank, and the
// visited set is a table of 1,024 recent ranks in shared memory.  Forgetting is harmless: a vertex evaluated
// again is in the pool, where the merge drops it and the patience rule does not count it, or lies beyond the
// worst of the full pool.  100,000 objects of 384 bytes, ten layers: 60 ms (76.8 with rows staged by bulk copies,
// a bitmap of atomics in L2 and the key-by-key merge; 69 with every new key merged).
template <int EPL>
__global__ void __launch_bounds__(BWARPS * 32, 10)      // 96 registers: 60 ms; 72: 68 ms
sibling_search_kernel(const BuildArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int SPOOL = 32 * EPL;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const BWarp W = bwarp_carve(smem_raw + bwarp_bytes(A.d_pad, SPOOL) * warp, A.d_pad, SPOOL);
    const uint32_t lt_mask = (1u << lane) - 1u;
    uint32_t* const seen = reinterpret_cast<uint32_t*>(W.stage);
    auto slot_of = [&](uint32_t v) -> uint32_t* { return seen + ((v * 0x9E3779B1u) >> (32 - SEEN_BITS)); };
    const int nwarps = gridDim.x * BWARPS;
    for (int u = blockIdx.x * BWARPS + warp; u < A.n; u += nwarps) {
        int L, R;
        segment_of(A.n, A.h, u, L, R);
        const int mid = L + ((R - L) >> 1);
        const int sL = u <= mid ? mid + 1 : L, sR = u <= mid ? R : mid;      // sibling child segment
        load_query(A, W, u, lane);
        W.pool[lane] = KEY_EMPTY;
        W.pool[lane + 32] = KEY_EMPTY;
        for (int i = lane; i < SPOOL; i += 32) W.spool[i] = KEY_EMPTY;
        __syncwarp();
        {   // the m nearest of the own child segment, found one layer below
            uint64_t key = KEY_EMPTY;
            if (lane < A.m) {
                const uint32_t id = A.ann_cur[(size_t)u * A.m + lane];
                if (id != BOT) key = make_key(A.pd_cur[(size_t)u * A.m + lane], id, 1u);
            }
            merge_batch<2>(W.pool, key, CAND, lane);
            __syncwarp();
        }
        if (sL <= sR) {
            const uint4 e4 = make_uint4(BOT, BOT, BOT, BOT);
            for (int i = lane; i < (1 << SEEN_BITS) / 4; i += 32) reinterpret_cast<uint4*>(seen)[i] = e4;
            __syncwarp();
            const uint32_t ep = (uint32_t)(sL + ((sR - sL) >> 1));            // entry point: middle rank
            const float d2 = batch_dist2<4>(A.V, A.d_pad, W.q, ep, 1, lane);
            if (lane == 0) {
                *slot_of(ep) = ep;
                W.keys[0] = make_key(d2, ep, 0u);
            }
            __syncwarp();
            int first = (int)merge_ranked<EPL, true>(W.spool, W.keys, 1, A.ef_c, lane);
            int pat = A.patience;
            for (int it = 0; first < A.ef_c && it < 4 * A.ef_c; ++it) {
                const uint32_t x = key_rank(W.spool[first]);
                const uint64_t mth = W.spool[A.m - 1];                         // m-th best before this expansion
                __syncwarp();
                if (lane == 0) W.spool[first] |= 1ull;
                uint32_t v = BOT;
                if (lane < A.m) v = __ldg(A.pg_cur + (size_t)x * A.m + lane);
                bool keep = false;
                if (v != BOT) {
                    uint32_t* const slot = slot_of(v);
                    keep = *slot != v;
                    if (keep) *slot = v;
                }
                const uint32_t M = __ballot_sync(FULL, keep);
                if (keep) W.cand[__popc(M & lt_mask)] = v;
                __syncwarp();
                const int ns = __popc(M);
                uint64_t key = KEY_EMPTY;
                if (ns > 0) {
                    const uint32_t id = W.cand[lane < ns ? lane : 0];
                    const float d2 = batch_dist2<4>(A.V, A.d_pad, W.q, id, ns, lane);
                    if (lane < ns) key = make_key(d2, id, 0u);
                }
                // only what a full pool does not reject goes through the merge
                const bool close = (key | 1ull) < (W.spool[A.ef_c - 1] | 1ull);
                const uint32_t C = __ballot_sync(FULL, close);
                if (close) W.keys[__popc(C & lt_mask)] = key;
                __syncwarp();
                bool entered = false;
                if (C) first = (int)merge_ranked<EPL, true>(W.spool, W.keys, __popc(C), A.ef_c, lane, &entered);
                else first = (int)next_open<EPL>(W.spool, first, lane);
                // something enters the top m
                const bool improved = __any_sync(FULL, entered && (W.keys[lane] | 1ull) < (mth | 1ull));
                __syncwarp();
                if (improved) pat = A.patience;
                else if (--pat <= 0) break;
            }
            __syncwarp();
            W.keys[lane] = KEY_EMPTY;
            __syncwarp();
            uint64_t key = KEY_EMPTY;
            if (lane < A.m) {
                key = W.spool[lane];
                if (key != KEY_EMPTY) key |= 1ull;
            }
            merge_batch<2>(W.pool, key, CAND, lane);
            __syncwarp();
        }
        A.c1[(size_t)u * CAND + lane] = W.pool[lane];
        A.c1[(size_t)u * CAND + lane + 32] = W.pool[lane + 32];
        __syncwarp();
    }
}

// ---- reverse edges of the forward graph ---------------------------------------------------------
__global__ void rev_count_kernel(const uint32_t* __restrict__ fwd, size_t edges, uint32_t* cnt) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < edges) {
        const uint32_t v = fwd[e];
        if (v != BOT) atomicAdd(cnt + v, 1u);
    }
}
__global__ void rev_fill_kernel(const uint32_t* __restrict__ fwd, size_t edges, int m, const uint32_t* __restrict__ off,
                                uint32_t* cur, uint32_t* src) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < edges) {
        const uint32_t v = fwd[e];
        if (v != BOT) src[off[v] + atomicAdd(cur + v, 1u)] = (uint32_t)(e / (size_t)m);
    }
}

// ---- candidates + sources of incoming edges, nearest CAND -----------------------------------------
__global__ void __launch_bounds__(BWARPS * 32)
pool_kernel(const BuildArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const BWarp W = bwarp_carve(smem_raw + bwarp_bytes(A.d_pad, 0) * warp, A.d_pad, 0);
    if (lane == 0) mbar_init(W.bar, 1u);
    __syncwarp();
    uint32_t phase = 0;
    const int nwarps = gridDim.x * BWARPS;
    for (int u = blockIdx.x * BWARPS + warp; u < A.n; u += nwarps) {
        load_query(A, W, u, lane);
        W.pool[lane] = A.c1[(size_t)u * CAND + lane];
        W.pool[lane + 32] = A.c1[(size_t)u * CAND + lane + 32];
        __syncwarp();
        const uint32_t e1 = A.rev_off[u + 1];
        for (uint32_t e0 = A.rev_off[u]; e0 < e1; e0 += 32) {
            const int ns = (int)min(32u, e1 - e0);
            if (lane < ns) W.cand[lane] = A.rev_src[e0 + lane];
            __syncwarp();
            const uint64_t key = cand_keys(A, W, ns, 1u, phase, lane);
            merge_batch<2>(W.pool, key, CAND, lane);          // a source that is already a candidate is dropped
            __syncwarp();
        }
        A.c2[(size_t)u * CAND + lane] = W.pool[lane];
        A.c2[(size_t)u * CAND + lane + 32] = W.pool[lane + 32];
        __syncwarp();
    }
}

// ---- selection: the RNG rule over the candidates of an object -----------------------------------------
// The rule visits the candidates in order and keeps c iff d(u,c) < d(c,p) for every kept p.  Here a kept
// candidate strikes out, in one step, every later one that it rules out: the next one to keep is the first
// that nobody has struck.  The same set is kept, and of the K (K - 1) / 2 pair distances only those between
// kept candidates and later ones still standing are computed (about a fifth of 2,016).  A team of 8 lanes
// per pair; the candidate rows lie in shared memory (bulk copies), or are read from L2 where 64 of them do not fit.
// Bounded by shared-memory reads of the rows.  100,000 objects of 384 bytes, eleven layers, both selections: 38 ms
// (212 with one warp per object and all pair distances).
struct SelSmem {
    uint64_t* keys;      // CAND
    double* fus;         // CAND fusion distances
    uint64_t* bar;
    uint32_t* dead;      // 3 x 2 words: positions struck out in a round (three rounds take turns)
    uint8_t* ord;        // CAND: candidate at each position of the visiting order
    uint8_t* list;       // CAND per warp: positions still standing
    float4* rows;        // CAND rows (staged form)
};
constexpr int SEL_MIN_WARPS = 2, SEL_MAX_WARPS = 8;      // 384-byte rows: 4 warps are 11 % slower than 2
constexpr size_t SEL_FIXED = CAND * 8 + CAND * 8 + 16 + 32 + CAND + SEL_MAX_WARPS * CAND;
static_assert(SEL_FIXED % 16 == 0, "the rows follow at a 16-byte boundary");
inline size_t sel_bytes(int d_pad, bool staged) { return SEL_FIXED + (staged ? (size_t)CAND * d_pad * 4 : 0); }

// Returns the kept positions (at most m) of ord[0..K) as a mask.  Called by the whole CTA.
__device__ __forceinline__ uint64_t rng_keep(const SelSmem& S, const char* const rows, const uint64_t* keys, bool staged,
                                             int row_bytes, int K, int m) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int sub = lane & 7, team = threadIdx.x >> 3, teams = blockDim.x >> 3;
    uint8_t* const list = S.list + warp * CAND;
    auto row_of = [&](int c) {
        return reinterpret_cast<const float4*>(rows + (size_t)(staged ? (uint32_t)c : key_rank(keys[c])) * (size_t)row_bytes);
    };
    uint64_t standing = K < 64 ? (1ull << K) - 1ull : ~0ull, kept = 0;
    int nk = 0;
    for (int round = 0; standing; ++round) {
        const int t = __ffsll((long long)standing) - 1;
        standing &= standing - 1ull;
        kept |= 1ull << t;
        if (++nk == m || standing == 0) break;
        // positions still standing, in order (one copy per warp)
        const uint32_t lo = (uint32_t)standing, hi = (uint32_t)(standing >> 32), lt = (1u << lane) - 1u;
        if ((lo >> lane) & 1u) list[__popc(lo & lt)] = (uint8_t)lane;
        if ((hi >> lane) & 1u) list[__popc(lo) + __popc(hi & lt)] = (uint8_t)(lane + 32);
        uint32_t* const dead = S.dead + 2 * (round % 3);
        if (threadIdx.x < 2) S.dead[2 * ((round + 1) % 3) + threadIdx.x] = 0u;
        __syncwarp();
        const float4* const xc = row_of(S.ord[t]);
        const int na = __popcll(standing);
        for (int j0 = 0; j0 < na; j0 += 2 * teams) {            // uniform trip count: the sums need whole warps
            const int j[2] = {j0 + team, j0 + team + teams};
            int pos[2], cand[2];
            const float4* x[2];
            float d[2] = {0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                pos[i] = list[min(j[i], na - 1)];
                cand[i] = S.ord[pos[i]];
                x[i] = row_of(cand[i]);
            }
            const bool two = j0 + teams < na;                    // CTA-uniform
            for (int c0 = 0; c0 < row_bytes; c0 += STAGE_CHUNK) {
                const int g_lo = c0 >> 4, g_n = min(STAGE_CHUNK, row_bytes - c0) >> 4;
                float a0 = 0.f, a1 = 0.f;
#pragma unroll
                for (int c = 0; c < STAGE_CHUNK / 128; ++c) {
                    const int g = sub + 8 * c;
                    if (g < g_n) {
                        const float4 p = xc[g_lo + g], y = x[0][g_lo + g];
                        float w;
                        w = p.x - y.x; a0 = fmaf(w, w, a0);
                        w = p.y - y.y; a0 = fmaf(w, w, a0);
                        w = p.z - y.z; a0 = fmaf(w, w, a0);
                        w = p.w - y.w; a0 = fmaf(w, w, a0);
                        if (two) {
                            const float4 z = x[1][g_lo + g];
                            w = p.x - z.x; a1 = fmaf(w, w, a1);
                            w = p.y - z.y; a1 = fmaf(w, w, a1);
                            w = p.z - z.z; a1 = fmaf(w, w, a1);
                            w = p.w - z.w; a1 = fmaf(w, w, a1);
                        }
                    }
                }
                a0 += __shfl_xor_sync(FULL, a0, 4);
                a1 += __shfl_xor_sync(FULL, a1, 4);
                a0 += __shfl_xor_sync(FULL, a0, 2);
                a1 += __shfl_xor_sync(FULL, a1, 2);
                a0 += __shfl_xor_sync(FULL, a0, 1);
                a1 += __shfl_xor_sync(FULL, a1, 1);
                d[0] += a0;
                d[1] += a1;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (sub == 0 && j[i] < na && !(key_dist2(keys[cand[i]]) < d[i]))
                    atomicOr(dead + (pos[i] >> 5), 1u << (pos[i] & 31));
        }
        __syncthreads();
        standing &= ~((uint64_t)dead[0] | (uint64_t)dead[1] << 32);
    }
    // round 0 of the next call finds its words zero
    __syncthreads();
    if (threadIdx.x < 2) S.dead[threadIdx.x] = 0u;
    __syncthreads();
    return kept;
}

template <bool FINAL, bool STAGED>
__global__ void __launch_bounds__(SEL_MAX_WARPS * 32)
select_kernel(const BuildArgs A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SelSmem S;
    S.keys = reinterpret_cast<uint64_t*>(smem_raw);
    S.fus = reinterpret_cast<double*>(S.keys + CAND);
    S.bar = reinterpret_cast<uint64_t*>(S.fus + CAND);
    S.dead = reinterpret_cast<uint32_t*>(S.bar + 2);
    S.ord = reinterpret_cast<uint8_t*>(S.dead + 8);
    S.list = S.ord + CAND;
    S.rows = reinterpret_cast<float4*>(smem_raw + SEL_FIXED);
    const int lane = lane_id(), tid = threadIdx.x;
    if (tid == 0) mbar_init(S.bar, 1u);
    if (tid < 8) S.dead[tid] = 0u;
    __syncthreads();
    uint32_t phase = 0;
    const uint64_t* cin = FINAL ? A.c2 : A.c1;
    const int row_bytes = A.d_pad * 4;
    const char* const rows = STAGED ? reinterpret_cast<const char*>(S.rows) : reinterpret_cast<const char*>(A.V);
    for (int u = blockIdx.x; u < A.n; u += gridDim.x) {
        const uint64_t k0 = cin[(size_t)u * CAND + lane], k1 = cin[(size_t)u * CAND + lane + 32];   // every warp, for K
        const int K = __popc(__ballot_sync(FULL, k0 != KEY_EMPTY)) + __popc(__ballot_sync(FULL, k1 != KEY_EMPTY));
        if (tid < 32) {
            S.keys[lane] = k0;
            S.keys[lane + 32] = k1;
            S.ord[lane] = (uint8_t)lane;                           // vector-distance order: the keys are ascending
            S.ord[lane + 32] = (uint8_t)(lane + 32);
            if (STAGED && lane == 0 && !A.skip_copies) mbar_expect_tx(S.bar, (uint32_t)(K * row_bytes));
        }
        __syncthreads();
        if (STAGED) {
            for (int r = tid; r < K; r += blockDim.x)
                if (!A.skip_copies)
                    tma_load_1d(reinterpret_cast<char*>(S.rows) + (size_t)r * row_bytes,
                                reinterpret_cast<const char*>(A.V) + (size_t)key_rank(S.keys[r]) * row_bytes,
                                (uint32_t)row_bytes, S.bar);
            wait_copies(A, S.bar, phase);
            phase ^= 1u;
        }
        // temporary graph row: kept candidates in vector-distance order, then the others up to m
        const uint64_t kept = rng_keep(S, rows, S.keys, STAGED, row_bytes, K, A.m);
        const int nk = __popcll(kept);
        uint32_t* grow = (FINAL ? A.pg_nxt : A.fwd) + (size_t)u * A.m;
        for (int i = tid; i < CAND; i += blockDim.x) {
            const uint64_t below = (1ull << i) - 1ull;
            const int at = (kept >> i) & 1ull ? __popcll(kept & below) : nk + __popcll(~kept & below);
            if (i < K && at < A.m) grow[at] = key_rank(S.keys[i]);
            if (i >= K && i < A.m) grow[i] = BOT;
        }
        if (FINAL) {
            for (int i = tid; i < CAND; i += blockDim.x) {
                if (i < A.m) {
                    const bool has = i < K;
                    A.ann_nxt[(size_t)u * A.m + i] = has ? key_rank(S.keys[i]) : BOT;
                    A.pd_nxt[(size_t)u * A.m + i] = has ? key_dist2(S.keys[i]) : 0.f;
                }
                // ENC row: the same rule with the candidates in ascending fusion distance (Eq. 3)
                if (i < K) {
                    const double dv = sqrt((double)key_dist2(S.keys[i]));
                    const double da = fabs((double)u - (double)key_rank(S.keys[i])) * A.inv_span;
                    const double za = A.gamma == 0.5 ? sqrt(da) : pow(da, A.gamma);   // sqrt is exact on both builders
                    S.fus[i] = dv * (1.0 - A.beta * (1.0 - za));
                }
            }
            __syncthreads();
            for (int i = tid; i < K; i += blockDim.x) {
                const double fi = S.fus[i];
                const uint32_t ri = key_rank(S.keys[i]);
                int pos = 0;
                for (int j = 0; j < K; ++j) {
                    const double fj = S.fus[j];
                    pos += (fj < fi || (fj == fi && key_rank(S.keys[j]) < ri)) ? 1 : 0;
                }
                S.ord[pos] = (uint8_t)i;
            }
            __syncthreads();
            const uint64_t all = K < 64 ? (1ull << K) - 1ull : ~0ull;
            uint64_t enc = 0ull;                               // as it stands: the m fusion-nearest
            if (!A.fusion_nearest) enc = rng_keep(S, rows, S.keys, STAGED, row_bytes, K, A.m);
            uint64_t spare = all & ~enc;
            for (int x = __popcll(enc); x < A.m && spare; ++x) {
                enc |= spare & (0ull - spare);
                spare &= spare - 1ull;
            }
            // the chosen candidates in ascending fusion distance
            uint32_t* erow = A.enc + ((size_t)u * A.H + A.h) * A.m;
            for (int i = tid; i < CAND; i += blockDim.x) {
                if ((enc >> i) & 1ull) erow[__popcll(enc & ((1ull << i) - 1ull))] = key_rank(S.keys[S.ord[i]]);
                if (i >= __popcll(enc) && i < A.m) erow[i] = BOT;
            }
        }
        __syncthreads();                                           // everyone is done with the rows and keys
    }
}

// rows of the caller's array to their places in rank order, zero-padded to d_pad
__global__ void rank_rows_kernel(const float* __restrict__ raw, const int32_t* __restrict__ ranks, int d, int d_pad, size_t elems,
                                 float* __restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / d_pad;
        const int c = (int)(i - r * d_pad);
        out[(size_t)ranks[r] * d_pad + c] = c < d ? raw[r * d + c] : 0.f;
    }
}

// ---- host side ------------------------------------------------------------------------------------
bool write_all(FILE* f, const void* p, size_t bytes) {
    const char* c = static_cast<const char*>(p);
    while (bytes) {
        const size_t chunk = std::min<size_t>(bytes, (size_t)1 << 30);
        if (fwrite(c, 1, chunk, f) != chunk) return false;
        c += chunk;
        bytes -= chunk;
    }
    return true;
}
bool pad_to(FILE* f, uint64_t& pos, uint64_t target) {
    static const char zeros[128] = {0};
    while (pos < target) {
        const size_t c = (size_t)std::min<uint64_t>(target - pos, sizeof(zeros));
        if (fwrite(zeros, 1, c, f) != c) return false;
        pos += c;
    }
    return true;
}
inline uint64_t align128(uint64_t x) { return (x + 127) & ~(uint64_t)127; }

struct DeviceBuffers {
    std::vector<void*> ptrs;
    ~DeviceBuffers() { for (void* p : ptrs) cudaFree(p); }
    template <typename T> int alloc(T** out, size_t count) {
        void* p = nullptr;
        cudaError_t e = cudaMalloc(&p, count * sizeof(T));
        if (e != cudaSuccess) {
            cudaGetLastError();
            froghost::set_cuda_error(e);
            return FROG_ERR_NOMEM;
        }
        ptrs.push_back(p);
        *out = static_cast<T*>(p);
        return FROG_OK;
    }
};

int ceil_log2_i64(int64_t n) {
    int b = 0;
    while (((int64_t)1 << b) < n) ++b;
    return b;
}

int build_index(const float* vectors, const int32_t* attrs, int64_t n64, int32_t d, const frog_build_params_t* params, int device,
                const char* path) {
    if (!vectors || !attrs || !path || n64 < 1 || d < 1 || n64 >= ((int64_t)1 << 31) - 1 || device < 0)
        return FROG_ERR_INVALID_ARG;
    frog_build_params_t P{};
    if (params) P = *params;
    else { P.n_inv = -1; P.beta = -1.f; }
    if (P.m == 0) P.m = d <= 300 ? 16 : 32;
    if (P.ef_c == 0) P.ef_c = d <= 300 ? 128 : 256;
    if (P.n_inv < 0) P.n_inv = d <= 300 ? 7 : 6;
    if (P.patience == 0) P.patience = 30;
    if (P.beta < 0) P.beta = 0.2f;
    if (P.gamma <= 0) P.gamma = 0.5f;
    if (P.m < 1 || P.ef_c < P.m || P.patience < 1) return FROG_ERR_INVALID_ARG;
    if (P.m > 32 || P.ef_c > 256) return FROG_ERR_UNSUPPORTED;
    const int n = (int)n64, m = P.m;
    int H = ceil_log2_i64(n64) + 1 - P.n_inv;
    if (H < 1) H = 1;
    const int d_pad = (d + 3) / 4 * 4;

    int dev_count = 0;
    FROG_CUDA_TRY(cudaGetDeviceCount(&dev_count));
    if (device >= dev_count) return FROG_ERR_INVALID_ARG;
    FROG_CUDA_TRY(cudaSetDevice(device));
    cudaDeviceProp prop;
    FROG_CUDA_TRY(cudaGetDeviceProperties(&prop, device));

    // Sec. 4: rank domain (host)
    std::vector<int32_t> rank2id((size_t)n);
    std::iota(rank2id.begin(), rank2id.end(), 0);
    std::stable_sort(rank2id.begin(), rank2id.end(), [&](int32_t a, int32_t b) { return attrs[a] < attrs[b]; });
    std::vector<int32_t> sorted_attr((size_t)n);
    for (int64_t r = 0; r < n; ++r) sorted_attr[r] = attrs[rank2id[r]];

    DeviceBuffers buf;
    BuildArgs A{};
    float* dV = nullptr;
    int rc;
    const size_t nm = (size_t)n * m;
    uint32_t *annA, *annB, *pgA, *pgB;
    float *pdA, *pdB;
    if ((rc = buf.alloc(&dV, (size_t)n * d_pad)) || (rc = buf.alloc(&A.c1, (size_t)n * CAND)) ||
        (rc = buf.alloc(&A.c2, (size_t)n * CAND)) || (rc = buf.alloc(&annA, nm)) || (rc = buf.alloc(&annB, nm)) ||
        (rc = buf.alloc(&pgA, nm)) || (rc = buf.alloc(&pgB, nm)) || (rc = buf.alloc(&pdA, nm)) ||
        (rc = buf.alloc(&pdB, nm)) || (rc = buf.alloc(&A.fwd, nm)) || (rc = buf.alloc(&A.enc, nm * H)) ||
        (rc = buf.alloc(&A.rev_cnt, (size_t)n + 1)) || (rc = buf.alloc(&A.rev_off, (size_t)n + 1)) ||
        (rc = buf.alloc(&A.rev_cur, (size_t)n)) || (rc = buf.alloc(&A.rev_src, nm)) || (rc = buf.alloc(&A.fail, 1)))
        return rc;
    FROG_CUDA_TRY(cudaMemset(A.fail, 0, sizeof(uint32_t)));
    const bool reverse_edges = !(P.reserved & FROG_BUILD_NO_REVERSE_EDGES);
    A.fusion_nearest = (P.reserved & FROG_BUILD_ENC_FUSION_NEAREST) ? 1 : 0;
    // test hook (bits 16..31 of `reserved`): a nonzero value v makes every wait give up after v polls
    // and neither arms the barriers nor issues a copy, so that the give-up path runs with nothing in flight
    A.wait_limit = (P.reserved >> 16) ? (P.reserved >> 16) : (1 << 22);
    A.skip_copies = (P.reserved >> 16) ? 1 : 0;
    {   // rows in rank order, padded, are put together on the device, from slabs of the caller's array of at most 256 MB
        DeviceBuffers once;
        float* raw = nullptr;
        int32_t* ranks = nullptr;
        const size_t slab = std::min<size_t>((size_t)n, std::max<size_t>(((size_t)64 << 20) / d, 1));
        if ((rc = once.alloc(&raw, slab * d)) || (rc = once.alloc(&ranks, (size_t)n))) return rc;
        std::vector<int32_t> rank_of((size_t)n);
        for (int r = 0; r < n; ++r) rank_of[rank2id[r]] = r;
        FROG_CUDA_TRY(cudaMemcpy(ranks, rank_of.data(), (size_t)n * 4, cudaMemcpyHostToDevice));
        for (size_t i0 = 0; i0 < (size_t)n; i0 += slab) {
            const size_t rows = std::min(slab, (size_t)n - i0), elems = rows * d_pad;
            FROG_CUDA_TRY(cudaMemcpy(raw, vectors + i0 * d, rows * d * 4, cudaMemcpyHostToDevice));
            const unsigned grid = (unsigned)std::min<size_t>((elems + 255) / 256, (size_t)prop.multiProcessorCount * 32);
            rank_rows_kernel<<<grid, 256>>>(raw, ranks + i0, d, d_pad, elems, dV);
            FROG_CUDA_TRY(cudaGetLastError());
        }
        FROG_CUDA_TRY(cudaDeviceSynchronize());
    }
    A.V = dV;
    A.n = n; A.d_pad = d_pad; A.H = H; A.m = m; A.ef_c = P.ef_c; A.patience = P.patience;
    A.beta = P.beta; A.gamma = P.gamma; A.inv_span = n > 1 ? 1.0 / (double)(n - 1) : 0.0;
    A.ann_cur = annA; A.ann_nxt = annB; A.pg_cur = pgA; A.pg_nxt = pgB; A.pd_cur = pdA; A.pd_nxt = pdB;

    // launch shapes
    const int spool_slots = P.ef_c <= 32 ? 32 : P.ef_c <= 64 ? 64 : P.ef_c <= 128 ? 128 : 256;
    const size_t smem_plain = bwarp_bytes(d_pad, 0) * BWARPS, smem_search = bwarp_bytes(d_pad, spool_slots) * BWARPS;
    void (*search_fn)(const BuildArgs) = spool_slots == 32 ? sibling_search_kernel<1>
                                       : spool_slots == 64 ? sibling_search_kernel<2>
                                       : spool_slots == 128 ? sibling_search_kernel<4> : sibling_search_kernel<8>;
    if (smem_search > froghost::MAX_SMEM) return FROG_ERR_UNSUPPORTED;
    // the selection stages all 64 rows where they fit; about 16 warps per SM share its shared memory, and a CTA
    // is given more of them the fewer CTAs that leaves room for
    const bool staged = sel_bytes(d_pad, true) <= froghost::MAX_SMEM;
    const size_t smem_sel = sel_bytes(d_pad, staged);
    const int sel_ctas = std::max<int>(1, (int)(froghost::MAX_SMEM / (smem_sel + 1024)));
    const int sel_warps = std::min(SEL_MAX_WARPS, std::max(SEL_MIN_WARPS, 16 / sel_ctas));
    void (*sel0)(const BuildArgs) = staged ? select_kernel<false, true> : select_kernel<false, false>;
    void (*sel1)(const BuildArgs) = staged ? select_kernel<true, true> : select_kernel<true, false>;
    FROG_CUDA_TRY(froghost::allow_smem(leaf_cand_kernel));
    FROG_CUDA_TRY(froghost::allow_smem(pool_kernel));
    FROG_CUDA_TRY(froghost::allow_smem(search_fn));
    FROG_CUDA_TRY(froghost::allow_smem(sel0));
    FROG_CUDA_TRY(froghost::allow_smem(sel1));
    auto grid_for = [&](const void* fn, int threads, size_t smem, int per_cta) {
        int per_sm = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
        if (per_sm < 1) per_sm = 1;
        long long g = (long long)per_sm * prop.multiProcessorCount;
        const long long need = ((long long)n + per_cta - 1) / per_cta;
        return (int)std::max<long long>(1, std::min(g, need));
    };
    const int g_plain = grid_for((const void*)leaf_cand_kernel, BWARPS * 32, smem_plain, BWARPS);
    const int g_pool = grid_for((const void*)pool_kernel, BWARPS * 32, smem_plain, BWARPS);
    const int g_search = grid_for((const void*)search_fn, BWARPS * 32, smem_search, BWARPS);
    const int g_sel0 = grid_for((const void*)sel0, sel_warps * 32, smem_sel, 1);
    const int g_sel1 = grid_for((const void*)sel1, sel_warps * 32, smem_sel, 1);

    const size_t edges = nm;
    const int eb = 256, eg = (int)((edges + eb - 1) / eb);
    for (int h = H - 1; h >= 0; --h) {
        A.h = h;
        if (h == H - 1) leaf_cand_kernel<<<g_plain, BWARPS * 32, smem_plain>>>(A);
        else search_fn<<<g_search, BWARPS * 32, smem_search>>>(A);
        sel0<<<g_sel0, sel_warps * 32, smem_sel>>>(A);
        FROG_CUDA_TRY(cudaMemsetAsync(A.rev_cnt, 0, ((size_t)n + 1) * 4));
        FROG_CUDA_TRY(cudaMemsetAsync(A.rev_cur, 0, (size_t)n * 4));
        if (reverse_edges) {
            rev_count_kernel<<<eg, eb>>>(A.fwd, edges, A.rev_cnt);
            thrust::exclusive_scan(thrust::device, A.rev_cnt, A.rev_cnt + n + 1, A.rev_off);
            rev_fill_kernel<<<eg, eb>>>(A.fwd, edges, m, A.rev_off, A.rev_cur, A.rev_src);
        } else {
            FROG_CUDA_TRY(cudaMemsetAsync(A.rev_off, 0, ((size_t)n + 1) * 4));      // no incoming sources
        }
        pool_kernel<<<g_pool, BWARPS * 32, smem_plain>>>(A);
        sel1<<<g_sel1, sel_warps * 32, smem_sel>>>(A);
        FROG_CUDA_TRY(cudaGetLastError());
        std::swap(A.ann_cur, A.ann_nxt);
        std::swap(A.pd_cur, A.pd_nxt);
        std::swap(A.pg_cur, A.pg_nxt);
    }
    FROG_CUDA_TRY(cudaDeviceSynchronize());
    {
        uint32_t failed = 0;
        FROG_CUDA_TRY(cudaMemcpy(&failed, A.fail, sizeof(failed), cudaMemcpyDeviceToHost));
        if (failed) return FROG_ERR_CUDA;      // a bulk copy never completed: no file is written
    }

    // the index file (same layout as the host builder writes)
    unsigned char hdr[256];
    std::memset(hdr, 0, sizeof(hdr));
    std::memcpy(hdr, "FROGIDX1", 8);
    const uint32_t u32s[8] = {1u, (uint32_t)d, (uint32_t)d_pad, (uint32_t)H, (uint32_t)m,
                              (uint32_t)P.n_inv, (uint32_t)P.ef_c, (uint32_t)P.patience};
    std::memcpy(hdr + 8, u32s, sizeof(u32s));
    std::memcpy(hdr + 40, &P.beta, 4);
    std::memcpy(hdr + 44, &P.gamma, 4);
    const uint64_t nn = (uint64_t)n;
    std::memcpy(hdr + 48, &nn, 8);
    std::memcpy(hdr + 56, &P.seed, 8);
    const uint32_t bot = BOT;
    std::memcpy(hdr + 64, &bot, 4);
    const uint32_t flags = (uint32_t)P.reserved & (FROG_BUILD_NO_REVERSE_EDGES | FROG_BUILD_ENC_FUSION_NEAREST);
    std::memcpy(hdr + 68, &flags, 4);
    const uint64_t off_attr = 256, off_r2i = align128(off_attr + nn * 4), off_vec = align128(off_r2i + nn * 4),
                   off_enc = align128(off_vec + nn * d_pad * 4), total = off_enc + nn * H * m * 4;
    const uint64_t offs[5] = {off_attr, off_r2i, off_vec, off_enc, total};
    std::memcpy(hdr + 72, offs, sizeof(offs));
    FILE* f = fopen(path, "wb");
    if (!f) return FROG_ERR_IO;
    struct stat file;
    const bool regular = fstat(fileno(f), &file) == 0 && S_ISREG(file.st_mode);
    // The arrays of a regular file are written by several threads, out of order, so the length says nothing about
    // how far they got: until all of them are there the header is zeros, which frog_index_load refuses.
    const unsigned char unfinished[256] = {0};
    uint64_t pos = 256;
    bool ok = write_all(f, regular ? unfinished : hdr, 256) && write_all(f, sorted_attr.data(), (size_t)n * 4);
    pos += nn * 4;
    ok = ok && pad_to(f, pos, off_r2i) && write_all(f, rank2id.data(), (size_t)n * 4);
    pos += nn * 4;
    ok = ok && pad_to(f, pos, off_vec) && fflush(f) == 0;
    rc = ok ? FROG_OK : FROG_ERR_IO;
    if (ok && regular) {
        // (the gap before the ENC array reads as zeros)
        const froghost::FileSection sections[2] = {{off_vec, dV, (size_t)n * d_pad * 4}, {off_enc, A.enc, nm * H * 4}};
        rc = froghost::transfer_sections(fileno(f), device, sections, 2, false);
        if (rc == FROG_OK && pwrite(fileno(f), hdr, sizeof(hdr), 0) != (ssize_t)sizeof(hdr)) rc = FROG_ERR_IO;
    } else if (ok) {
        // not a file one can write out of order (a pipe): both arrays through host memory, in order
        std::unique_ptr<char[]> host(new (std::nothrow) char[std::max((size_t)n * d_pad, nm * H) * 4]);
        if (!host) rc = FROG_ERR_NOMEM;
        auto copy = [&](const void* dev, size_t bytes) {
            const cudaError_t e = cudaMemcpy(host.get(), dev, bytes, cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) { froghost::set_cuda_error(e); rc = FROG_ERR_CUDA; }
            else if (!write_all(f, host.get(), bytes)) rc = FROG_ERR_IO;
        };
        if (rc == FROG_OK) copy(dV, (size_t)n * d_pad * 4);
        pos += nn * d_pad * 4;
        if (rc == FROG_OK && !pad_to(f, pos, off_enc)) rc = FROG_ERR_IO;
        if (rc == FROG_OK) copy(A.enc, nm * H * 4);
    }
    if (fclose(f) != 0 && rc == FROG_OK) rc = FROG_ERR_IO;
    return rc;
}

}  // namespace

extern "C" int frog_index_build_gpu(const float* vectors, const int32_t* attrs, int64_t n, int32_t d,
                                    const frog_build_params_t* params, int device, const char* path) {
    try {
        return build_index(vectors, attrs, n, d, params, device, path);
    } catch (...) {                    // the standard containers' way to say that host memory is short
        return FROG_ERR_NOMEM;
    }
}
