// The search kernel for batches that leave warps idle: one CTA per query.
//
// A query is a chain: the next vertex to expand is known only after the candidates of the last one have
// been merged.  With one warp per query (the kernels of frog_search.cu and frog_search_lean.cu) a link of
// that chain costs an ENC load, a round of L2 atomics and a gather that takes a few rows at a time; that is
// the right use of a full GPU, but a batch with fewer queries than warps ends when its longest chain does.
// Here a whole CTA shortens the chain of one query; results are the same, bit for bit:
//   * the first SPEC unexpanded vertices of the pool are prepared together (ENC scan, distances of their
//     ENs) and committed in Alg. 2's order: the j-th of them comes next after its predecessors iff none of
//     their new keys lies before it, so one merge takes the longest such run of them (about two of four).
//     Preparing does not depend on the pool (Alg. 4 under a lazy hash check reads neither pool nor visited
//     set); a prepared vertex that has to wait keeps its slot while it stays among the first;
//   * the visited set is a small direct-mapped table in shared memory that forgets.  That is sound because
//     the merge drops a key the pool already holds, and a vertex the pool has rejected or evicted can
//     never enter later (the pool is full by then and its worst key only falls): forgetting costs a
//     repeated distance, never a result.  It replaces global atomics and slab clearing;
//   * all rows of a step are in flight at once (8-lane teams, register loads, two rows each), and a row
//     longer than 512 bytes is given up as soon as its partial sum exceeds the worst distance of a full
//     pool: sums of squares only grow, rounding included, so the key would be rejected.
// What bounds it: the dependent chain of a round.  Measured for one query on 100,000 512-byte rows (beam 64,
// B 64, 8 warps), cycles of a round that commits two vertices: 3,300 distances, 640 + 1,700 + 790 choice,
// merge and assignment by warp 0, 1,300 ENC scan; 233 us with one warp per query, 138 us here.
#include "frog_device.cuh"
#include "frog_internal.h"

using namespace frogdev;

namespace {

constexpr int TEAM_SPEC = 4;         // vertices prepared ahead (8: 10 % slower, the extra ones are used too seldom)
constexpr int TEAM_CAND = 128;       // candidates of one prepared vertex (largest budget; also >= entry points)
constexpr int DEDUP_BITS = 8;        // per-slot table that drops repeats inside one EN list

template <int SPEC>
struct TeamCtl {
    uint32_t best[SPEC];             // smallest squared distance of the slot's prom list (bits)
    uint64_t key[SPEC];              // the first SPEC unexpanded pool entries: key,
    int pos[SPEC];                   // position in the pool
    int ord[SPEC];                   // and the slot that prepares it
    uint32_t u[SPEC];                // vertex of each slot, BOT = none
    int ncand[SPEC], nprom[SPEC];    // entries of the slot's cand and prom lists
    int part[SPEC][4];               // in-range ENs that each warp of a slot saw
    int n_top, fill_mask, done, next_q;
    uint64_t batch[32];
};

template <int EPL, int SPEC>
struct TeamLayout {
    static constexpr int POOL = 32 * EPL;
    static constexpr size_t OFF_PROM = (size_t)POOL * 8;                              // u64 keys, SPEC x TEAM_CAND
    static constexpr size_t OFF_CAND = OFF_PROM + (size_t)SPEC * TEAM_CAND * 8;
    static constexpr size_t OFF_DEDUP = OFF_CAND + (size_t)SPEC * TEAM_CAND * 4;
    static constexpr size_t OFF_CTL = OFF_DEDUP + ((size_t)SPEC << DEDUP_BITS) * 4;
    static constexpr size_t OFF_Q = (OFF_CTL + sizeof(TeamCtl<SPEC>) + 15) / 16 * 16;       // query, then the visited table
    static size_t bytes(int q_len, int vis_bits) { return OFF_Q + (size_t)q_len * 4 + ((size_t)4 << vis_bits); }
};

template <bool F16>
__device__ __forceinline__ float4 load_group(const char* row, int g) {
    if (F16) {
        uint2 raw;
        asm("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(raw.x), "=r"(raw.y) : "l"(row + g * 8));
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        return make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    return ldg_stream_f4(reinterpret_cast<const float4*>(row) + g);
}
__device__ __forceinline__ float team_sum(float a) {
    a = a + __shfl_xor_sync(FULL, a, 4);
    a = a + __shfl_xor_sync(FULL, a, 2);
    return a + __shfl_xor_sync(FULL, a, 1);
}
__device__ __forceinline__ float add_sq(float acc, const float4& x, const float4& q) {
    float t;
    t = x.x - q.x; acc = fmaf(t, t, acc);
    t = x.y - q.y; acc = fmaf(t, t, acc);
    t = x.z - q.z; acc = fmaf(t, t, acc);
    t = x.w - q.w; return fmaf(t, t, acc);
}

template <int EPL, int W, int SPEC, bool F16>
__global__ void __launch_bounds__(W * 32, W == 16 ? 1 : W == 8 ? 2 : 5)
frog_search_team_kernel(const __grid_constant__ FrogSearchArgs A) {
    using L = TeamLayout<EPL, SPEC>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint64_t* const pool = reinterpret_cast<uint64_t*>(smem_raw);
    uint64_t* const prom = reinterpret_cast<uint64_t*>(smem_raw + L::OFF_PROM);
    uint32_t* const cand = reinterpret_cast<uint32_t*>(smem_raw + L::OFF_CAND);
    uint32_t* const dedup = reinterpret_cast<uint32_t*>(smem_raw + L::OFF_DEDUP);
    TeamCtl<SPEC>& ctl = *reinterpret_cast<TeamCtl<SPEC>*>(smem_raw + L::OFF_CTL);
    const float4* const qs = reinterpret_cast<const float4*>(smem_raw + L::OFF_Q);
    uint32_t* const vis = reinterpret_cast<uint32_t*>(smem_raw + L::OFF_Q + (size_t)A.q_len * 4);
    const int lane = lane_id();
    const int warp = threadIdx.x >> 5;
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int vis_shift = 32 - A.hash_bits;
    const int G = (A.d + 3) >> 2;                                  // 4-element groups of a row
    const char* const rows = static_cast<const char*>(A.rows);
    if (blockIdx.x == 0 && threadIdx.x == 0) A.work_counter[1] = 0u;   // nothing to report: no copy that could time out

    auto vis_slot = [&](uint32_t v) -> uint32_t* { return vis + ((v * 0x9E3779B1u) >> vis_shift); };
    auto dd_slot = [&](int s, uint32_t v) -> uint32_t* {
        return dedup + (s << DEDUP_BITS) + ((v * 0x85EBCA6Bu) >> (32 - DEDUP_BITS));
    };
    // distances of the candidates of the slots in `mask`; keys that would enter the pool as it stands go
    // to the slots' prom lists (any order), the others are marked visited (they can never enter)
    auto distances = [&](int mask, uint32_t new_flag, int L_start, int total) {
        int end[SPEC], n = 0;
#pragma unroll
        for (int s = 0; s < SPEC; ++s) {
            if ((mask >> s) & 1) n += ctl.ncand[s];
            end[s] = n;
        }
        const uint64_t worst = pool[A.ef_s - 1];
        const float worst_d = key_dist2(worst);                   // not a number while the pool is not full
        const int team = warp * 4 + (lane >> 3), sub = lane & 7;
#pragma unroll 1
        for (int j0 = 0; j0 < n; j0 += 8 * W) {
            const int j[2] = {j0 + team, j0 + team + 4 * W};
            uint32_t id[2];
            int sl[2];
            const char* row[2];
            bool on[2];
            float acc[2] = {0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                on[i] = j[i] < n;
                int s = 0, base = 0;
#pragma unroll
                for (int t = 0; t + 1 < SPEC; ++t)
                    if (j[i] >= end[t]) { s = t + 1; base = end[t]; }
                sl[i] = s;
                id[i] = on[i] ? cand[s * TEAM_CAND + j[i] - base] : 0u;
                row[i] = rows + (size_t)id[i] * (size_t)A.row_bytes;
            }
            const bool was[2] = {on[0], on[1]};
#pragma unroll 1
            for (int g0 = 0; g0 < G; g0 += 32) {
                float4 x[2][4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int g = g0 + 8 * c + sub;
                    if (on[0] && g < G) x[0][c] = load_group<F16>(row[0], g);
                    if (on[1] && g < G) x[1][c] = load_group<F16>(row[1], g);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int g = g0 + 8 * c + sub;
                    if (g < G) {
                        const float4 q = qs[g];
                        if (on[0]) acc[0] = add_sq(acc[0], x[0][c], q);
                        if (on[1]) acc[1] = add_sq(acc[1], x[1][c], q);
                    }
                }
                if (g0 + 32 < G) {
                    const float p0 = team_sum(acc[0]), p1 = team_sum(acc[1]);
                    on[0] = on[0] && !(p0 > worst_d);
                    on[1] = on[1] && !(p1 > worst_d);
                    if (!__any_sync(FULL, on[0] || on[1])) break;
                }
            }
            const float d[2] = {team_sum(acc[0]), team_sum(acc[1])};
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint64_t key = make_key(d[i], id[i], new_flag);
                const bool enters = on[i] && (key | 1ull) < (worst | 1ull);
                if (enters && sub == 0) {
                    prom[sl[i] * TEAM_CAND + atomicAdd(&ctl.nprom[sl[i]], 1)] = key;
                    atomicMin(&ctl.best[sl[i]], (uint32_t)(key >> 32));
                }
                if (!enters && was[i] && sub == 0) *vis_slot(id[i]) = id[i];
                if (enters && sub * 32 < total) {                  // it may be expanded: its ENC rows towards L2
                    const uint32_t* hot = A.enc + ((size_t)id[i] * A.H + L_start) * A.m;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(hot + sub * 32));
                }
            }
        }
    };
    // merge the prom lists of the first c prepared vertices (warp 0); returns the first unexpanded position
    auto merge_lists = [&](int c) {
        int end[SPEC], n = 0;
#pragma unroll
        for (int j = 0; j < SPEC; ++j) {
            if (j < c) n += ctl.nprom[ctl.ord[j]];
            end[j] = n;
        }
        for (int off = 0; off < n; off += 32) {
            const int t = off + lane;
            int j = 0, base = 0;
#pragma unroll
            for (int x = 0; x + 1 < SPEC; ++x)
                if (t >= end[x]) { j = x + 1; base = end[x]; }
            __syncwarp();
            if (t < n) {
                const uint64_t key = prom[ctl.ord[j] * TEAM_CAND + t - base];
                ctl.batch[lane] = key;
                *vis_slot(key_rank(key)) = key_rank(key);
            }
            __syncwarp();
            merge_ranked<EPL, true>(pool, ctl.batch, min(32, n - off), A.ef_s, lane);
        }
    };

    for (int i = blockIdx.x; i < A.nq;) {
        const int q = A.order ? __ldg(A.order + i) : i;
        // ---- per-query set-up ---------------------------------------------------------------
        {
            float* qf = reinterpret_cast<float*>(smem_raw + L::OFF_Q);
            const float* src = A.queries + (size_t)q * A.d;
            for (int c = threadIdx.x; c < A.q_len; c += W * 32) qf[c] = c < A.d ? __ldg(src + c) : 0.f;
            for (int c = threadIdx.x; c < L::POOL; c += W * 32) pool[c] = KEY_EMPTY;
            const uint4 e4 = make_uint4(HASH_EMPTY, HASH_EMPTY, HASH_EMPTY, HASH_EMPTY);
            for (int c = threadIdx.x; c < (1 << A.hash_bits) / 4; c += W * 32) reinterpret_cast<uint4*>(vis)[c] = e4;
            for (int c = threadIdx.x; c < (SPEC << DEDUP_BITS) / 4; c += W * 32) reinterpret_cast<uint4*>(dedup)[c] = e4;
            if (threadIdx.x < SPEC) {
                ctl.u[threadIdx.x] = BOT;
                ctl.ord[threadIdx.x] = threadIdx.x;
                ctl.nprom[threadIdx.x] = 0;
            }
        }
        const int32_t lo = __ldg(A.lo + q), hi = __ldg(A.hi + q);
        int l_q, r_q;
        if (A.ranges) {
            const int2 lr = __ldg(A.ranges + q);
            l_q = lr.x;
            r_q = lr.y;
        } else {
            warp_rank_interval(A.sorted_attr, A.n, lo, hi, lane, l_q, r_q);    // Sec. 4
        }
        const int w = (lo > hi) ? 0 : (r_q - l_q + 1);
        uint32_t st = 0;
        __syncthreads();

        if (w <= 0) {
            st |= FROG_ST_EMPTY;
        } else if (w <= A.exact_w) {
            // every valid object is evaluated, the pool keeps the ef_s nearest: exact answer
            st |= FROG_ST_EXACT;
            for (int b0 = 0; b0 < w; b0 += SPEC * TEAM_CAND) {
                const int cnt = min(SPEC * TEAM_CAND, w - b0);
                for (int c = threadIdx.x; c < cnt; c += W * 32) cand[c] = (uint32_t)(l_q + b0 + c);
                if (threadIdx.x < SPEC) {
                    ctl.ncand[threadIdx.x] = max(0, min(TEAM_CAND, cnt - (int)threadIdx.x * TEAM_CAND));
                    ctl.nprom[threadIdx.x] = 0;
                }
                __syncthreads();
                distances((1 << SPEC) - 1, 1u, 0, 0);
                __syncthreads();
                if (warp == 0) merge_lists(SPEC);
                __syncthreads();
            }
        } else {
            int L_start, L_end;
            hotspot_layers(l_q, r_q, A.H, A.n, L_start, L_end);          // Alg. 2 line 1
            if (A.no_hotspot) { L_start = 0; L_end = A.H - 1; }
            const int total = (L_end - L_start + 1) * A.m;
            const uint32_t span = (uint32_t)(r_q - l_q);
            int n_exp = 0;                                               // kept by warp 0
            if (warp == 0) {                                             // lines 2-5
                const uint32_t ep = entry_point(A.seed, (uint32_t)l_q, (uint32_t)r_q, lane);
                const bool keep = lane < A.epn && atomicExch(dd_slot(0, ep), ep) != ep;
                const uint32_t M = __ballot_sync(FULL, keep);
                if (keep) cand[__popc(M & lt_mask)] = ep;
                if (lane == 0) {
                    ctl.ncand[0] = __popc(M);
                    ctl.fill_mask = 1;
                    ctl.n_top = 0;                                       // nothing to expand yet
                    ctl.best[0] = 0xFFFFFFFFu;
                }
            }
            __syncthreads();
            for (;;) {
                distances(ctl.fill_mask, 0u, L_start, total);
                __syncthreads();
                if (warp == 0) {
                    // lines 7-17 for as many of the prepared vertices as come next in any case: the j-th
                    // is the first unexpanded one after its predecessors' merges if all of their new
                    // keys lie behind it
                    const int n_top = ctl.n_top;
                    int c = 1;                                           // the entry points' list
                    if (n_top > 0) {
                        bool next = lane < n_top;
                        const uint64_t mine = ctl.key[lane < SPEC ? lane : 0];
#pragma unroll
                        for (int j = 0; j + 1 < SPEC; ++j)
                            next = next && (j >= lane || ctl.best[ctl.ord[j]] > (uint32_t)(mine >> 32));
                        c = min(__ffs(~__ballot_sync(FULL, next)) - 1, A.max_iters - n_exp);
                        if (lane < c) {
                            pool[ctl.pos[lane]] = mine | 1ull;           // line 9
                            ctl.u[ctl.ord[lane]] = BOT;
                        }
                        n_exp += c;
                    }
                    __syncwarp();
                    merge_lists(c);
                    // the first SPEC unexpanded vertices; those not prepared yet take free slots
                    int have = 0;
                    for (int e = 0; e < EPL && have < SPEC; ++e) {
                        const uint64_t key = pool[lane + 32 * e];
                        const bool open = key != KEY_EMPTY && !(key & 1ull);
                        const uint32_t M = __ballot_sync(FULL, open);
                        const int at = have + __popc(M & lt_mask);
                        if (open && at < SPEC) {
                            ctl.key[at] = key;
                            ctl.pos[at] = lane + 32 * e;
                        }
                        have += __popc(M);
                    }
                    have = min(have, SPEC);
                    __syncwarp();
                    const uint32_t want = lane < have ? key_rank(ctl.key[lane]) : BOT;
                    int slot = -1;
#pragma unroll
                    for (int s = 0; s < SPEC; ++s)
                        if (ctl.u[s] == want) slot = s;
                    const bool fresh = lane < have && slot < 0;
                    uint32_t spare = ~__reduce_or_sync(FULL, lane < have && slot >= 0 ? 1u << slot : 0u);
                    const int r = __popc(__ballot_sync(FULL, fresh) & lt_mask);
                    if (fresh) {
                        for (int x = 0; x < r; ++x) spare &= spare - 1;
                        slot = __ffs(spare) - 1;
                        ctl.u[slot] = want;
                        ctl.ncand[slot] = 0;
                        ctl.nprom[slot] = 0;
                        ctl.best[slot] = 0xFFFFFFFFu;
                    }
                    if (lane < have) ctl.ord[lane] = slot;
                    const uint32_t fill = __reduce_or_sync(FULL, fresh ? 1u << slot : 0u);
                    const bool cap = have > 0 && n_exp >= A.max_iters;
                    if (cap) st |= FROG_ST_ITER_CAP;
                    if (lane == 0) {
                        ctl.n_top = have;
                        ctl.fill_mask = (int)fill;
                        ctl.done = have == 0 || cap;
                    }
                }
                __syncthreads();
                if (ctl.done) break;
                // line 10, Alg. 4 over rows L_start..L_end of ENC(u): 256 entries per round trip, a share of
                // them per warp of the slot, admission under budget B across them in order; lines 12-13: what
                // the visited table still knows, and repeats inside the list, are dropped
                constexpr int WPS = W >= SPEC ? W / SPEC : 1;            // warps per slot
                constexpr int CH = 8 / WPS;                              // 32-entry chunks per warp and trip
                const int fill_mask = ctl.fill_mask;
                const int part = W >= SPEC ? warp / SPEC : 0;
                for (int s = warp % SPEC; s < SPEC; s += W) {
                    if (!((fill_mask >> s) & 1)) continue;
                    const uint32_t* hot = A.enc + ((size_t)ctl.u[s] * A.H + L_start) * A.m;
                    const uint4 e4 = make_uint4(HASH_EMPTY, HASH_EMPTY, HASH_EMPTY, HASH_EMPTY);
                    for (int c = lane + 32 * part; c < (1 << DEDUP_BITS) / 4; c += 32 * WPS)
                        reinterpret_cast<uint4*>(dedup + (s << DEDUP_BITS))[c] = e4;
                    auto slot_sync = [&]() {
                        if (WPS == 1) __syncwarp();
                        else asm volatile("bar.sync %0, %1;" ::"r"(s + 1), "n"(32 * WPS) : "memory");
                    };
                    int cnt = 0;
                    for (int c0 = 0; c0 < total && cnt < A.B; c0 += 256) {
                        uint32_t v[CH], M[CH];
                        const int b0 = c0 + 32 * CH * part;
#pragma unroll
                        for (int c = 0; c < CH; ++c) v[c] = b0 + 32 * c + lane < total ? __ldg(hot + b0 + 32 * c + lane) : BOT;
                        int sum = 0;
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            M[c] = __ballot_sync(FULL, (v[c] - (uint32_t)l_q) <= span);
                            sum += __popc(M[c]);
                        }
                        int rank = cnt;
                        if (WPS > 1) {
                            if (lane == 0) ctl.part[s][part] = sum;
                            slot_sync();
#pragma unroll
                            for (int x = 0; x < WPS; ++x) {
                                const int y = ctl.part[s][x];
                                if (x < part) rank += y;
                                cnt += y;
                            }
                        } else {
                            slot_sync();
                            cnt += sum;
                        }
                        uint32_t seen[CH];
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            if (!((M[c] >> lane) & 1u) || rank + __popc(M[c] & lt_mask) >= A.B) v[c] = BOT;
                            rank += __popc(M[c]);
                            seen[c] = v[c] != BOT ? *vis_slot(v[c]) : BOT;
                        }
#pragma unroll
                        for (int c = 0; c < CH; ++c)
                            if (v[c] != seen[c]) seen[c] = atomicExch(dd_slot(s, v[c]), v[c]);
                        int kept = 0;
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            M[c] = __ballot_sync(FULL, v[c] != seen[c]);
                            kept += __popc(M[c]);
                        }
                        int at = 0;
                        if (lane == 0 && kept) at = atomicAdd(&ctl.ncand[s], kept);
                        at = __shfl_sync(FULL, at, 0);
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            if (v[c] != seen[c]) cand[s * TEAM_CAND + at + __popc(M[c] & lt_mask)] = v[c];
                            at += __popc(M[c]);
                        }
                        if (c0 + 256 < total) slot_sync();               // the counts are read before they change
                    }
                }
                __syncthreads();
            }
        }

        // ---- line 18: first k of the pool ---------------------------------------------------
        __syncthreads();
        int got = 0;
        for (int j = threadIdx.x; j < A.k; j += W * 32) {
            const uint64_t key = pool[j];
            int32_t oid = -1;
            float dist = __int_as_float(0x7F800000);
            if (key != KEY_EMPTY) {
                oid = __ldg(A.rank2id + key_rank(key));
                dist = __fsqrt_rn(key_dist2(key));
            }
            A.out_ids[(size_t)q * A.k + j] = oid;
            A.out_dists[(size_t)q * A.k + j] = dist;
        }
        if (A.status && warp == 0) {
            for (int j = lane; j < A.k; j += 32) got += pool[j] != KEY_EMPTY ? 1 : 0;
            got = __reduce_add_sync(FULL, got);
            if (got < A.k) st |= FROG_ST_SHORT;
            if (lane == 0) A.status[q] = st;
        }
        // ---- next query: the first gridDim.x of them are handed out by block index --------------
        if ((int)gridDim.x >= A.nq) break;
        if (threadIdx.x == 0) ctl.next_q = (int)gridDim.x + (int)atomicAdd(A.work_counter, 1u);
        __syncthreads();
        i = ctl.next_q;
        __syncthreads();
    }
}

template <int W, bool F16>
frog_kernel_fn team_pick(int ef_s, int q_len, int vis_bits, size_t* smem) {
    constexpr int SPEC = TEAM_SPEC;
    if (ef_s <= 32) { *smem = TeamLayout<1, SPEC>::bytes(q_len, vis_bits); return frog_search_team_kernel<1, W, SPEC, F16>; }
    if (ef_s <= 64) { *smem = TeamLayout<2, SPEC>::bytes(q_len, vis_bits); return frog_search_team_kernel<2, W, SPEC, F16>; }
    if (ef_s <= 128) { *smem = TeamLayout<4, SPEC>::bytes(q_len, vis_bits); return frog_search_team_kernel<4, W, SPEC, F16>; }
    if (ef_s <= 256) { *smem = TeamLayout<8, SPEC>::bytes(q_len, vis_bits); return frog_search_team_kernel<8, W, SPEC, F16>; }
    *smem = TeamLayout<16, SPEC>::bytes(q_len, vis_bits);
    return frog_search_team_kernel<16, W, SPEC, F16>;
}

}  // namespace

namespace froghost {

frog_kernel_fn team_kernel(int warps, int ef_s, int q_len, int vis_bits, bool f16, size_t* smem) {
    if (warps == 16) return f16 ? team_pick<16, true>(ef_s, q_len, vis_bits, smem) : team_pick<16, false>(ef_s, q_len, vis_bits, smem);
    if (warps == 8) return f16 ? team_pick<8, true>(ef_s, q_len, vis_bits, smem) : team_pick<8, false>(ef_s, q_len, vis_bits, smem);
    return f16 ? team_pick<4, true>(ef_s, q_len, vis_bits, smem) : team_pick<4, false>(ef_s, q_len, vis_bits, smem);
}

}  // namespace froghost
