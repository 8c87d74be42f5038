// Alg. 1 for few queries over wide rows, and the layered search: one block of several warps per query.
//
// With one warp per query a handful of queries leaves the GPU idle while each search is one long chain, and at
// 768 coordinates most of it is the neighbours' rows, read a few at a time. Here the first warp of a block (the
// leader) keeps the pool, picks the vertex to expand and filters its neighbours, all warps form the distances of
// their share of them at once (every load of an expansion in flight together), and the leader inserts them; it
// also reads the adjacency row of the entry that will be expanded next if no nearer vertex turns
// up. The pool, the order of expansions and every distance are those of beam_search. Inverse norms
// (cosine) are formed from the rows as they are read, with the additions of k_inv_norms, instead of from a pass
// over the whole base set, and BF16 rows need no FP32 copy (92 and 70 of the 1,412 us of 100 queries over 100,000
// rows of d = 768, now 376). Layers above the graph (HNSW) are descended in the same launch, their
// vectors read through the layer's member list. Bound by the chain of an expansion: adjacency row, rows (two
// rounds of loads), butterflies, insertion: 4 us.
#include "k_beam.cuh"

namespace fgim {

// Sums of up to four rows (wide rows: four chunks of every row, 16 loads, in flight); lane r < U gets row r's
// sum in the canonical order and, SELF, the row's own squared norm in that order.
template <int METRIC, typename RT, bool SELF>
__device__ __forceinline__ float rows_few(const RT* __restrict__ base, const int32_t* rid, int U, const Query& Q, int d,
                                          int lane, float& self) {
    const int nc4 = d >> 2;
    const RT* rowp[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) rowp[t] = base + (long long)rid[t < U ? t : 0] * d;
    float acc[4][4], own[4][4];
#pragma unroll
    for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[t][i] = own[t][i] = 0.f;
#pragma unroll (sizeof(RT) == 2 ? 6 : 4)
    for (int c = lane; c < nc4; c += 32) {
        const float4 x = reinterpret_cast<const float4*>(Q.q)[c];
        float4 y[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) y[t] = t < U ? row_chunk(rowp[t], c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            if (METRIC == FGIM_L2SQ) {
                const float e0 = __fsub_rn(x.x, y[t].x), e1 = __fsub_rn(x.y, y[t].y);
                const float e2 = __fsub_rn(x.z, y[t].z), e3 = __fsub_rn(x.w, y[t].w);
                acc[t][0] = fmaf(e0, e0, acc[t][0]);
                acc[t][1] = fmaf(e1, e1, acc[t][1]);
                acc[t][2] = fmaf(e2, e2, acc[t][2]);
                acc[t][3] = fmaf(e3, e3, acc[t][3]);
            } else {
                acc[t][0] = fmaf(x.x, y[t].x, acc[t][0]);
                acc[t][1] = fmaf(x.y, y[t].y, acc[t][1]);
                acc[t][2] = fmaf(x.z, y[t].z, acc[t][2]);
                acc[t][3] = fmaf(x.w, y[t].w, acc[t][3]);
            }
            if (SELF) {
                own[t][0] = fmaf(y[t].x, y[t].x, own[t][0]);
                own[t][1] = fmaf(y[t].y, y[t].y, own[t][1]);
                own[t][2] = fmaf(y[t].z, y[t].z, own[t][2]);
                own[t][3] = fmaf(y[t].w, y[t].w, own[t][3]);
            }
        }
    }
    float mine = 0.f;
    self = 0.f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float v = warp_butterfly(__fadd_rn(__fadd_rn(acc[t][0], acc[t][1]), __fadd_rn(acc[t][2], acc[t][3])));
        if (lane == t) mine = v;
        if (SELF) {
            const float o = warp_butterfly(__fadd_rn(__fadd_rn(own[t][0], own[t][1]), __fadd_rn(own[t][2], own[t][3])));
            if (lane == t) self = o;
        }
    }
    return mine;
}

// the same for rows of up to 128 coordinates (one chunk per lane)
template <int METRIC, typename RT, bool SELF>
__device__ __forceinline__ float rows_few_small(const RT* __restrict__ base, const int32_t* rid, int U, float4 q, int d,
                                                int lane, float& self) {
    const bool has = lane < (d >> 2);
    float4 y[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        y[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < U && has) y[t] = row_chunk(base + (long long)rid[t] * d, lane);
    }
    float mine = 0.f;
    self = 0.f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float v = warp_butterfly(has ? chunk_part<METRIC>(q, y[t]) : 0.f);
        if (lane == t) mine = v;
        if (SELF) {
            const float o = warp_butterfly(chunk_part<FGIM_IP>(y[t], y[t]));
            if (lane == t) self = o;
        }
    }
    return mine;
}

__device__ __forceinline__ float inv_norm_of(float s) { return s > 0.f ? __fdiv_rn(1.f, __fsqrt_rn(s)) : 0.f; }

// shared memory of a block: the pool and table of its query, the rows of an expansion, and the query itself
struct TeamLayout {
    int pool, ht, rid, dist, ctl, q, bytes;
};
__host__ __device__ inline TeamLayout team_layout(int d, int L, int htbits) {
    TeamLayout t;
    int o = 0;
    t.pool = o;
    o += pool_entries(L) * 8;
    t.ht = o;
    o += (1 << htbits) * 2;
    t.rid = o;
    o += 32 * 4;
    t.dist = o;
    o += 32 * 4;
    t.ctl = o;
    o += 16;
    t.q = o;
    o += align16(d * 4);
    t.bytes = o;
    return t;
}

struct TeamSmem {
    uint64_t* pool;
    uint16_t* ht;
    int32_t* rid;     // rows of the expansion (row numbers of the base)
    float* dist;      // their distances
    int* ctl;         // [0] their number, or -1: the search is over; [1] the result
    const float* q;
};

// Distances of rid[0 .. U) into dist by all warps of the block (a contiguous share each).
template <int METRIC, bool SMALLD, typename RT>
__device__ __forceinline__ void team_delta(const RT* __restrict__ X, const float* __restrict__ inv_norm,
                                           const TeamSmem& S, int U, float qinv, int d, int warp, int nw, int lane) {
    constexpr bool SELF = METRIC == FGIM_COSINE;
    const int per = (U + nw - 1) / nw;
    const int r1 = min(U, (warp + 1) * per);
    Query Q;
    Q.q = S.q;
    const float4 qc = SMALLD && lane < (d >> 2) ? reinterpret_cast<const float4*>(S.q)[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = warp * per; r0 < r1; r0 += 4) {
        const int n = min(4, r1 - r0);
        float self;
        float dd;
        if constexpr (SMALLD) dd = rows_few_small<METRIC, RT, SELF>(X, S.rid + r0, n, qc, d, lane, self);
        else dd = rows_few<METRIC, RT, SELF>(X, S.rid + r0, n, Q, d, lane, self);
        if (lane < n) {
            float inv = 1.f;
            if (METRIC == FGIM_COSINE) inv = __fmul_rn(qinv, inv_norm ? inv_norm[S.rid[r0 + lane]] : inv_norm_of(self));
            S.dist[r0 + lane] = delta_finish<METRIC>(dd, inv);
        }
    }
}

// Alg. 1 over one graph of nt vertices by the whole block; vertex v's row is X[members ? members[v] : v]. Leaves the
// pool (keys with the local ids) in S.pool and returns its size to every warp.
template <int METRIC, bool SMALLD, typename RT, int MAXS>
__device__ __forceinline__ int team_search(const RT* __restrict__ X, const int32_t* __restrict__ members, long long nbase,
                                           const float* __restrict__ inv_norm, const int32_t* __restrict__ adj, int M, int nt, int ep,
                                           const TeamSmem& S, float qinv, int d, int L, int htbits, WarpCounters& ctr,
                                           int* status) {
    const int lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const VisitedHash H(nt, htbits);
    const int hop_budget = status[1];
    const unsigned budget = hop_budget > 0 ? (unsigned)hop_budget : (unsigned)nt + 1u;
    uint64_t pk[MAXS];
    unsigned it = 0, ndc = 0;
    // the leader's place in the current adjacency row, the local ids of the rows handed out (one per lane), and the
    // adjacency chunk read ahead for vertex ahead_u
    int u = -1, c0 = 0, U = 0, mine = -1, ahead_u = -1, ahead = -1;
    if (warp == 0) {
        ht_clear(S.ht, htbits, lane);
#pragma unroll
        for (int s = 0; s < MAXS; ++s) {
            pk[s] = kEmptyKey;
            S.pool[32 * s + lane] = kEmptyKey;
        }
        __syncwarp();
        const bool bad = ep < 0 || ep >= nt || L < 1 || L > 32 * MAXS;
        if (bad && lane == 0) atomicOr(status, kErrBounds);
        if (!bad) {   // the entry is the first row to be evaluated
            U = 1;
            if (lane == 0) {
                mine = ep;
                H.add(S.ht, ep);
            }
        } else {
            U = -1;
        }
    }
    for (;;) {
        if (warp == 0) {
            while (U == 0) {   // the next neighbours to evaluate
                if (u >= 0) {
                    c0 += 32;
                    if (c0 >= M) u = -1;
                }
                if (u < 0) {
                    int slot, src;
                    uint32_t lo;
                    u = pool_next<MAXS>(pk, slot, src, lo);
                    if (u < 0 || it >= budget) {
                        if (u >= 0 && lane == 0) atomicOr(status, kErrTimeout);
                        U = -1;
                        break;
                    }
                    if (lane == src) {
#pragma unroll
                        for (int s = 0; s < MAXS; ++s)
                            if (slot == s) pk[s] |= 1ull;
                        reinterpret_cast<uint32_t*>(S.pool)[2 * (32 * slot + lane)] = lo | 1u;
                    }
                    ++it;
                    c0 = 0;
                }
                const int32_t* row = adj + (long long)u * M;
                int v = c0 == 0 && u == ahead_u ? ahead : c0 + lane < M ? row[c0 + lane] : -1;
                if (v >= nt) {
                    atomicOr(status, kErrBounds);
                    v = -1;
                }
                const unsigned same = __match_any_sync(kFull, v);   // a neighbour listed twice is evaluated once
                if ((same & lt) != 0u) v = -1;
                if (v >= 0 && H.seen(S.ht, v)) v = -1;
                const unsigned m = __ballot_sync(kFull, v >= 0);
                U = __popc(m);
                if (U == 0) continue;
                if (v >= 0) S.rid[__popc(m & lt)] = v;   // lane r takes the r-th of them
                __syncwarp();
                mine = lane < U ? S.rid[lane] : -1;
                __syncwarp();
                int sl, sr;   // read ahead the row of the next entry in line
                uint32_t lw;
                ahead_u = pool_next<MAXS>(pk, sl, sr, lw);
                if (ahead_u >= 0) ahead = lane < M ? adj[(long long)ahead_u * M + lane] : -1;
            }
            if (lane < U) {
                int r = members ? members[mine] : mine;
                if (r < 0 || r >= nbase) {
                    atomicOr(status, kErrBounds);
                    r = 0;
                }
                S.rid[lane] = r;
            }
            if (lane == 0) S.ctl[0] = U;
        }
        __syncthreads();
        const int n = S.ctl[0];
        if (n < 0) break;
        team_delta<METRIC, SMALLD, RT>(X, inv_norm, S, n, qinv, d, warp, nw, lane);
        __syncthreads();
        if (warp == 0) {
            ndc += (unsigned)n;
            const uint64_t cand = lane < n ? mkkey(S.dist[lane], (int32_t)((uint32_t)mine << 1)) : kEmptyKey;
            U = 0;
            pool_insert<MAXS>(pk, S.pool, cand, L, lane);
        }
    }
    if (warp == 0) {
        ctr.ndc += ndc;
        ctr.hops += it;
        int n = 0;
#pragma unroll
        for (int s = 0; s < MAXS; ++s) {
            n += __popc(__ballot_sync(kFull, pk[s] != kEmptyKey));
            if (pk[s] != kEmptyKey) S.pool[32 * s + lane] = (pk[s] & 0xffffffff00000000ull) | ((uint32_t)pk[s] >> 1);
        }
        if (lane == 0) S.ctl[1] = n;
    }
    __syncthreads();
    const int n = S.ctl[1];
    return n;
}

template <int METRIC, bool SMALLD, typename RT, int MAXS>
__global__ void __launch_bounds__(kTeamThreads, SMALLD ? 4 : 2) k_search_team(
    const RT* __restrict__ X, const float* __restrict__ inv_norm, long long n, int d, const int32_t* __restrict__ graph,
    int R, int entry, const int32_t* __restrict__ qentry, TeamLayers layers, int ef_up, const RT* __restrict__ Q,
    const int32_t* __restrict__ qids, int topk, int L, int htbits, int32_t* __restrict__ out_ids, float* __restrict__ out_dist, int32_t* __restrict__ out_start,
    unsigned long long* counters, int* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const long long qi = blockIdx.x;
    const TeamLayout lay = team_layout(d, L > ef_up ? L : ef_up, htbits);
    TeamSmem S;
    S.pool = reinterpret_cast<uint64_t*>(smem + lay.pool);
    S.ht = reinterpret_cast<uint16_t*>(smem + lay.ht);
    S.rid = reinterpret_cast<int32_t*>(smem + lay.rid);
    S.dist = reinterpret_cast<float*>(smem + lay.dist);
    S.ctl = reinterpret_cast<int*>(smem + lay.ctl);
    float* q = reinterpret_cast<float*>(smem + lay.q);
    S.q = q;
    const RT* qrow = qids ? X + (long long)qids[qi] * d : Q + qi * d;
    for (int c = threadIdx.x; c < (d >> 2); c += blockDim.x) reinterpret_cast<float4*>(q)[c] = row_chunk(qrow, c);
    __syncthreads();
    float qinv = 1.f;
    if (METRIC == FGIM_COSINE) {   // every warp forms it for itself
        const float4* q4 = reinterpret_cast<const float4*>(q);
        qinv = inv_norm_of(warp_butterfly(lane_part<FGIM_IP>(q4, q4, d >> 2, lane)));
    }
    WarpCounters ctr;
    int start = qentry ? qentry[qi] : entry;
    for (int l = 0; l < layers.count; ++l) {   // from the top layer down: its nearest vertex starts the next
        const TeamLayer ly = layers.l[l];
        int lo = 0, hi = ly.n;   // the start's position in the layer
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ly.members[mid] < start) lo = mid + 1;
            else hi = mid;
        }
        if (lo >= ly.n || ly.members[lo] != start) {
            if (threadIdx.x == 0) atomicOr(status, kErrBounds);
            lo = 0;
        }
        const int np = team_search<METRIC, SMALLD, RT, MAXS>(X, ly.members, n, nullptr, ly.adj, ly.M, ly.n, lo, S, qinv, d, ef_up,
                                                             htbits, ctr, status);
        if (np > 0) {
            const int32_t g = ly.members[key_id(S.pool[0])];
            if (g >= 0 && g < n) start = g;
        }
        __syncthreads();   // the pool has been read
    }
    if (out_start && threadIdx.x == 0) out_start[qi] = start;
    const int np = team_search<METRIC, SMALLD, RT, MAXS>(X, nullptr, n, inv_norm, graph, R, (int)n, start, S, qinv, d, L, htbits,
                                                         ctr, status);
    for (int s = threadIdx.x; s < topk; s += blockDim.x) {
        out_ids[qi * topk + s] = s < np ? key_id(S.pool[s]) : -1;
        out_dist[qi * topk + s] = s < np ? key_dist(S.pool[s]) : __int_as_float(0x7f800000);
    }
    if (warp == 0) warp_add_counters(ctr, counters);
}

cudaError_t launch_search_team(const void* X, bool bf16, const float* inv_norm, long long n, int d, int metric,
                               const int32_t* graph, int R, int entry, const int32_t* qentry, const TeamLayers& layers,
                               int ef_up, const void* Q, const int32_t* qids, long long nq, int topk, int L, int32_t* out_ids,
                               float* out_dist, int32_t* out_start, unsigned long long* counters, int* status,
                               cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int Lp = L > ef_up ? L : ef_up;
    const int htbits = ht_bits_for(Lp);
    const size_t smem = (size_t)team_layout(d, Lp, htbits).bytes;
    const int threads = nq <= kTeamWide ? kTeamThreads : kTeamThreads / 2;
    cudaError_t e = cudaSuccess;
#define FGIM_LAUNCH_T(MT, SD, RT, MS)                                                                              \
    do {                                                                                                           \
        e = allow_smem(k_search_team<MT, SD, RT, MS>, smem); \
        if (e != cudaSuccess) break;                                                                               \
        LaunchScope ls("k_search", s);                                                                             \
        k_search_team<MT, SD, RT, MS><<<(unsigned)nq, threads, smem, s>>>(                                    \
            static_cast<const RT*>(X), inv_norm, n, d, graph, R, entry, qentry, layers, ef_up, static_cast<const RT*>(Q),  \
            qids, topk, L, htbits, out_ids, out_dist, out_start, counters, status);                                \
        e = cudaGetLastError();                                                                                    \
    } while (0)
    if (bf16) FGIM_DISPATCH_ALL_WIDE(metric, Lp, FGIM_LAUNCH_T, uint16_t);
    else FGIM_DISPATCH_ALL(metric, d, Lp, FGIM_LAUNCH_T, float);
#undef FGIM_LAUNCH_T
    return e;
}

}  // namespace fgim
