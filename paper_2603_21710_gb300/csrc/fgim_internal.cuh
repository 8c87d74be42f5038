// Internal device and host helpers of the FGIM CUDA library (sm_103a).
//
// Keys. Every list, pool and candidate set orders entries by (distance, global id).
// Both are packed in one 64-bit key: the high word is the distance's IEEE bits mapped
// to an order-preserving unsigned integer, the low word the id. Key order equals the
// lexicographic (distance, id) order for every non-NaN distance.
//
// Distance. One definition gives every distance that enters a list or decides a
// comparison (the canonical FP32 distance). The d dimensions form float4 chunks
// c = 0 .. d/4-1; lane l of a warp owns the chunks c = l, l+32, l+64, ... and adds them
// in increasing c into four accumulators s_j += e_j * e_j with e = a - b (fused
// multiply-add; inner product: s_j += a_j * b_j), its partial is (s0 + s1) + (s2 + s3);
// the 32 partials are summed by a butterfly over lane offsets 16, 8, 4, 2, 1. Inner
// product gives 1 - sum, cosine 1 - sum * (inv_a * inv_b). Every step is a single
// rounded operation whose operands are symmetric in a and b, so delta(a, b) equals
// delta(b, a) bit for bit, and the same (id, distance) pair always yields the same key.
// Warps compute it one row at a time (butterfly) or several rows at a time, eight lanes per row or
// the rows' partials exchanged together (the same sums, added in the same tree).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/fgim.h"

namespace fgim {

constexpr uint32_t kFull = 0xffffffffu;
constexpr uint64_t kEmptyKey = ~0ull;
constexpr int kMaxShards = FGIM_MAX_SHARDS;

// Every call passes its kernels a device status array int[4]: status[0] collects the error
// bits below; status[1] is the beam searches' expansion budget (0 = unbounded), set only by
// the "hop_budget" test hook; status[2] is scratch for one host read (the adjacency check).
// device status word bits
constexpr int kErrOverflow = 1;   // a bounded buffer overflowed (handled by the host)
constexpr int kErrBounds = 2;     // an index failed a bounds check (the access was skipped)
constexpr int kErrTimeout = 4;    // a bounded wait ran out

// The input shards of one merge, or of a batch of independent merges run as one problem over
// the disjoint union of their vertices (fgim_merge_batch): the shards of merge m are the
// consecutive range grp[i] .. gend[i] - 1 of every shard i of m, and the cross query of a vertex
// of shard i searches the other shards of that range with the pool gL[i] (its merge's L).
constexpr int kMaxTableShards = 512;
struct ShardTable {
    int h;                               // shards in the table
    int dim;
    long long off[kMaxTableShards + 1];  // first global id of every shard
    const int32_t* adj[kMaxTableShards];
    int M[kMaxTableShards];
    int entry[kMaxTableShards];          // local entry of every input PG
    int grp[kMaxTableShards];            // first shard of the shard's merge
    int gend[kMaxTableShards];           // one past the last shard of the shard's merge
    int gL[kMaxTableShards];             // cross-query pool of the shard's merge
};

__host__ __device__ inline uint32_t f2ord(float f) {
#ifdef __CUDA_ARCH__
    uint32_t u = __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, 4);
#endif
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__host__ __device__ inline float ord2f(uint32_t o) {
    uint32_t u = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}

__host__ __device__ inline uint64_t mkkey(float d, int32_t id) {
    return ((uint64_t)f2ord(d) << 32) | (uint32_t)id;
}
__host__ __device__ inline int32_t key_id(uint64_t k) { return (int32_t)(uint32_t)(k & 0xffffffffu); }
__host__ __device__ inline float key_dist(uint64_t k) { return ord2f((uint32_t)(k >> 32)); }

__device__ __forceinline__ int shard_of(const ShardTable& t, long long g) {
    int lo = 0, hi = t.h - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (g >= t.off[mid]) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Neighbour-selection rule of Alg. 5 (Sec. 4.3.1 names RNG, MRNG and tau-MNG as interchangeable;
// fgim_params.prune_rule). u is the vertex, w a kept neighbour, v the candidate; duv, duw, dwv
// their squared-type distances. Every rule also keeps v when T(v) = 1 (checked by the caller).
//   0 alpha-RNG: w occludes v iff alpha^2 dwv >= duv (product rounded once in FP32);
//   1 MRNG (NSG's edge selection): w occludes v iff dwv < duv;
//   2 tau-MNG: on the metric distances sqrt(delta), w occludes v iff sqrt(duw) < sqrt(duv) and
//     sqrt(dwv) < sqrt(duv) - 3 tau; in FP32: t = sqrt(duv) - 3tau, occluded iff t > 0,
//     duw < duv and dwv < t * t (every operation a single correctly rounded one).
struct PruneRule {
    int kind;
    float alpha2;   // alpha^2 rounded once to FP32 (alpha-RNG)
    float tau3;     // 3 tau rounded once to FP32 (tau-MNG)
};

// MRNG and tau-MNG: w occludes v iff dwv < rule_thr(duv) (tau-MNG also needs duw < duv); -inf
// when no distance is below it.
__device__ __forceinline__ float rule_thr(const PruneRule& r, float duv) {
    if (r.kind == 1) return duv;
    const float t = __fsub_rn(__fsqrt_rn(duv), r.tau3);
    return t > 0.f ? __fmul_rn(t, t) : __int_as_float(0xff800000);
}

__device__ __forceinline__ bool rule_occludes(const PruneRule& r, float duv, float duw, float dwv) {
    if (r.kind == 0) return !(duv < __fmul_rn(r.alpha2, dwv));
    if (r.kind == 2 && !(duw < duv)) return false;
    return dwv < rule_thr(r, duv);
}

// Byte rows: the vectors stored as one byte per coordinate, used when every coordinate is an
// integer in [0, 255] and d <= 128, d % 16 == 0 (distances are then exact integers below 2^24).
__host__ __device__ inline bool byte_rows_ok(int d) { return d % 16 == 0 && d <= 128; }

// lanes per byte row: 16-byte chunks per row rounded up to a power of two (d <= 128)
__device__ __forceinline__ int byte_lanes(int d) {
    const int c16 = d >> 4;
    return c16 <= 1 ? 1 : c16 <= 2 ? 2 : c16 <= 4 ? 4 : 8;
}
// i / n for 0 <= i; 32-bit unsigned division when i fits (the usual case of per-entry grids
// over N x R or N x k entries), else 64-bit
__device__ __forceinline__ long long div_idx(long long i, int n) {
    return i < 0x100000000LL ? (long long)((uint32_t)i / (uint32_t)n) : i / n;
}
// log2 of byte_lanes(d)
__device__ __forceinline__ int byte_lanes_log2(int d) {
    const int c16 = d >> 4;
    return c16 <= 1 ? 0 : c16 <= 2 ? 1 : c16 <= 4 ? 2 : 3;
}
// sum of v over the 2^lsh lanes of this lane's row group (lsh <= 3)
__device__ __forceinline__ uint32_t row_group_sum(uint32_t v, int lsh) {
#pragma unroll
    for (int b = 0; b < 3; ++b)
        if (b < lsh) v += __shfl_xor_sync(0xffffffffu, v, 1 << b);
    return v;
}

// ----------------------------------------------------------------------------
// canonical distance (see the file comment); rows are 16-byte aligned float4 arrays
// ----------------------------------------------------------------------------
template <int METRIC>
__device__ __forceinline__ float lane_part(const float4* __restrict__ a, const float4* __restrict__ b, int nc4,
                                           int lane) {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    for (int c = lane; c < nc4; c += 32) {
        const float4 x = a[c];
        const float4 y = b[c];
        if (METRIC == FGIM_L2SQ) {
            const float e0 = __fsub_rn(x.x, y.x), e1 = __fsub_rn(x.y, y.y);
            const float e2 = __fsub_rn(x.z, y.z), e3 = __fsub_rn(x.w, y.w);
            s0 = fmaf(e0, e0, s0);
            s1 = fmaf(e1, e1, s1);
            s2 = fmaf(e2, e2, s2);
            s3 = fmaf(e3, e3, s3);
        } else {
            s0 = fmaf(x.x, y.x, s0);
            s1 = fmaf(x.y, y.y, s1);
            s2 = fmaf(x.z, y.z, s2);
            s3 = fmaf(x.w, y.w, s3);
        }
    }
    return __fadd_rn(__fadd_rn(s0, s1), __fadd_rn(s2, s3));
}

// the lane partial for one float4 chunk per lane (d = 128), as lane_part computes it
template <int METRIC>
__device__ __forceinline__ float chunk_part(const float4 x, const float4 y) {
    float s0, s1, s2, s3;
    if (METRIC == FGIM_L2SQ) {
        const float e0 = __fsub_rn(x.x, y.x), e1 = __fsub_rn(x.y, y.y);
        const float e2 = __fsub_rn(x.z, y.z), e3 = __fsub_rn(x.w, y.w);
        s0 = fmaf(e0, e0, 0.f);
        s1 = fmaf(e1, e1, 0.f);
        s2 = fmaf(e2, e2, 0.f);
        s3 = fmaf(e3, e3, 0.f);
    } else {
        s0 = fmaf(x.x, y.x, 0.f);
        s1 = fmaf(x.y, y.y, 0.f);
        s2 = fmaf(x.z, y.z, 0.f);
        s3 = fmaf(x.w, y.w, 0.f);
    }
    return __fadd_rn(__fadd_rn(s0, s1), __fadd_rn(s2, s3));
}

template <int METRIC>
__device__ __forceinline__ float delta_finish(float s, float inv_ab) {
    if (METRIC == FGIM_L2SQ) return s;
    if (METRIC == FGIM_IP) return __fsub_rn(1.f, s);
    return __fsub_rn(1.f, __fmul_rn(s, inv_ab));
}

// butterfly sum of one value per lane; every lane gets the same result
__device__ __forceinline__ float warp_butterfly(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// rounding margin between two FP32 evaluations of the same distance that both follow
// sums of at most d/4 + 8 terms per chain: the worst-case relative error of either is
// below (d/4 + 8) * 2^-24 of the sum of |terms| (Higham, Accuracy and Stability of
// Numerical Algorithms, 2nd ed., Sec. 3.1), so they differ by less than twice that.
__host__ __device__ inline float fp32_pair_margin(int d) { return 2.f * (float)(d / 4 + 8) * 5.9604645e-8f; }

// ----------------------------------------------------------------------------
// warp helpers
// ----------------------------------------------------------------------------
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
    lo = __shfl_sync(kFull, lo, src);
    hi = __shfl_sync(kFull, hi, src);
    return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ uint64_t shfl_xor64(uint64_t v, int m) {
    uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
    lo = __shfl_xor_sync(kFull, lo, m);
    hi = __shfl_xor_sync(kFull, hi, m);
    return ((uint64_t)hi << 32) | lo;
}

// ascending bitonic sort of one 64-bit key per lane across the warp
__device__ __forceinline__ uint64_t warp_sort32(uint64_t v) {
    const int lane = lane_id();
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            uint64_t o = shfl_xor64(v, stride);
            bool up = ((lane & size) == 0);
            bool lower = ((lane & stride) == 0);
            uint64_t mn = v < o ? v : o;
            uint64_t mx = v < o ? o : v;
            v = (up == lower) ? mn : mx;
        }
    }
    return v;
}

// Merge one candidate key per lane (kEmptyKey = none) into a sorted list of at most
// `cap` keys held in shared memory, keeping the `cap` smallest. `aux` (optional) is a
// byte that travels with each list entry; every candidate of one call enters with the
// same `cand_aux`. Duplicates are removed by id: a candidate whose id is already in
// the list is dropped (the list copy wins), and among lanes offering the same id only
// the smallest key survives. BY_ID = false checks list membership by key equality,
// which is exact when every copy of an id carries the same key (canonical distances).
// Called by all 32 lanes with identical n, cap and cand_aux; cap <= 128. Returns the
// new list size.
template <bool BY_ID>
__device__ int warp_merge(uint64_t* list, uint8_t* aux, int n, int cap, uint64_t cand, uint8_t cand_aux) {
    const int lane = lane_id();
    bool valid = cand != kEmptyKey;
    if (valid && n >= cap && cand >= list[cap - 1]) valid = false;
    if (!__any_sync(kFull, valid)) return n;   // nothing can enter the list
    if (valid) {
        if (BY_ID) {
            const int32_t cid = key_id(cand);
            for (int t = 0; t < n; ++t)
                if (key_id(list[t]) == cid) { valid = false; break; }
        } else {
            int lo = 0, hi = n;
            while (lo < hi) {
                int mid = (lo + hi) >> 1;
                if (list[mid] < cand) lo = mid + 1;
                else hi = mid;
            }
            if (lo < n && list[lo] == cand) valid = false;
        }
    }
    // duplicates among lanes: keep the smallest key of each id (lowest lane on equal keys)
    {
        const int32_t cid = valid ? key_id(cand) : -1 - lane;
        const unsigned grp = __match_any_sync(kFull, cid);
        if (__any_sync(kFull, valid && __popc(grp) > 1)) {
            for (int src = 0; src < 32; ++src) {
                uint64_t ok = shfl64(cand, src);
                if (valid && ((grp >> src) & 1u) && src != lane && (ok < cand || (ok == cand && src < lane)))
                    valid = false;
            }
        }
    }
    const uint64_t sorted = warp_sort32(valid ? cand : kEmptyKey);
    const int m = __popc(__ballot_sync(kFull, sorted != kEmptyKey));
    if (m == 0) return n;
    // final position of every list entry: its index plus the candidates below it
    const int per = (n + 31) >> 5;
    uint64_t lk[4];
    uint8_t la[4];
    int lpos[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        lk[r] = kEmptyKey;
        la[r] = 0;
        lpos[r] = cap;
        if (r < per) {
            const int i = lane + 32 * r;
            const bool act = i < n;
            if (act) {
                lk[r] = list[i];
                la[r] = aux ? aux[i] : (uint8_t)0;
            }
            int lo = 0, hi = m;
#pragma unroll
            for (int step = 0; step < 6; ++step) {
                const int mid = (lo + hi) >> 1;
                const uint64_t mk = shfl64(sorted, mid < 31 ? mid : 31);
                if (lo < hi) {
                    if (mk < lk[r]) lo = mid + 1;
                    else hi = mid;
                }
            }
            if (act) lpos[r] = i + lo;
        }
    }
    // final position of every candidate: its rank plus the list entries below it
    int cpos = cap;
    if (lane < m) {
        int lo = 0, hi = n;
        while (lo < hi) {
            int mid = (lo + hi) >> 1;
            if (list[mid] < sorted) lo = mid + 1;
            else hi = mid;
        }
        cpos = lane + lo;
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (lpos[r] < cap) {
            list[lpos[r]] = lk[r];
            if (aux) aux[lpos[r]] = la[r];
        }
    }
    if (cpos < cap) {
        list[cpos] = sorted;
        if (aux) aux[cpos] = cand_aux;
    }
    __syncwarp();
    const int nn = n + m;
    return nn < cap ? nn : cap;
}

// ----------------------------------------------------------------------------
// host-side launch accounting (defined in fgim_abi.cu)
// ----------------------------------------------------------------------------
struct LaunchScope {
    const char* name;
    cudaStream_t stream;
    cudaEvent_t e0, e1;
    bool timed;
    LaunchScope(const char* n, cudaStream_t s);
    ~LaunchScope();
};

}  // namespace fgim
