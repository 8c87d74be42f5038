// Input proximity graphs on the GPU: the batch-incremental insertion the synthetic workloads use
// for their input indexes (one flat HNSW-style graph per shard), built from the library's own
// Alg. 1 search and neighbour-selection kernels.
//
// The insertion order starts with the medoid (the row nearest, in FP64 squared L2, to the FP64
// mean of the rows; the lowest id on ties), then every other row in id order. Rows are inserted
// in batches of b = min(max(c / 2, 1), 1024) rows once c rows are in: every row of a batch
// searches the graph as it stood when the batch started (Alg. 1 from the medoid with pool ef,
// the same search HNSW's two-heap layer search performs), keeps up to M of the results with
// HNSW's heuristic (a candidate is dropped when a kept one is strictly nearer to it than the
// inserted row: the MRNG rule, no indegree clause), and gets that list; then every vertex that
// received reverse edges takes its list and the new edges, in ascending (distance, id), keeps
// all of them when they are at most M and otherwise the heuristic's M. The mean and the medoid
// distances are summed in the same sequential FP64 order as a plain loop, so the medoid is that
// of the plain loop bit for bit.
#include <cstddef>

#include "fgim_launch.h"

namespace fgim {

static inline long long cdivp(long long a, long long b) { return (a + b - 1) / b; }

// x as FP64 by its bits (exact), for zero and normal x; other exponents: false
__device__ __forceinline__ bool widens(float x) {
    const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
    return u == 0u || (u >= 0x00800000u && u < 0x7f800000u);
}
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7fffffffu;
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + (m ? 0x38000000u : 0u))), (int)(u << 29));
}

// mean[t] = (sum over rows i, in order, of X[i][t]) / n, in FP64. One lane per dimension, one warp per 32: a chain of
// n additions, bound by their latency (54 ns a row, whatever the lanes per warp), so the next kMeanRows rows are read
// while the current ones are added, and the values are widened by their bits: the conversion shares the FP64 pipe
// (60,000 rows of d = 96: 4.15 ms converted, 3.2 ms so; 250,000 of d = 128: 20.3 and 13.4).
constexpr int kMeanRows = 32;
__global__ void __launch_bounds__(32) k_col_mean(const float* __restrict__ X, long long n, int d, double* __restrict__ mean) {
    const int t = blockIdx.x * 32 + threadIdx.x;
    if (t >= d) return;
    const float* p = X + t;
    float cur[kMeanRows], nxt[kMeanRows];
    double s = 0.0;
    const long long full = n / kMeanRows;
    if (full > 0) {
#pragma unroll
        for (int r = 0; r < kMeanRows; ++r) cur[r] = p[(long long)r * d];
    }
    for (long long b = 0; b < full; ++b) {
        p += (long long)kMeanRows * d;
        if (b + 1 < full) {
#pragma unroll
            for (int r = 0; r < kMeanRows; ++r) nxt[r] = p[(long long)r * d];
        }
        bool bits = true;
#pragma unroll
        for (int r = 0; r < kMeanRows; ++r) bits = bits && widens(cur[r]);
        if (bits) {
#pragma unroll
            for (int r = 0; r < kMeanRows; ++r) s = __dadd_rn(s, widen(cur[r]));
        } else {
#pragma unroll
            for (int r = 0; r < kMeanRows; ++r) s = __dadd_rn(s, (double)cur[r]);
        }
#pragma unroll
        for (int r = 0; r < kMeanRows; ++r) cur[r] = nxt[r];
    }
    for (long long i = full * kMeanRows; i < n; ++i) s = __dadd_rn(s, (double)X[i * d + t]);
    mean[t] = __ddiv_rn(s, (double)n);
}

// The same from byte rows: every partial sum is an integer below 255 n < 2^39, exact in FP64, so the sum over any
// order is the sequential one's. Block (x, y): 32 dimensions, rows y * rows ..; sums[t] += its part.
__global__ void __launch_bounds__(256) k_col_sums_u8(const uint8_t* __restrict__ X8, long long n, int d, long long rows,
                                                     unsigned long long* __restrict__ sums) {
    __shared__ unsigned long long part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * 32 + lane;
    const long long r0 = blockIdx.y * rows, r1 = min(n, r0 + rows);
    unsigned long long s = 0;
    if (t < d)
#pragma unroll 8
        for (long long i = r0 + warp; i < r1; i += 8) s += X8[i * d + t];
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && t < d) {
        for (int w = 1; w < 8; ++w) s += part[w][lane];
        atomicAdd(sums + t, s);
    }
}

__global__ void k_col_mean_u8(const unsigned long long* __restrict__ sums, long long n, int d, double* __restrict__ mean) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < d) mean[t] = __ddiv_rn((double)sums[t], (double)n);
}

// squared FP64 distance of every row to the mean (sequential over the dimensions), the smallest
// one's bits (non-negative doubles order like their bits) folded into *best
__global__ void k_medoid_dist(const float* __restrict__ X, long long n, int d, const double* __restrict__ mean,
                              unsigned long long* __restrict__ dist_bits, unsigned long long* best) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double a = 0.0;
    for (int t = 0; t < d; ++t) {
        const double z = __dsub_rn((double)X[i * d + t], mean[t]);
        a = __dadd_rn(a, __dmul_rn(z, z));
    }
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    dist_bits[i] = b;
    atomicMin(best, b);
}

// the lowest row at the smallest distance
__global__ void k_medoid_pick(const unsigned long long* __restrict__ dist_bits, long long n,
                              const unsigned long long* best, int* medoid) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && dist_bits[i] == *best) atomicMin(medoid, (int)i);
}

// insertion order: the medoid, then every other row in id order; and the empty graph
__global__ void k_pg_init(long long n, int M, const int* medoid, int32_t* __restrict__ order,
                          int32_t* __restrict__ nbr, float* __restrict__ nd, int32_t* __restrict__ cnt,
                          int32_t* __restrict__ zeros, int32_t* __restrict__ cin, int32_t* __restrict__ fill) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int m = *medoid;
    if (i < n) {
        order[i] = i == 0 ? m : (i - 1 < m ? (int32_t)(i - 1) : (int32_t)i);
        cnt[i] = 0;
        zeros[i] = 0;
        cin[i] = 0;
        fill[i] = 0;
    }
    if (i < n * M) {
        nbr[i] = -1;
        nd[i] = __int_as_float(0x7f800000);
    }
}

// The reverse edges of a batch are grouped by target without a pass over all n vertices (two prefix sums, a
// compaction and two fills over n took seven launches and a host read per batch): the first edge to a
// vertex puts it in the list of targets, every target takes its segment of rev from a counter, and the merge
// leaves cin and fill zero for the next batch. The order of targets and segments is arbitrary; a target's keys
// are put in order when they are merged.
struct PgCounters {   // of one batch, zeroed before it
    int targets, edges, overflow;
};

// the batch's lists go in; their entries become reverse-edge candidates of their targets
__global__ void k_pg_install(const int32_t* __restrict__ rows, long long b, int M, const int32_t* __restrict__ e_ids,
                             const float* __restrict__ e_dist, const int32_t* __restrict__ e_cnt,
                             int32_t* __restrict__ nbr, float* __restrict__ nd, int32_t* __restrict__ cnt,
                             int32_t* __restrict__ cin, int32_t* __restrict__ targets, PgCounters* ctr) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= b * M) return;
    const long long bi = i / M;
    const int t = (int)(i - bi * M);
    const int32_t p = rows[bi];
    const int c = e_cnt[bi];
    if (t == 0) cnt[p] = c;
    nbr[(long long)p * M + t] = t < c ? e_ids[i] : -1;
    nd[(long long)p * M + t] = t < c ? e_dist[i] : __int_as_float(0x7f800000);
    if (t < c && atomicAdd(cin + e_ids[i], 1) == 0) targets[atomicAdd(&ctr->targets, 1)] = e_ids[i];
}

__global__ void k_pg_segments(const int32_t* __restrict__ targets, const int32_t* __restrict__ cin,
                              int32_t* __restrict__ off, PgCounters* ctr) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ctr->targets) return;
    off[targets[i]] = atomicAdd(&ctr->edges, cin[targets[i]]);
}

__global__ void k_pg_rev_fill(const int32_t* __restrict__ rows, long long b, int M, const int32_t* __restrict__ e_ids,
                              const float* __restrict__ e_dist, const int32_t* __restrict__ e_cnt,
                              const int32_t* __restrict__ off, int32_t* __restrict__ fill,
                              uint64_t* __restrict__ rev) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= b * M) return;
    const long long bi = i / M;
    const int t = (int)(i - bi * M);
    if (t >= e_cnt[bi]) return;
    const int32_t v = e_ids[i];
    rev[off[v] + atomicAdd(fill + v, 1)] = mkkey(e_dist[i], rows[bi]);
}

constexpr int kMergeCap = 128;   // the longest list warp_merge can hold

// Per target v (warp per target): its list and its new reverse edges in ascending (distance, id);
// at most M of them stay as they are, more go to the overflow lists for the heuristic.
__global__ void __launch_bounds__(128) k_pg_rev_merge(const int32_t* __restrict__ targets,
                                                      const int32_t* __restrict__ off, int32_t* __restrict__ cin,
                                                      int32_t* __restrict__ fill,
                                                      const uint64_t* __restrict__ rev, int M, int W,
                                                      int32_t* __restrict__ nbr, float* __restrict__ nd,
                                                      int32_t* __restrict__ cnt, int32_t* __restrict__ ov_ids,
                                                      float* __restrict__ ov_dist, int32_t* __restrict__ ov_tgt,
                                                      PgCounters* ctr) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = lane_id();
    const long long ti = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (ti >= ctr->targets) return;
    const int32_t v = targets[ti];
    uint64_t* list = reinterpret_cast<uint64_t*>(smem) + (size_t)warp * W;
    const int c0 = cnt[v];
    const long long b0 = off[v], m = cin[v];
    __syncwarp();
    if (lane == 0) cin[v] = fill[v] = 0;
    if (c0 + m > kMergeCap) {
        // a hub: more keys than a merged list may hold (the keys are distinct and at most W, more than M):
        // each key's place is the number of smaller ones, written straight to the overflow list
        const int total = (int)(c0 + m);
        for (int s = lane; s < total; s += 32)
            list[s] = s < c0 ? mkkey(nd[(long long)v * M + s], nbr[(long long)v * M + s]) : rev[b0 + (s - c0)];
        __syncwarp();
        int slot = 0;
        if (lane == 0) slot = atomicAdd(&ctr->overflow, 1);
        slot = __shfl_sync(kFull, slot, 0);
        for (int s = lane; s < total; s += 32) {
            const uint64_t key = list[s];
            int r = 0;
            for (int q = 0; q < total; ++q) r += list[q] < key ? 1 : 0;
            ov_ids[(long long)slot * W + r] = key_id(key);
            ov_dist[(long long)slot * W + r] = key_dist(key);
        }
        for (int s = total + lane; s < W; s += 32) {
            ov_ids[(long long)slot * W + s] = -1;
            ov_dist[(long long)slot * W + s] = __int_as_float(0x7f800000);
        }
        if (lane == 0) ov_tgt[slot] = v;
        return;
    }
    int n = 0;
    for (int s0 = 0; s0 < c0; s0 += 32) {
        const uint64_t key = s0 + lane < c0 ? mkkey(nd[(long long)v * M + s0 + lane], nbr[(long long)v * M + s0 + lane])
                                            : kEmptyKey;
        n = warp_merge<false>(list, nullptr, n, W, key, 0);
    }
    for (long long s0 = 0; s0 < m; s0 += 32) {
        const uint64_t key = s0 + lane < m ? rev[b0 + s0 + lane] : kEmptyKey;
        n = warp_merge<false>(list, nullptr, n, W, key, 0);
    }
    if (n <= M) {
        for (int s = lane; s < M; s += 32) {
            nbr[(long long)v * M + s] = s < n ? key_id(list[s]) : -1;
            nd[(long long)v * M + s] = s < n ? key_dist(list[s]) : __int_as_float(0x7f800000);
        }
        if (lane == 0) cnt[v] = n;
        return;
    }
    int slot = 0;
    if (lane == 0) slot = atomicAdd(&ctr->overflow, 1);
    slot = __shfl_sync(kFull, slot, 0);
    for (int s = lane; s < W; s += 32) {
        ov_ids[(long long)slot * W + s] = s < n ? key_id(list[s]) : -1;
        ov_dist[(long long)slot * W + s] = s < n ? key_dist(list[s]) : __int_as_float(0x7f800000);
    }
    if (lane == 0) ov_tgt[slot] = v;
}

// the heuristic's lists of the overflowing targets back into the graph
__global__ void k_pg_write_back(const int32_t* __restrict__ ov_tgt, long long nov, int M,
                                const int32_t* __restrict__ e_ids, const float* __restrict__ e_dist,
                                const int32_t* __restrict__ e_cnt, int32_t* __restrict__ nbr, float* __restrict__ nd,
                                int32_t* __restrict__ cnt) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nov * M) return;
    const long long r = i / M;
    const int t = (int)(i - r * M);
    const int32_t v = ov_tgt[r];
    if (t == 0) cnt[v] = e_cnt[r];
    nbr[(long long)v * M + t] = e_ids[i];
    nd[(long long)v * M + t] = e_dist[i];
}

cudaError_t launch_pg_medoid(const float* X, const uint8_t* X8, long long n, int d, double* mean, unsigned long long* dist_bits,
                             unsigned long long* best, int* medoid, cudaStream_t s) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(best, 0xff, sizeof(unsigned long long), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(medoid, 0x7f, sizeof(int), s)) != cudaSuccess) return e;
    if (X8) {   // the sums stand where the distances go afterwards (dist_bits has room for n and for d of them)
        if ((e = cudaMemsetAsync(dist_bits, 0, sizeof(unsigned long long) * d, s)) != cudaSuccess) return e;
        const long long rows = std::max(512LL, cdivp(n, 4096));
        {
            LaunchScope ls("k_col_sums_u8", s);
            k_col_sums_u8<<<dim3((unsigned)cdivp(d, 32), (unsigned)cdivp(n, rows)), 256, 0, s>>>(X8, n, d, rows, dist_bits);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        LaunchScope ls("k_col_mean", s);
        k_col_mean_u8<<<(unsigned)cdivp(d, 128), 128, 0, s>>>(dist_bits, n, d, mean);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else {
        LaunchScope ls("k_col_mean", s);
        k_col_mean<<<(unsigned)cdivp(d, 32), 32, 0, s>>>(X, n, d, mean);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls("k_medoid_dist", s);
        k_medoid_dist<<<(unsigned)cdivp(n, 256), 256, 0, s>>>(X, n, d, mean, dist_bits, best);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    LaunchScope ls("k_medoid_pick", s);
    k_medoid_pick<<<(unsigned)cdivp(n, 256), 256, 0, s>>>(dist_bits, n, best, medoid);
    return cudaGetLastError();
}

cudaError_t launch_pg_init(long long n, int M, const int* medoid, int32_t* order, int32_t* nbr, float* nd, int32_t* cnt,
                           int32_t* zeros, int32_t* cin, int32_t* fill, cudaStream_t s) {
    LaunchScope ls("k_pg_init", s);
    k_pg_init<<<(unsigned)cdivp(n * M, 256), 256, 0, s>>>(n, M, medoid, order, nbr, nd, cnt, zeros, cin, fill);
    return cudaGetLastError();
}

// The batch's lists into the graph, and its reverse edges into their targets' lists; counters (kPgCounters ints)
// [kPgOverflow] becomes the number of overflow lists.
cudaError_t launch_pg_edges(const int32_t* rows, long long b, int M, const int32_t* e_ids, const float* e_dist,
                            const int32_t* e_cnt, int32_t* nbr, float* nd, int32_t* cnt, int32_t* cin, int32_t* fill,
                            int32_t* off, int32_t* targets, uint64_t* rev, int32_t* ov_ids, float* ov_dist,
                            int32_t* ov_tgt, int* counters, cudaStream_t s) {
    static_assert(sizeof(PgCounters) == kPgCounters * sizeof(int) && offsetof(PgCounters, overflow) == kPgOverflow * sizeof(int));
    PgCounters* ctr = reinterpret_cast<PgCounters*>(counters);
    cudaError_t e = cudaMemsetAsync(ctr, 0, sizeof(PgCounters), s);
    if (e != cudaSuccess) return e;
    const long long edges = b * M;   // no more targets than edges
    const unsigned blocks = (unsigned)cdivp(edges, 256);
    {
        LaunchScope ls("k_pg_install", s);
        k_pg_install<<<blocks, 256, 0, s>>>(rows, b, M, e_ids, e_dist, e_cnt, nbr, nd, cnt, cin, targets, ctr);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls("k_pg_segments", s);
        k_pg_segments<<<blocks, 256, 0, s>>>(targets, cin, off, ctr);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    {
        LaunchScope ls("k_pg_rev_fill", s);
        k_pg_rev_fill<<<blocks, 256, 0, s>>>(rows, b, M, e_ids, e_dist, e_cnt, off, fill, rev);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int wpb = 4, W = M + (int)b;
    const size_t smem = (size_t)wpb * W * 8;
    if ((e = allow_smem(k_pg_rev_merge, smem)) != cudaSuccess)
        return e;
    LaunchScope ls("k_pg_rev_merge", s);
    k_pg_rev_merge<<<(unsigned)cdivp(edges, wpb), wpb * 32, smem, s>>>(targets, off, cin, fill, rev, M, W, nbr, nd, cnt,
                                                                      ov_ids, ov_dist, ov_tgt, ctr);
    return cudaGetLastError();
}

cudaError_t launch_pg_write_back(const int32_t* ov_tgt, long long nov, int M, const int32_t* e_ids, const float* e_dist,
                                 const int32_t* e_cnt, int32_t* nbr, float* nd, int32_t* cnt, cudaStream_t s) {
    if (nov <= 0) return cudaSuccess;
    LaunchScope ls("k_pg_write_back", s);
    k_pg_write_back<<<(unsigned)cdivp(nov * M, 256), 256, 0, s>>>(ov_tgt, nov, M, e_ids, e_dist, e_cnt, nbr, nd, cnt);
    return cudaGetLastError();
}

}  // namespace fgim
