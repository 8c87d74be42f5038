// Host-side launchers of the FGIM kernels (one declaration per kernel family).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fgim_internal.cuh"

namespace fgim {

// a call's counters[kItemCounter]: the items a beam-search launch has handed out to its warps (zeroed by the launch)
constexpr int kItemCounter = 8;

// ---- k_search.cu
// X: FP32 rows; X8: the same rows as bytes when every coordinate is an integer in [0, 255]
// (searches then read X8, with identical results), else nullptr
// phi / src (optional): the ID mapping with invalid vertices; nq = the number of output rows
// (valid vertices), src[r] = the input row of output row r, phi maps input rows to output ids
// (-1 = dropped)
cudaError_t launch_cross_query(const ShardTable& t, const float* X, const uint8_t* X8, const float* inv_norm,
                               long long N, int metric, int k, int L, fgim_knng* out, unsigned long long* counters,
                               int* status, cudaStream_t s, const int32_t* phi = nullptr,
                               const int32_t* src = nullptr, long long nq = -1, const uint16_t* Xh = nullptr);
cudaError_t launch_search(const float* X, const uint8_t* X8, const float* inv_norm, long long n, int d, int metric,
                          const int32_t* graph, int R, int entry, const float* Q, const float* q_inv,
                          const int32_t* qids, long long nq, int topk, int L, int32_t* out_ids, float* out_dist,
                          unsigned long long* counters, int* status, cudaStream_t s, const uint16_t* Xh = nullptr,
                          const int32_t* qentry = nullptr);
// ---- k_team.cu: one block per query (few queries). X and Q: FP32 rows, or BF16 ones (bf16: d > 128,
// 8-byte aligned); Q == nullptr: queries are the rows qids of X; inv_norm == nullptr (cosine): formed from the rows.
// layers: the non-empty HNSW layers, top first (count 0: the search starts at `entry`), searched with pool ef_up
constexpr int kTeamThreads = 256;            // half of them above kTeamWide queries
constexpr long long kTeamWide = 304;         // two blocks per SM
// Queries up to which a block each is faster than a warp each. Wide rows (100k, d = 768 BF16, cosine): 100
// queries 0.74 -> 0.33 ms, 300: 0.69 -> 0.38, 1,000: 0.73 and 0.69 (and the FP32 d = 960 form slower). Rows of up to
// 128 coordinates: never (one query 0.122 and 0.132 ms, 1,000: 0.26 and 0.31): there the leader's own steps
// are the chain. With HNSW layers the single launch counts (a warp each, a launch per layer, against a block each; pool
// 64, layers' pool 8): 1,000 queries of 100k d = 96 0.345 -> 0.254 ms, 60k d = 768 BF16 0.735 -> 0.615, 60k d = 960
// 1.183 -> 1.117, 100k d = 132 0.589 -> 0.506; 1,216 queries 0.336 -> 0.255, 0.742 -> 0.642, 1.186 -> 1.230, 0.631 ->
// 0.628. With pool 128 (layers' pool 32) wide rows cross earlier: 1,000 queries 1.005 -> 1.119 (d = 768), 0.793 -> 0.922
// (d = 132), 2.078 -> 1.702 (d = 960), d = 96 0.503 -> 0.453; one line serves all.
constexpr long long kTeamQueries = 608;
constexpr long long kTeamLayered = 1216;
struct TeamLayer {
    const int32_t* members;
    const int32_t* adj;
    int n;
    int M;
};
struct TeamLayers {
    TeamLayer l[FGIM_MAX_LEVELS];
    int count;
};
cudaError_t launch_search_team(const void* X, bool bf16, const float* inv_norm, long long n, int d, int metric,
                               const int32_t* graph, int R, int entry, const int32_t* qentry, const TeamLayers& layers,
                               int ef_up, const void* Q, const int32_t* qids, long long nq, int topk, int L, int32_t* out_ids,
                               float* out_dist, int32_t* out_start, unsigned long long* counters, int* status,
                               cudaStream_t s);
// X8[i] = X[i] as a byte; *flag |= 1 unless every X[i] is an integer in [0, 255] (n_elems % 4 == 0)
cudaError_t launch_narrow_u8(const float* X, long long n_elems, uint8_t* X8, int* flag, cudaStream_t s);

// Lets launches of `kernel` ask for `smem` bytes of dynamic shared memory. The limit belongs to the kernel, not to the
// launch, so a call must not set it to its own size: a call of another thread may stand between its setting and its launch,
// and a smaller limit would make that launch fail. Every call that needs more than the default (48 KB) sets the
// same value, the most a block can have; the others leave the limit alone.
template <typename K>
cudaError_t allow_smem(K kernel, size_t smem) {
    constexpr size_t kByDefault = 47 * 1024;   // beside up to 1 KB of static shared memory
    if (smem <= kByDefault) return cudaSuccess;
    int dev = 0, most = 0;
    cudaFuncAttributes a;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess) return e;
    most -= (int)a.sharedSizeBytes;
    if (smem > (size_t)most) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// the grid of a cooperative launch: `want` blocks, at most as many as are resident at once (the grid-wide
// barriers wait for all of them)
template <typename K>
cudaError_t coop_grid(K kernel, int threads, long long want, int* blocks) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    const long long most = (long long)per_sm * sms;
    *blocks = (int)(want < 1 ? 1 : want < most ? want : most);
    return cudaSuccess;
}

// Rounds that commit a prefix of a window (indegree repair, reachability fix): blocks of 16 warps, so that a
// full window has a warp per item in at most 128 blocks (a grid-wide barrier costs less the fewer blocks
// arrive: the 1M merge's reachability rounds 11.4 ms with 512 blocks of 4 warps, 7.4 ms so, 7.9 ms with 64 blocks
// of 32); the next round looks at four times the items the last one committed, within [256, most] (what
// lies past the first conflict is planned for nothing). The window changes no result.
constexpr int kRoundThreads = 512;
__device__ __forceinline__ long long round_window(long long committed, long long most) {
    const long long w = 4 * committed;
    return w < 256 ? 256 : w < most ? w : most;
}

// ---- k_util.cu
// exclusive scan of n int32 counts into n + 1 int64 offsets (out[n] = total)
cudaError_t scan_counts(const int32_t* in, long long n, long long* out, void* scratch, size_t scratch_bytes,
                        cudaStream_t s);
cudaError_t scan_counts2(const int32_t* in0, const int32_t* in1, long long n, long long* out0, long long* out1,
                         void* scratch, size_t scratch_bytes, cudaStream_t s);   // two arrays of n at once
size_t scan_scratch_bytes(long long n);
cudaError_t scan_local_bytes(size_t* bytes);   // local memory per thread of the scan kernels (test hook)
cudaError_t launch_inv_norms(const float* X, long long n, int d, float* inv, cudaStream_t s);
// the same of BF16 rows (8-byte aligned), without an FP32 copy
cudaError_t launch_inv_norms_bf16(const uint16_t* X, long long n, int d, float* inv, cudaStream_t s);
// out[i] = the FP32 value of the bfloat16 encoding in[i]
cudaError_t launch_bf16_to_f32(const uint16_t* in, long long n, float* out, cudaStream_t s);
// flag[i] = (mask == nullptr || mask[i] != 0)
cudaError_t launch_valid_flags(const uint8_t* mask, long long n, int32_t* flag, cudaStream_t s);
// phi[i] = flag[i] ? off[i] : -1 (off = exclusive prefix sums of flag)
cudaError_t launch_phi(const int32_t* flag, const long long* off, long long n, int32_t* phi, cudaStream_t s);
// out[r] = X[src[r]] for r < nv (rows of d floats)
cudaError_t launch_gather_rows(const float* X, const int32_t* src, long long nv, int d, float* out, cudaStream_t s);
// indices i (ascending) with flag[i] != 0, written to out; count to *count (device)
cudaError_t compact_flags(const int32_t* flag, long long n, int32_t* out, long long* offsets_scratch,
                          void* scan_scratch, size_t scan_bytes, cudaStream_t s);

// ---- k_refine.cu
struct RefineBuffers {
    // reverse lists
    int32_t* cntN;            // cntN, cntO, fillN, fillO: one block of 4 N
    int32_t* cntO;
    int32_t* fillN;
    int32_t* fillO;
    long long* offN;
    long long* offO;
    uint64_t* revN;
    uint64_t* revO;
    long long rev_capacity;   // entries of revN / revO (N * k each)
    int32_t* topN;            // [N, rev_cap]
    int32_t* topO;
    int32_t* ntopN;
    int32_t* ntopO;
    // candidate sets
    int32_t* cand;            // [N, cmax]
    int32_t* nn;
    int32_t* no;
    int cmax;
    // proposals
    int32_t* prop_tgt;
    uint64_t* prop_key;
    long long prop_cap;
    unsigned long long* prop_count;   // device counter
    uint64_t* prop_sorted;
    int32_t* pcnt;            // proposals per target (counted by the join), pcnt and pfill: one block of 2 N
    int32_t* pfill;
    long long* poff;
    uint8_t* pending;
    int32_t* pend_flag;
    int32_t* pend_list;
    long long* pend_off;
    // scan scratch
    void* scan_tmp;
    size_t scan_bytes;
    // largest candidate set and C_n of a pass and the four launch lists' sizes and largest
    // sets (device, 10 ints), a pinned host slot to read them, and the launch lists (4 x cap)
    int32_t* max_nc;
    int32_t* host_i32;
    long long class_count[5];   // out of refine_join: vertices per form (TC <= 64, <= 128, > 128; FP32 tile;
                                // warp per vertex)
    uint64_t* wk;               // worst key of every list (filled by refine_join for the Update launches)
    int sparse_nn;              // vertices with |C_n| <= sparse_nn (and |C| <= 128) join one warp each
                                // (byte rows; 0: never)
    bool fp8;                   // Xb holds E4M3 rows with per-vector scales (tcm.w) instead of 16-bit ones
    int32_t* blist;
    long long blist_cap;
    // tensor-core filter inputs: BF16, FP16 (f16) or E4M3 (fp8) copy of the vectors, rows of dp >= dim
    // values, and per row (|x|^2, bound on |x|, bound on the conversion error, value of one unit)
    int join_filter;
    void* Xb;
    float4* tcm;
    int dp;
    bool f16;
    // the vectors as bytes when every coordinate is an integer in [0, 255], else nullptr
    const uint8_t* X8;
};

cudaError_t rev_select_local_bytes(size_t* bytes);   // local memory per thread of k_rev_select (test hook)
cudaError_t refine_visit(const fgim_knng& g, int rev_cap, RefineBuffers& b, cudaStream_t s);
cudaError_t refine_join(const ShardTable& t, const float* X, const float* inv_norm, int metric, const fgim_knng& g,
                        RefineBuffers& b, const int32_t* vlist, long long nv, unsigned long long* pairs,
                        unsigned long long* cands, int* status, cudaStream_t s);
cudaError_t refine_merge(const fgim_knng& g, RefineBuffers& b, long long nprop, cudaStream_t s);
cudaError_t launch_prep_fp8(const float* X, long long N, int d, int dp, uint8_t* Xq, float4* tcm, cudaStream_t s);
// the lists for which the E4M3 tile's error bound is too coarse to decide much
cudaError_t launch_fp8_coarse(const fgim_knng& g, const float4* tcm, const float* inv_norm, int metric, int* count,
                              cudaStream_t s);
// *out = some adjacency row of the input graphs repeats an id within a 32-entry chunk (uses
// status[2] as scratch; synchronizes the stream)
cudaError_t adjacency_has_repeats(const ShardTable& t, long long N, int* status, cudaStream_t s, bool* out);
cudaError_t launch_prep_bf16(const float* X, long long N, int d, int dp, void* Xb, float4* tcm, cudaStream_t s);
// *not_bf16 = some coordinate is not a BF16 value
cudaError_t launch_prep_f16(const float* X, long long N, int d, int dp, void* Xb, float4* tcm, int* not_bf16,
                            cudaStream_t s);
cudaError_t launch_indegree(const int32_t* ids, long long N, int k, int32_t* T, bool clear_replaced, uint8_t* flags,
                            cudaStream_t s);
// Alg. 4 for the vertices zeros[0 .. *nz) (ascending), in one cooperative launch; ff: 3 words, plan: scratch of
// kRepairWindow entries, owner [g.n]; *zero_count = *nz
constexpr int kRepairWindow = 2048;
cudaError_t launch_repair(fgim_knng& g, int32_t* T, const int32_t* zeros, const long long* nz, long long* ff,
                          unsigned long long* owner, int4* plan, unsigned long long* repaired,
                          unsigned long long* zero_count, int* status, cudaStream_t s);
cudaError_t launch_zero_flags(const int32_t* T, long long N, int32_t* flag, cudaStream_t s);
cudaError_t launch_nonzero_flags(const uint8_t* v, long long N, int32_t* flag, cudaStream_t s);

// ---- k_select.cu
// Alg. 5 neighbour selection of the g.n lists of g (ids in 0 .. N - 1, rows of X; X8 and Xh: the same
// rows as bytes and as BF16, or nullptr) with `rule`
cudaError_t launch_prune(const float* X, const uint8_t* X8, const uint16_t* Xh, const float* inv_norm, long long N,
                         int d, int metric, const fgim_knng& g, const int32_t* T, int R, PruneRule rule, int32_t* e_ids, float* e_dist,
                         int32_t* e_cnt, int* status, cudaStream_t s);
// ---- k_prune.cu
struct ReverseBuffers {
    int32_t* cnt;
    long long* off;
    int32_t* fill;
    uint64_t* rev;
    void* scan_tmp;
    size_t scan_bytes;
};
cudaError_t launch_reverse_insert(long long N, int R, const int32_t* e_ids, const float* e_dist, const int32_t* e_cnt,
                                  ReverseBuffers& b, int32_t* out_ids, float* out_dist, int32_t* out_deg,
                                  cudaStream_t s);
// batches run as one problem: start[r] = entries[m] of the merge m (id range off[m] .. off[m+1]-1)
// holding reps[r]; the rows of one merge copied out of the union graph, ids minus base
cudaError_t launch_rep_starts(const int32_t* reps, long long nr, const long long* off, const int32_t* entries, int nm,
                              int32_t* start, cudaStream_t s);
cudaError_t launch_split_rows(const int32_t* ids, const float* dist, const int32_t* deg, long long n, int R,
                              int32_t base, int32_t* out_ids, float* out_dist, int32_t* out_deg, cudaStream_t s);
// BFS from `entry` (entries == nullptr) or from the ne sources `entries` (device), in one cooperative launch:
// visited[y] = level (sources 1, unreached 0); fa, fb [N]; st: 8 ints, reached vertices (int64) at st[4]
cudaError_t launch_bfs(const int32_t* graph, int R, long long N, int entry, const int32_t* entries, int ne,
                       int32_t* visited, int32_t* fa, int32_t* fb, int32_t* st, int* status, cudaStream_t s);
cudaError_t launch_bfs_parents(const int32_t* graph, int R, long long N, const int32_t* level, int32_t* npar,
                               cudaStream_t s);
// label[x] = the smallest id of x's weak component among the unreached vertices (-1: reached), in one
// cooperative launch; list [N], st: 4 ints
cudaError_t launch_cc(const int32_t* graph, int R, long long N, const int32_t* visited, int32_t* label, int32_t* list,
                      int32_t* st, cudaStream_t s);
cudaError_t launch_rep_flags(const int32_t* visited, const int32_t* label, long long N, int32_t* flag,
                             cudaStream_t s);
// the attachment of the nr representatives in one cooperative launch; ff: 3 words, ff[0] = 0; plan: scratch of
// kReachWindow entries, owner all ones
constexpr int kReachWindow = 2048;
cudaError_t launch_reach_rounds(int32_t* graph, float* gdist, int32_t* deg, const int32_t* level, int32_t* npar,
                                int R, const int32_t* reps, long long nr, long long* ff, const int32_t* cand,
                                const float* cdist, int beam, unsigned long long* owner, int4* plan,
                                unsigned long long* attached, int* status, cudaStream_t s);

// ---- k_hnsw.cu (HNSW-adaptive merging, Sec. 4.3.3)
constexpr int kMaxHnswLevels = 16;
struct HnswThresholds {   // T_l = floor((2^64 - 1) / M^l), l = 1 .. count
    int count;
    unsigned long long t[kMaxHnswLevels];
};
cudaError_t launch_hnsw_levels(long long n, unsigned long long seed, const HnswThresholds& th, int32_t* levels,
                               cudaStream_t s);
// flag[v] = levels[v] >= level
cudaError_t launch_level_flags(const int32_t* levels, long long n, int level, int32_t* flag, cudaStream_t s);
// rows of width M into rows of width w (padding -1 / +inf)
cudaError_t launch_widen(const int32_t* ids, const float* dist, long long n, int M, int w, int32_t* oids, float* odist,
                         cudaStream_t s);
// the kk nearest rows of every row of Xl among the rows before it (n rows, FP32; X8l: the same
// as bytes or nullptr)
cudaError_t launch_layer_knn(const float* Xl, const uint8_t* X8l, const float* inv, long long n, int d, int metric,
                             int kk, int32_t* out_ids, float* out_dist, cudaStream_t s);
// hand-over between layer searches: best (positions in mem) -> qpos (positions in next) or,
// with next == nullptr, start (global ids); first: every query starts at entry's position
cudaError_t launch_hnsw_next(const int32_t* best, const int32_t* mem, long long nmem, const int32_t* next,
                             long long nnext, long long nq, int first, int entry, int32_t* qpos, int32_t* start,
                             int* status, cudaStream_t s);

// ---- k_pgbuild.cu: input PGs by batch-incremental insertion (see the file comment)
cudaError_t launch_pg_medoid(const float* X, const uint8_t* X8, long long n, int d, double* mean, unsigned long long* dist_bits,
                             unsigned long long* best, int* medoid, cudaStream_t s);
cudaError_t launch_pg_init(long long n, int M, const int* medoid, int32_t* order, int32_t* nbr, float* nd, int32_t* cnt,
                           int32_t* zeros, int32_t* cin, int32_t* fill, cudaStream_t s);
constexpr int kPgCounters = 3, kPgOverflow = 2;   // ints of launch_pg_edges' counters; the overflow lists' number
cudaError_t launch_pg_edges(const int32_t* rows, long long b, int M, const int32_t* e_ids, const float* e_dist,
                            const int32_t* e_cnt, int32_t* nbr, float* nd, int32_t* cnt, int32_t* cin, int32_t* fill,
                            int32_t* off, int32_t* targets, uint64_t* rev, int32_t* ov_ids, float* ov_dist,
                            int32_t* ov_tgt, int* counters, cudaStream_t s);
cudaError_t launch_pg_write_back(const int32_t* ov_tgt, long long nov, int M, const int32_t* e_ids, const float* e_dist,
                                 const int32_t* e_cnt, int32_t* nbr, float* nd, int32_t* cnt, cudaStream_t s);

// ---- fgim_abi.cu: launch shapes chosen by the autotuner (fgim_autotune)
// Beam-search kernels (cross query, searches): warps per block and visited-table bits, keyed by
// (metric, bytes per coordinate read, dim, pool L) on the current device; untuned keys keep the
// defaults passed in. Neither changes a result (the visited table may only forget ids).
unsigned long long beam_shape_key(int metric, int row_bytes, int dim, int L);
void tuned_beam_shape(unsigned long long key, int* wpb, int* htbits);

}  // namespace fgim
