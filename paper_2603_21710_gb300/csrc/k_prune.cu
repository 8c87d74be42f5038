// Stage (c): the connectivity enhancement of Alg. 5 and the reachability fix (the neighbour
// selection is in k_select.cu).
//
// Connectivity enhancement builds the reverse lists of the pruned snapshot E' by a
// counting sort and merges them into E'(u), keeping the R smallest (delta, id).
#include <algorithm>

#include <cooperative_groups.h>

#include "fgim_launch.h"

namespace fgim {

namespace cg = cooperative_groups;

static inline long long cdivl(long long a, long long b) { return (a + b - 1) / b; }

// ---------------------------------------------------------------------------- reverse insertion
__global__ void k_e_count(const int32_t* __restrict__ e_ids, long long total, int32_t* __restrict__ cnt) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int32_t v = e_ids[i];
    if (v >= 0) atomicAdd(cnt + v, 1);
}

__global__ void k_e_fill(const int32_t* __restrict__ e_ids, const float* __restrict__ e_dist, long long total, int R,
                         const long long* __restrict__ off, int32_t* __restrict__ fill, uint64_t* __restrict__ rev) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int32_t v = e_ids[i];
    if (v < 0) return;
    const int p = atomicAdd(fill + v, 1);
    rev[off[v] + p] = mkkey(e_dist[i], (int32_t)div_idx(i, R));
}

__global__ void __launch_bounds__(128) k_e_merge(const int32_t* __restrict__ e_ids, const float* __restrict__ e_dist,
                                                 const int32_t* __restrict__ e_cnt, long long N, int R,
                                                 const long long* __restrict__ off, const uint64_t* __restrict__ rev,
                                                 int32_t* __restrict__ out_ids, float* __restrict__ out_dist,
                                                 int32_t* __restrict__ out_deg) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = lane_id();
    const long long u = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    if (u >= N) return;
    uint64_t* list = reinterpret_cast<uint64_t*>(smem) + (size_t)warp * R;
    const int ne = e_cnt[u];
    for (int s = lane; s < ne; s += 32) list[s] = mkkey(e_dist[u * R + s], e_ids[u * R + s]);
    __syncwarp();
    int n = ne;
    const long long b = off[u], m = off[u + 1] - off[u];
    for (long long c0 = 0; c0 < m; c0 += 32) {
        const uint64_t key = (c0 + lane < m) ? rev[b + c0 + lane] : kEmptyKey;
        n = warp_merge<true>(list, nullptr, n, R, key, 0);
    }
    for (int s = lane; s < R; s += 32) {
        if (s < n) {
            out_ids[u * R + s] = key_id(list[s]);
            out_dist[u * R + s] = key_dist(list[s]);
        } else {
            out_ids[u * R + s] = -1;
            out_dist[u * R + s] = __int_as_float(0x7f800000);
        }
    }
    if (lane == 0) out_deg[u] = n;
}

cudaError_t launch_reverse_insert(long long N, int R, const int32_t* e_ids, const float* e_dist, const int32_t* e_cnt,
                                  ReverseBuffers& b, int32_t* out_ids, float* out_dist, int32_t* out_deg,
                                  cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    const long long total = N * R;
    cudaError_t e;
    if ((e = cudaMemsetAsync(b.cnt, 0, sizeof(int32_t) * N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(b.fill, 0, sizeof(int32_t) * N, s)) != cudaSuccess) return e;
    const unsigned gb = (unsigned)cdivl(total, 256);
    {
        LaunchScope ls("k_e_count", s);
        k_e_count<<<gb, 256, 0, s>>>(e_ids, total, b.cnt);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = scan_counts(b.cnt, N, b.off, b.scan_tmp, b.scan_bytes, s)) != cudaSuccess) return e;
    {
        LaunchScope ls("k_e_fill", s);
        k_e_fill<<<gb, 256, 0, s>>>(e_ids, e_dist, total, R, b.off, b.fill, b.rev);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int wpb = 4;
    LaunchScope ls("k_e_merge", s);
    k_e_merge<<<(unsigned)cdivl(N, wpb), wpb * 32, (size_t)wpb * R * 8, s>>>(e_ids, e_dist, e_cnt, N, R, b.off, b.rev,
                                                                             out_ids, out_dist, out_deg);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- reachability fix
// BFS state: st[0..2] frontier sizes (level L reads st[L % 3], writes st[(L + 1) % 3] and
// clears st[(L + 2) % 3] for the level after), st[4..5] the number of reached vertices (int64).
// All levels in one cooperative launch, a grid-wide barrier per level: the levels are short (a launch each
// and a host read every eight cost 0.3 of the 4.4 ms of a 20,000-vertex merge).
__global__ void __launch_bounds__(512) k_bfs(const int32_t* __restrict__ graph, int R, long long N, int entry,
                                             const int32_t* __restrict__ entries, int ne, int32_t* visited,
                                             int32_t* fa, int32_t* fb, int32_t* st, int* status) {
    cg::grid_group grid = cg::this_grid();
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    const int lane = lane_id();
    for (long long i = tid; i < N; i += nt) visited[i] = 0;
    if (tid == 0) {
        st[0] = st[2] = 0;
        st[1] = entries ? ne : 1;
        *reinterpret_cast<long long*>(st + 4) = entries ? ne : 1;
    }
    grid.sync();
    for (long long i = tid; i < (entries ? ne : 1); i += nt) {
        int32_t e = entries ? entries[i] : entry;
        if (e < 0 || e >= N) {
            atomicOr(status, kErrBounds);
            e = 0;
        }
        visited[e] = 1;
        fa[i] = e;
    }
    grid.sync();
    int sum = 0;
    for (int level = 1; level <= N; ++level) {
        const long long work = (long long)__ldcg(st + level % 3) * R;
        if (work == 0) break;
        if (tid == 0) st[(level + 2) % 3] = 0;
        const int32_t* fin = (level & 1) ? fa : fb;
        int32_t* fout = (level & 1) ? fb : fa;
        int32_t* nout = st + (level + 1) % 3;
        for (long long i0 = tid - lane; i0 < work; i0 += nt) {   // whole warps
            const long long i = i0 + lane;
            int32_t y = -1;
            if (i < work) {
                const long long fi = div_idx(i, R);
                y = graph[(long long)__ldcg(fin + fi) * R + (i - fi * R)];
            }
            const bool add = y >= 0 && y < N && __ldcg(visited + y) == 0 && atomicCAS(visited + y, 0, level + 1) == 0;
            const unsigned m = __ballot_sync(kFull, add);
            if (m == 0u) continue;
            int base = 0;
            if (lane == 0) base = atomicAdd(nout, __popc(m));
            base = __shfl_sync(kFull, base, 0);
            if (add) fout[base + __popc(m & ((1u << lane) - 1u))] = y;
            sum += __popc(m);
        }
        grid.sync();
    }
    if (lane == 0 && sum) atomicAdd(reinterpret_cast<unsigned long long*>(st + 4), (unsigned long long)sum);
}

cudaError_t launch_bfs(const int32_t* graph, int R, long long N, int entry, const int32_t* entries, int ne,
                       int32_t* visited, int32_t* fa, int32_t* fb, int32_t* st, int* status, cudaStream_t s) {
    int blocks = 0;
    const cudaError_t e = coop_grid(k_bfs, 512, std::min<long long>(cdivl(N * (long long)R, 512 * 4), 608), &blocks);
    if (e != cudaSuccess) return e;
    LaunchScope ls("k_bfs", s);
    void* args[] = {&graph, &R, &N, &entry, &entries, &ne, &visited, &fa, &fb, &st, &status};
    return cudaLaunchCooperativeKernel((const void*)k_bfs, dim3(blocks), dim3(512), args, 0, s);
}

// number of BFS parents of every reached vertex: in-neighbours at a smaller level
__global__ void k_bfs_parents(const int32_t* __restrict__ graph, int R, long long N, const int32_t* __restrict__ level,
                              int32_t* __restrict__ npar) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * R) return;
    const int32_t lx = level[div_idx(i, R)];
    if (lx == 0) return;
    const int32_t y = graph[i];
    if (y >= 0 && y < N && level[y] > lx) atomicAdd(npar + y, 1);
}

cudaError_t launch_bfs_parents(const int32_t* graph, int R, long long N, const int32_t* level, int32_t* npar,
                               cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(npar, 0, sizeof(int32_t) * N, s);
    if (e != cudaSuccess) return e;
    LaunchScope ls("k_bfs_parents", s);
    k_bfs_parents<<<(unsigned)cdivl(N * R, 256), 256, 0, s>>>(graph, R, N, level, npar);
    return cudaGetLastError();
}

// min-label propagation over the undirected edges between unreached vertices, all passes in one
// cooperative launch over the list of the unreached vertices, so that the host reads nothing between passes (14
// launches of a 1M merge become 5, 1.9 -> 1.2 ms; a batch of 64 merges takes as long as with a launch per pass, 9 ms).
// st[0]: their number, st[1 + it % 3]: pass it changed a label.
__global__ void __launch_bounds__(512) k_cc(const int32_t* __restrict__ graph, int R, long long N,
                                            const int32_t* __restrict__ visited, int32_t* label, int32_t* list,
                                            int32_t* st) {
    cg::grid_group grid = cg::this_grid();
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    const int lane = lane_id();
    for (long long i0 = tid - lane; i0 < N; i0 += nt) {
        const long long i = i0 + lane;
        const bool un = i < N && visited[i] == 0;
        if (i < N) label[i] = un ? (int32_t)i : -1;
        const unsigned m = __ballot_sync(kFull, un);
        if (m == 0u) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(st, __popc(m));
        base = __shfl_sync(kFull, base, 0);
        if (un) list[base + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
    }
    grid.sync();
    const long long work = (long long)__ldcg(st) * R;
    for (long long it = 0; it <= N; ++it) {
        bool changed = false;
        if (tid == 0) st[1 + (it + 1) % 3] = 0;
        for (long long i = tid; i < work; i += nt) {
            const long long li = div_idx(i, R);
            const int32_t x = __ldcg(list + li);
            const int32_t y = graph[(long long)x * R + (i - li * R)];
            if (y < 0 || y >= N || visited[y]) continue;
            const int32_t lx = __ldcg(label + x), ly = __ldcg(label + y);
            if (lx < ly) changed |= atomicMin(label + y, lx) > lx;
            else if (ly < lx) changed |= atomicMin(label + x, ly) > ly;
        }
        if (__any_sync(kFull, changed) && lane == 0) st[1 + it % 3] = 1;
        grid.sync();
        if (__ldcg(st + 1 + it % 3) == 0) break;
    }
}

cudaError_t launch_cc(const int32_t* graph, int R, long long N, const int32_t* visited, int32_t* label, int32_t* list,
                      int32_t* st, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(st, 0, 4 * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    int blocks = 0;
    if ((e = coop_grid(k_cc, 512, std::min<long long>(cdivl(N * (long long)R, 512 * 4), 304), &blocks)) != cudaSuccess) return e;
    LaunchScope ls("k_cc", s);
    void* args[] = {&graph, &R, &N, &visited, &label, &list, &st};
    return cudaLaunchCooperativeKernel((const void*)k_cc, dim3(blocks), dim3(512), args, 0, s);
}

__global__ void k_rep_flags(const int32_t* __restrict__ visited, const int32_t* __restrict__ label, long long N,
                            int32_t* __restrict__ flag) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) flag[i] = (!visited[i] && label[i] == (int32_t)i) ? 1 : 0;
}

cudaError_t launch_rep_flags(const int32_t* visited, const int32_t* label, long long N, int32_t* flag,
                             cudaStream_t s) {
    LaunchScope ls("k_rep_flags", s);
    k_rep_flags<<<(unsigned)cdivl(N, 256), 256, 0, s>>>(visited, label, N, flag);
    return cudaGetLastError();
}

// Attachment of the representatives with the result of the sequential loop over them in
// ascending id, computed in parallel rounds (warp per representative). The action of x:
// the first search result p with room gets x appended; otherwise the first search result
// with a replaceable neighbour y (reached, keeps a BFS parent other than p) has its
// farthest such y replaced by x. Reads that other actions cannot change are not reserved:
// a full list stays full (degrees only grow) and a neighbour that is not replaceable stays
// so (parent counts only shrink). Only p (its list and degree) and y (its parent count)
// are reserved with atomicMin of a tag ordered by (round, representative index); the
// longest ascending prefix of the round's window holding its reservations is committed,
// the rest recomputed in the next round.
//
// Round rho works on the window [start, min(start + W, nr)), start = ff[(rho - 1) % 3], and leaves in
// ff[rho % 3] the first index it did not commit (the next round's start). Tags of later rounds are
// smaller than those of earlier ones, so owner needs no reset between rounds.
__device__ __forceinline__ unsigned long long reach_tag(long long rho, long long r) {
    return ((unsigned long long)(0xFFFFFFFFu - (uint32_t)rho) << 32) | (unsigned long long)(uint32_t)r;
}

// The action of representative r on the current graph (whole warp; the result is the same in
// every lane): (p, position in p's list, index of p among r's search results, victim or -1);
// p = -1: no action.
__device__ __forceinline__ int4 reach_plan(const int32_t* __restrict__ graph, const int32_t* __restrict__ deg,
                                           const int32_t* __restrict__ level, const int32_t* __restrict__ npar,
                                           int R, const int32_t* cr, int beam, int lane) {
    int p = -1, pos = -1, t_sel = -1;
    for (int t0 = 0; t0 < beam && p < 0; t0 += 32) {
        const int t = t0 + lane;
        const int32_t q = t < beam ? cr[t] : -1;
        const bool room = q >= 0 && deg[q] < R;
        const unsigned m = __ballot_sync(kFull, room);
        if (m) {
            t_sel = t0 + __ffs(m) - 1;
            p = cr[t_sel];
            pos = deg[p];
        }
    }
    for (int t = 0; t < beam && p < 0; ++t) {
        const int32_t q = cr[t];
        if (q < 0) break;
        const int dq = deg[q];
        const int32_t lq = level[q];
        int best = -1;
        for (int s0 = ((R - 1) >> 5) << 5; s0 >= 0 && best < 0; s0 -= 32) {
            const int s = s0 + lane;
            bool ok = false;
            if (s < dq) {
                const int32_t y = graph[(long long)q * R + s];
                const int32_t ly = level[y];
                ok = ly > 0 && npar[y] - (lq < ly ? 1 : 0) >= 1;
            }
            const unsigned m = __ballot_sync(kFull, ok);
            if (m) best = s0 + 31 - __clz(m);
        }
        if (best >= 0) {
            p = q;
            pos = best;
            t_sel = t;
        }
    }
    const int32_t victim = (p >= 0 && pos < deg[p]) ? graph[(long long)p * R + pos] : -1;
    return make_int4(p, pos, t_sel, victim);
}

// The rounds in one cooperative launch (warps stride over the window): plan
// (the action of every item and its reservations), check (the first item that lost one
// bounds the prefix), commit (the prefix); phases are separated by grid-wide barriers and an
// item's plan is computed once per round. Every round commits at least one item.
__global__ void __launch_bounds__(kRoundThreads) k_reach_rounds(int32_t* graph, float* gdist, int32_t* deg,
                                                      const int32_t* __restrict__ level, int32_t* npar, int R,
                                                      const int32_t* __restrict__ reps, long long nr, long long window,
                                                      long long* ff, const int32_t* __restrict__ cand,
                                                      const float* __restrict__ cdist, int beam,
                                                      unsigned long long* owner, int4* plan,
                                                      unsigned long long* attached, int* status) {
    cg::grid_group grid = cg::this_grid();
    const int lane = lane_id();
    const long long gw = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    long long win = window;
    for (long long rho = 1;; ++rho) {
        const long long start = __ldcg(ff + (rho - 1) % 3);   // written before the last barrier
        if (start >= nr) break;                               // the same for every thread: all leave together
        if (rho > nr) {
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kErrTimeout);
            break;
        }
        const long long wend = start + win < nr ? start + win : nr;
        if (blockIdx.x == 0 && threadIdx.x == 0) ff[rho % 3] = wend;
        for (long long r = start + gw; r < wend; r += nw) {
            const int4 pl = reach_plan(graph, deg, level, npar, R, cand + r * beam, beam, lane);
            if (lane == 0) {
                plan[r - start] = pl;
                if (pl.x >= 0) {
                    const unsigned long long tag = reach_tag(rho, r);
                    atomicMin(owner + pl.x, tag);
                    if (pl.w >= 0) atomicMin(owner + pl.w, tag);
                }
            }
        }
        grid.sync();
        for (long long r = start + gw * 32 + lane; r < wend; r += nw * 32) {
            const int4 pl = plan[r - start];
            const unsigned long long tag = reach_tag(rho, r);
            if (pl.x >= 0 && (owner[pl.x] != tag || (pl.w >= 0 && owner[pl.w] != tag)))
                atomicMin((unsigned long long*)(ff + rho % 3), (unsigned long long)r);
        }
        grid.sync();
        const long long cend = __ldcg(ff + rho % 3);
        win = round_window(cend - start, window);
        for (long long r = start + gw * 32 + lane; r < cend; r += nw * 32) {
            const int4 pl = plan[r - start];
            if (pl.x < 0) continue;
            const int32_t p = pl.x, victim = pl.w, x = reps[r];
            int pos = pl.y;
            int32_t* li = graph + (long long)p * R;
            float* ld = gdist + (long long)p * R;
            const float d = cdist[r * beam + pl.z];
            const uint64_t key = mkkey(d, x);
            if (pos == deg[p]) deg[p] += 1;
            else if (level[p] < level[victim]) npar[victim] -= 1;
            while (pos > 0 && mkkey(ld[pos - 1], li[pos - 1]) > key) {
                li[pos] = li[pos - 1];
                ld[pos] = ld[pos - 1];
                --pos;
            }
            while (pos + 1 < deg[p] && mkkey(ld[pos + 1], li[pos + 1]) < key) {
                li[pos] = li[pos + 1];
                ld[pos] = ld[pos + 1];
                ++pos;
            }
            li[pos] = x;
            ld[pos] = d;
            atomicAdd(attached, 1ull);
        }
        grid.sync();
    }
}

cudaError_t launch_reach_rounds(int32_t* graph, float* gdist, int32_t* deg, const int32_t* level, int32_t* npar,
                                int R, const int32_t* reps, long long nr, long long* ff, const int32_t* cand,
                                const float* cdist, int beam, unsigned long long* owner, int4* plan,
                                unsigned long long* attached, int* status, cudaStream_t s) {
    long long window = kReachWindow;
    int blocks = 0;
    const cudaError_t e = coop_grid(k_reach_rounds, kRoundThreads, cdivl(std::min(window, nr), kRoundThreads / 32), &blocks);
    if (e != cudaSuccess) return e;
    LaunchScope ls("k_reach_rounds", s);
    void* args[] = {&graph, &gdist, &deg, &level, &npar, &R, &reps, &nr, &window, &ff, &cand, &cdist, &beam, &owner, &plan, &attached, &status};
    return cudaLaunchCooperativeKernel((const void*)k_reach_rounds, dim3(blocks), dim3(kRoundThreads), args, 0, s);
}

}  // namespace fgim
