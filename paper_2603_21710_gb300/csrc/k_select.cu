// Stage (c), Alg. 5 neighbour selection.
//
// The candidates of a vertex u are taken in ascending (delta, id). A candidate v is kept unless a neighbour
// w kept before it occludes it (PruneRule: alpha-RNG delta(u, v) < alpha^2 * delta(w, v) keeps v,
// with alpha^2 rounded once to FP32 and the product in FP32; or MRNG; or tau-MNG); one whose only
// in-edge is u (T(v) = 1) is kept whatever occludes it; selection stops at R kept neighbours.
//
// The kernels go over the kept neighbours instead of over the candidates: the first candidate of a
// window that is left is kept, and every later one of the window that is left is tested against it at
// once and dropped if it is occluded; the candidates of the next window are tested against the kept
// neighbours in their order first. A candidate is tested against the kept neighbours before it, until
// the first that occludes it, so the pairs and the decisions are those of the loop over candidates;
// but the serial steps are the kept neighbours (about 10 of 64 candidates when alpha = 1) and the
// pairs of a step are independent. Windows (32 candidates, then 16 at a time) bound what is tested past the
// candidate that fills the list; where much is occluded (alpha <= 1 and the other rules) all candidates are
// one window. Every decision is taken on the canonical distance.
// Measured against one step per candidate with its rows staged in shared memory (33 KB per warp at d =
// 128) and one lane per kept neighbour: 300k, d = 96, k = 48: 11.5 -> 2.7 ms; 36k, d = 960, k = 64: 5.7 -> 3.6;
// 1M byte rows, d = 128, alpha = 1.2: 8.0 -> 6.0; the builder's 141 selections (k = 128 and up) 40.9 -> 6.0.
#include "k_beam.cuh"

namespace fgim {

constexpr uint16_t kProtected = 0x8000u;   // list entry: T(v) = 1, never occluded
constexpr int kListMask = 0x7fff;
// lists up to which four warps serve one vertex (a batch of the graph builder has at most 1,024: 5.9 ms for
// the 141 selections of a 60,000-vertex build, 7.2 ms with one warp per vertex)
constexpr long long kSplitRows = 2048;
constexpr int kStageBytes = 16384;   // of one vertex's rows

// shared memory of one vertex: ids and distances of its list, the kept positions, its rows (staged:
// short lists of short rows), and per warp the candidates that are left (positions), 32 row ids and, for
// wide rows, the kept neighbour's row
struct SelectLayout {
    int cid, dl, kept, heads, rows, warp0, q, scratch, list, warp_bytes, bytes;
};

__host__ __device__ inline SelectLayout select_layout(int k, int R, int d, int nw, bool stage) {
    SelectLayout l;
    int o = 0;
    l.cid = o;
    o += align16(k * 4);
    l.dl = o;
    o += align16(k * 4);
    l.kept = o;
    o += align16(R * 4);
    l.heads = o;
    o += 2 * 4 * 4;
    l.rows = o;
    if (stage) o += k * d * 4;
    l.warp0 = o;
    int w = 0;
    l.q = w;
    if (d > 128) w += align16(d * 4);
    l.scratch = w;
    w += 32 * 4;
    l.list = w;
    w += align16(((k + nw - 1) / nw) * 2);
    l.warp_bytes = w;
    l.bytes = o + nw * w;
    return l;
}

// The list of a vertex: its entries before the first that is no vertex id (an empty or negative one, or one of N
// or above, which is reported). Every lane gets their number; position s goes to cid[s] and dl[s] where this warp
// (vw of the vertex's NW) holds it. Positions past the list are not to be read: they may hold anything.
template <int NW>
__device__ __forceinline__ int load_list(const int32_t* __restrict__ ids, const float* __restrict__ dist, int k, long long N,
                                         int vw, int lane, int32_t* cid, float* dl, int* status) {
    int nv = k;
    for (int s0 = 0; s0 < k; s0 += 32) {
        const int s = s0 + lane;
        int32_t id = s < k ? ids[s] : -1;
        if (id >= N) {
            atomicOr(status, kErrBounds);
            id = -1;
        }
        if (s < k && (s0 >> 5) % NW == vw) {
            cid[s] = id;
            dl[s] = dist[s];
        }
        const unsigned none = __ballot_sync(kFull, id < 0);
        if (none) nv = min(nv, s0 + __ffs(none) - 1);
    }
    return nv;
}

// NW warps per vertex: 1 (four vertices per block), or 4 when there are too few vertices to fill the
// GPU with one warp each; warp w of a vertex then holds the candidates at positions w, w + 4, ..., all in
// one window, and the warps agree on the next kept neighbour (the smallest position left) once per step.
// STAGE: the rows of the list are copied to shared memory first (a step's reads depend on the last
// step's outcome, so their latency adds up).
template <int METRIC, bool SMALLD, typename RT, int NW, bool STAGE>
__global__ void __launch_bounds__(128, sizeof(RT) == 1 ? 8 : SMALLD ? 5 : 4) k_prune(
    const RT* __restrict__ Xr, const float* __restrict__ inv_norm, long long N, long long nrows, int d, int k,
    const int32_t* __restrict__ ids, const float* __restrict__ dist, const int32_t* __restrict__ T, int R,
    PruneRule rule, int32_t* __restrict__ e_ids, float* __restrict__ e_dist, int32_t* __restrict__ e_cnt,
    int* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const long long u = NW == 1 ? (long long)blockIdx.x * 4 + warp : (long long)blockIdx.x;
    if (u >= nrows) return;
    const int vw = NW == 1 ? 0 : warp;   // warp of the vertex
    const SelectLayout L = select_layout(k, R, d, NW, STAGE);
    unsigned char* base = smem + (NW == 1 ? (size_t)warp * L.bytes : 0);
    int32_t* cid = reinterpret_cast<int32_t*>(base + L.cid);
    float* dl = reinterpret_cast<float*>(base + L.dl);
    int32_t* kept = reinterpret_cast<int32_t*>(base + L.kept);
    int* heads = reinterpret_cast<int*>(base + L.heads);
    RT* rows = reinterpret_cast<RT*>(base + L.rows);
    unsigned char* wb = base + L.warp0 + (size_t)vw * L.warp_bytes;
    float* qs = reinterpret_cast<float*>(wb + L.q);
    int32_t* scratch = reinterpret_cast<int32_t*>(wb + L.scratch);
    uint16_t* list = reinterpret_cast<uint16_t*>(wb + L.list);
    auto vsync = [&]() {
        if (NW == 1) __syncwarp();
        else __syncthreads();
    };

    const int nv = load_list<NW>(ids + u * k, dist + u * k, k, N, vw, lane, cid, dl, status);
    vsync();
    if (STAGE) {
        const int c16 = d * (int)sizeof(RT) >> 4;   // 16-byte pieces per row
        for (int i = lane; i < nv * c16; i += 32) {
            const int r = i / c16, c = i - r * c16;
            reinterpret_cast<uint4*>(rows)[i] = reinterpret_cast<const uint4*>(Xr + (long long)cid[r] * d)[c];
        }
    }
    // this warp's candidates
    const int total = nv > vw ? (nv - vw + NW - 1) / NW : 0;
    for (int i = lane; i < total; i += 32) {
        const int t = vw + i * NW;
        list[i] = (uint16_t)(t | (T[cid[t]] == 1 ? kProtected : 0));
    }
    __syncwarp();
    // the window: list[a0 .. m), tested against kept[0 .. ki); list[nxt .. total) has not been looked at
    int a0 = 0, m = NW == 1 && rule.kind == 0 && rule.alpha2 > 1.f ? min(total, 32) : total, nxt = m, nk = 0, ki = 0;
    for (int step = 0;; ++step) {
        if (NW == 1 && a0 == m) {   // the next window
            if (nxt == total) break;
            a0 = nxt;
            nxt = min(nxt + 16, total);
            m = nxt;
            ki = 0;
        }
        if (ki == nk) {   // the first candidate left is kept
            int head = a0 < m ? (list[a0] & kListMask) : kListMask + 1;
            const int own = head;
            if (NW > 1) {
                int* h = heads + 4 * (step & 1);
                if (lane == 0) h[vw] = head;
                __syncthreads();
                head = min(min(h[0], h[1]), min(h[2], h[3]));
                if (head > kListMask) break;
            }
            a0 += own == head ? 1 : 0;
            if (lane == 0 && vw == 0) kept[nk] = head;
            ++nk;
            if (nk == R) break;
            vsync();
        }
        const int tw = kept[ki++];
        const int32_t w = cid[tw];
        if (a0 == m) continue;   // nothing to test
        const Query Q = row_query<SMALLD, RT>(STAGE ? rows + tw * d : Xr + (long long)w * d, qs, d, lane);
        const float duw = dl[tw];
        const float inv_w = METRIC == FGIM_COSINE ? inv_norm[w] : 1.f;
        int out = a0;
        for (int i0 = a0; i0 < m; i0 += 32) {
            const bool has = i0 + lane < m;
            const int a = has ? list[i0 + lane] : 0;
            const int t = a & kListMask;
            const int32_t v = has ? cid[t] : 0;
            const bool test = has && !(a & kProtected);
            const unsigned tm = __ballot_sync(kFull, test);
            bool occ = false;
            if (tm) {
                if (test) scratch[__popc(tm & lt)] = STAGE ? t : v;
                __syncwarp();
                const float dd = rows_delta<METRIC, SMALLD, RT>(STAGE ? rows : Xr, scratch, __popc(tm), Q, d, lane);
                const float sum = __shfl_sync(kFull, dd, __popc(tm & lt) & 31);
                if (test) {
                    const float inv = METRIC == FGIM_COSINE ? __fmul_rn(inv_w, inv_norm[v]) : 1.f;
                    occ = rule_occludes(rule, dl[t], duw, delta_finish<METRIC>(sum, inv));
                }
            }
            const unsigned km = __ballot_sync(kFull, has && !occ);
            if (has && !occ) list[out + __popc(km & lt)] = (uint16_t)a;   // at or before its old place
            out += __popc(km);
            __syncwarp();
        }
        m = out;
    }
    vsync();
    for (int s = vw * 32 + lane; s < R; s += NW * 32) {
        if (s < nk) {
            e_ids[u * R + s] = cid[kept[s]];
            e_dist[u * R + s] = dl[kept[s]];
        } else {
            e_ids[u * R + s] = -1;
            e_dist[u * R + s] = __int_as_float(0x7f800000);
        }
    }
    if (vw == 0 && lane == 0) e_cnt[u] = nk;
}

// Byte rows (every coordinate an integer in [0, 255], d <= 128), lists of at most 64: one lane per
// candidate. The canonical distance is the exact integer |a|^2 + |b|^2 - 2 a.b; a lane holds its candidate's
// row in registers and the kept neighbour's row is read from shared memory, the same address in every
// lane. In the second 32 candidates, when more than 16 neighbours are kept already (few candidates are
// occluded, and few are still needed), a lane holds a kept neighbour's row instead and the
// candidates come one after another. Bound by the 32 dot products per lane and step and the shared
// memory reads (8 of one address each; with both rows of a pair in shared memory it would be 40
// bank cycles per step).
constexpr int kBytesK = 64;
constexpr int kManyKept = 16;

__host__ __device__ inline int prune_bytes_per_warp(int k, int R, int d) {
    return k * (d + 16) + align16(k * 4) * 3 + align16(R * 4);
}

template <int METRIC>
__global__ void __launch_bounds__(128, 5) k_prune_bytes(
    const uint8_t* __restrict__ X8, const float* __restrict__ inv_norm, long long N, long long nrows, int d, int k,
    const int32_t* __restrict__ ids, const float* __restrict__ dist, const int32_t* __restrict__ T, int R,
    PruneRule rule, int32_t* __restrict__ e_ids, float* __restrict__ e_dist, int32_t* __restrict__ e_cnt,
    int* status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = lane_id();
    const long long u = (long long)blockIdx.x * 4 + warp;
    if (u >= nrows) return;
    const int stride = d + 16;
    unsigned char* rows = smem + (size_t)prune_bytes_per_warp(k, R, d) * warp;
    int32_t* cid = reinterpret_cast<int32_t*>(rows + k * stride);
    float* dl = reinterpret_cast<float*>(cid + align16(k * 4) / 4);
    uint32_t* n2 = reinterpret_cast<uint32_t*>(dl + align16(k * 4) / 4);
    int32_t* kept = reinterpret_cast<int32_t*>(n2 + align16(k * 4) / 4);
    const int c16n = d >> 4;
    const int lsh = byte_lanes_log2(d);
    const int rpi = 32 >> lsh;   // rows per warp load
    const int sub = lane >> lsh, part = lane & ((1 << lsh) - 1);

    const int nv = load_list<1>(ids + u * k, dist + u * k, k, N, 0, lane, cid, dl, status);
    __syncwarp();
    uint4 xr[8];   // this lane's row
    uint32_t x2 = 0u;
    float inv_l = 1.f, dl_l = 0.f;
    auto hold = [&](int t) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
            xr[c] = c < c16n ? *reinterpret_cast<const uint4*>(rows + t * stride + 16 * c) : make_uint4(0u, 0u, 0u, 0u);
        x2 = n2[t];
        dl_l = dl[t];
        if (METRIC == FGIM_COSINE) inv_l = inv_norm[cid[t]];
    };
    // delta(row t, this lane's row): the four chains are integer sums, any order gives the same total
    auto delta_to = [&](int t) -> float {
        uint32_t d0 = 0u, d1 = 0u, d2 = 0u, d3 = 0u;
        const uint4* r = reinterpret_cast<const uint4*>(rows + t * stride);
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c < c16n) {
                const uint4 y = r[c];
                d0 = __dp4a(y.x, xr[c].x, d0);
                d1 = __dp4a(y.y, xr[c].y, d1);
                d2 = __dp4a(y.z, xr[c].z, d2);
                d3 = __dp4a(y.w, xr[c].w, d3);
            }
        const uint32_t dot = (d0 + d1) + (d2 + d3);
        if (METRIC == FGIM_L2SQ) return (float)(n2[t] + x2 - 2u * dot);
        return delta_finish<METRIC>((float)dot, METRIC == FGIM_COSINE ? __fmul_rn(inv_norm[cid[t]], inv_l) : 1.f);
    };
    int nk = 0;
    for (int w0 = 0; w0 < nv && nk < R; w0 += 32) {
        const int wn = min(32, nv - w0);
        // the window's rows to shared memory with their squared norms, four warp loads at a time
        for (int r0 = 0; r0 < wn; r0 += 4 * rpi) {
            uint4 x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * rpi + sub;
                x[q] = make_uint4(0u, 0u, 0u, 0u);
                if (r < wn && part < c16n)
                    x[q] = *reinterpret_cast<const uint4*>(X8 + (long long)cid[w0 + r] * d + 16 * part);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * rpi + sub;
                uint32_t sq = __dp4a(x[q].x, x[q].x, 0u);
                sq = __dp4a(x[q].y, x[q].y, sq);
                sq = __dp4a(x[q].z, x[q].z, sq);
                sq = __dp4a(x[q].w, x[q].w, sq);
                sq = row_group_sum(sq, lsh);
                if (r < wn) {
                    if (part < c16n) *reinterpret_cast<uint4*>(rows + (w0 + r) * stride + 16 * part) = x[q];
                    if (part == 0) n2[w0 + r] = sq;
                }
            }
        }
        const bool has = lane < wn;
        const bool prot = has && T[cid[w0 + lane]] == 1;   // never occluded
        __syncwarp();
        if (nk > kManyKept && R <= 32) {
            const unsigned pm = __ballot_sync(kFull, prot);
            if (lane < nk) hold(kept[lane]);
            for (int j = 0; j < wn && nk < R; ++j) {
                const int t = w0 + j;
                bool occ = false;
                if (!((pm >> j) & 1u)) {
                    const float dd = delta_to(t);
                    occ = lane < nk && rule_occludes(rule, dl[t], dl_l, dd);
                }
                if (__any_sync(kFull, occ)) continue;
                if (lane == nk) {
                    kept[nk] = t;
                    hold(t);
                }
                ++nk;
            }
            __syncwarp();
            continue;
        }
        unsigned left = __ballot_sync(kFull, has);
        if (has) hold(w0 + lane);
        for (int ki = 0; left; ++ki) {
            if (ki == nk) {   // the first candidate left is kept
                const int t = __ffs(left) - 1;
                left &= left - 1;
                if (lane == 0) kept[nk] = w0 + t;
                __syncwarp();
                if (++nk == R || !left) break;
            }
            const int tw = kept[ki];
            const float dd = delta_to(tw);
            const bool occ = !prot && rule_occludes(rule, dl_l, dl[tw], dd);
            left &= ~__ballot_sync(kFull, occ);
        }
    }
    __syncwarp();
    for (int s = lane; s < R; s += 32) {
        if (s < nk) {
            e_ids[u * R + s] = cid[kept[s]];
            e_dist[u * R + s] = dl[kept[s]];
        } else {
            e_ids[u * R + s] = -1;
            e_dist[u * R + s] = __int_as_float(0x7f800000);
        }
    }
    if (lane == 0) e_cnt[u] = nk;
}

cudaError_t launch_prune(const float* X, const uint8_t* X8, const uint16_t* Xh, const float* inv_norm, long long N,
                         int d, int metric, const fgim_knng& g, const int32_t* T, int R, PruneRule rule,
                         int32_t* e_ids, float* e_dist, int32_t* e_cnt, int* status, cudaStream_t s) {
    const long long nrows = g.n;   // lists to prune (ids range over 0 .. N - 1)
    if (nrows <= 0) return cudaSuccess;
    const int k = g.k;
    if (k > kListMask) return cudaErrorInvalidValue;
    const bool bytes = X8 && byte_rows_ok(d);
    const bool bf16 = !bytes && Xh && d > 128 && (reinterpret_cast<uintptr_t>(Xh) & 7u) == 0;
    const bool split = nrows <= kSplitRows;
    cudaError_t e = cudaSuccess;
    if (bytes && k <= kBytesK && !split) {
        const size_t smem = (size_t)prune_bytes_per_warp(k, R, d) * 4;
#define FGIM_LAUNCH_PB(MT)                                                                                        \
    do {                                                                                                          \
        e = allow_smem(k_prune_bytes<MT>, smem); \
        if (e != cudaSuccess) break;                                                                              \
        LaunchScope ls("k_prune", s);                                                                             \
        k_prune_bytes<MT><<<(unsigned)((nrows + 3) / 4), 128, smem, s>>>(X8, inv_norm, N, nrows, d, k, g.ids, g.dist, \
                                                                         T, R, rule, e_ids, e_dist, e_cnt, status); \
        e = cudaGetLastError();                                                                                   \
    } while (0)
        if (metric == FGIM_L2SQ) FGIM_LAUNCH_PB(FGIM_L2SQ);
        else if (metric == FGIM_IP) FGIM_LAUNCH_PB(FGIM_IP);
        else FGIM_LAUNCH_PB(FGIM_COSINE);
#undef FGIM_LAUNCH_PB
        return e;
    }
    const bool stage = !split && !bytes && d <= 128 && k * d * 4 <= kStageBytes;
    const SelectLayout L = select_layout(k, R, d, split ? 4 : 1, stage);
    const size_t smem = (size_t)L.bytes * (split ? 1 : 4);
    const unsigned blocks = (unsigned)(split ? nrows : (nrows + 3) / 4);
#define FGIM_LAUNCH_P2(MT, SD, RT, W, ST, ROWS)                                                                   \
    do {                                                                                                          \
        e = allow_smem(k_prune<MT, SD, RT, W, ST>, smem); \
        if (e != cudaSuccess) break;                                                                              \
        LaunchScope ls("k_prune", s);                                                                             \
        k_prune<MT, SD, RT, W, ST><<<blocks, 128, smem, s>>>(ROWS, inv_norm, N, nrows, d, k, g.ids, g.dist, T, R, \
                                                             rule, e_ids, e_dist, e_cnt, status);                 \
        e = cudaGetLastError();                                                                                   \
    } while (0)
#define FGIM_LAUNCH_P(MT, SD, RT, ROWS)                                                                           \
    do {                                                                                                          \
        if (split) FGIM_LAUNCH_P2(MT, SD, RT, 4, false, ROWS);                                                    \
        else FGIM_LAUNCH_P2(MT, SD, RT, 1, false, ROWS);                                                          \
    } while (0)
#define FGIM_LAUNCH_PM(SD, RT, ROWS)                                                                              \
    do {                                                                                                          \
        if (metric == FGIM_L2SQ) FGIM_LAUNCH_P(FGIM_L2SQ, SD, RT, ROWS);                                          \
        else if (metric == FGIM_IP) FGIM_LAUNCH_P(FGIM_IP, SD, RT, ROWS);                                         \
        else FGIM_LAUNCH_P(FGIM_COSINE, SD, RT, ROWS);                                                            \
    } while (0)
    if (stage) {
        if (metric == FGIM_L2SQ) FGIM_LAUNCH_P2(FGIM_L2SQ, true, float, 1, true, X);
        else if (metric == FGIM_IP) FGIM_LAUNCH_P2(FGIM_IP, true, float, 1, true, X);
        else FGIM_LAUNCH_P2(FGIM_COSINE, true, float, 1, true, X);
    } else if (bytes) {
        FGIM_LAUNCH_PM(true, uint8_t, X8);
    } else if (bf16) {   // BF16 storage: the same values, half the bytes
        FGIM_LAUNCH_PM(false, uint16_t, Xh);
    } else if (d <= 128) {
        FGIM_LAUNCH_PM(true, float, X);
    } else {
        FGIM_LAUNCH_PM(false, float, X);
    }
#undef FGIM_LAUNCH_PM
#undef FGIM_LAUNCH_P
#undef FGIM_LAUNCH_P2
    return e;
}

}  // namespace fgim
