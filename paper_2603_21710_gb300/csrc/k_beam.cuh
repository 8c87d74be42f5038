// Alg. 1 (KNNSearch) on the GPU, shared by the cross query of Alg. 2 (k_cross.cu) and the
// evaluation / reachability searches (k_search.cu).
//
// One warp runs one beam search. The pool C (<= L keys, sorted by (delta, id)) lives in registers
// with a copy in shared memory; each expansion reads the expanded vertex's adjacency row (one id
// per lane), drops ids already evaluated, compacts the rest, loads their rows coalesced (eight
// lanes per row up to 128 coordinates), forms the canonical distances of up to 32 rows and merges
// those that beat the pool's worst entry into the pool all at once.
//
// Evaluated ids are remembered in a small direct-mapped table that may forget an id
// when another id lands on its slot (never the reverse). A forgotten id is evaluated
// again: its key equals its earlier key, so it is dropped if it is still in the pool,
// and otherwise it cannot beat the pool's worst entry (once the pool is full its worst
// key only decreases, and an id leaves the pool or is refused only when L better keys
// are present). The pool therefore evolves exactly as with an exact visited set
// (Alg. 1's "not visited" test); only the number of distance evaluations grows.
//
// Rows are read as FP32 or, when every coordinate of the data set is an integer in
// [0, 255], as one byte per coordinate (the merge checks this once). Both decode to the
// same FP32 values, so every distance, and with it every result, is the same; the byte
// rows move a quarter of the bytes, and at d = 128 a million of them fit in L2.
#pragma once
#include <algorithm>

#include "fgim_internal.cuh"
#include "fgim_launch.h"

namespace fgim {

// The table of evaluated ids: 2^htbits slots of 16 bits. A local id is multiplied by an odd constant
// modulo 2^b (b = the bits of a local id, at least htbits), which is a bijection; the product's top
// htbits bits are the slot and the rest is the tag kept there, so a slot names one id exactly. Ids whose
// tag needs more than 16 bits (graphs above 2^(htbits + 16) vertices) are not remembered, which is
// always allowed.
constexpr uint16_t kNoTag = 0xffffu;
struct VisitedHash {
    uint32_t mask;    // 2^b - 1
    uint32_t tmask;   // the tag's bits
    int sh;           // b - htbits
    __device__ __forceinline__ VisitedHash(int nt, int htbits) {
        const int b = max(nt > 1 ? 32 - __clz(nt - 1) : 1, htbits);
        mask = b >= 32 ? 0xffffffffu : (1u << b) - 1u;
        sh = b - htbits;
        tmask = (1u << sh) - 1u;
    }
    // true when v is in the table (it is after the call, if its tag fits)
    __device__ __forceinline__ bool seen(uint16_t* ht, int v) const {
        const uint32_t x = ((uint32_t)v * 2654435761u) & mask;
        const uint32_t tag = x & tmask;
        uint16_t* p = ht + (x >> sh);
        if (tag >= kNoTag) return false;
        if (*p == (uint16_t)tag) return true;
        *p = (uint16_t)tag;
        return false;
    }
    __device__ __forceinline__ void add(uint16_t* ht, int v) const { seen(ht, v); }
};

__device__ __forceinline__ void ht_clear(uint16_t* ht, int htbits, int lane) {
    uint4* p = reinterpret_cast<uint4*>(ht);
    for (int i = lane; i < (1 << htbits) / 8; i += 32) p[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
}

struct WarpCounters {   // the same in every lane
    unsigned long long ndc = 0;
    unsigned long long hops = 0;
};

__device__ __forceinline__ float4 u8x4_to_float4(uint32_t w) {
    return make_float4((float)(w & 0xffu), (float)((w >> 8) & 0xffu), (float)((w >> 16) & 0xffu), (float)(w >> 24));
}

// float4 chunk c (coordinates 4c .. 4c + 3) of a row of FP32, BF16 or byte storage (BF16 and
// bytes decode exactly to the FP32 values the merge works on)
__device__ __forceinline__ float4 row_chunk(const float* row, int c) { return reinterpret_cast<const float4*>(row)[c]; }
__device__ __forceinline__ float4 row_chunk(const uint16_t* row, int c) {
    const uint2 w = reinterpret_cast<const uint2*>(row)[c];
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ float4 row_chunk(const uint8_t* row, int c) {
    return u8x4_to_float4(*reinterpret_cast<const uint32_t*>(row + 4 * c));
}

// The query as the warp's lanes hold it. Byte rows: this lane's 16 bytes (chunk lane %
// lanes-per-row) and the sum of the squared coordinates. FP32 rows up to 128 coordinates: the
// lane's float4 chunks p, p + 8, p + 16, p + 24 (p = lane % 8; zero past the row). Wider rows: the
// whole query in shared memory.
struct Query {
    uint4 w;
    uint32_t q2;
    float4 c[4];
    const float* q;
};

__device__ __forceinline__ uint32_t pack4(const float4 v) {
    return __float2uint_rn(v.x) | (__float2uint_rn(v.y) << 8) | (__float2uint_rn(v.z) << 16) |
           (__float2uint_rn(v.w) << 24);
}

// src: the query's FP32 row in global memory; qs: d floats of this warp's shared memory (wide rows)
template <bool SMALLD, typename RT>
__device__ __forceinline__ Query load_query(const float* __restrict__ src, float* qs, int d, int lane) {
    Query Q;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    if constexpr (sizeof(RT) == 1) {
        const int lsh = byte_lanes_log2(d);
        const int part = lane & ((1 << lsh) - 1);
        Q.w = make_uint4(0u, 0u, 0u, 0u);
        if (part < (d >> 4)) {
            const float4* c = s4 + 4 * part;
            Q.w = make_uint4(pack4(c[0]), pack4(c[1]), pack4(c[2]), pack4(c[3]));
        }
        uint32_t s = __dp4a(Q.w.x, Q.w.x, 0u);
        s = __dp4a(Q.w.y, Q.w.y, s);
        s = __dp4a(Q.w.z, Q.w.z, s);
        s = __dp4a(Q.w.w, Q.w.w, s);
        Q.q2 = row_group_sum(s, lsh);   // integers: exact in any order
    } else if constexpr (SMALLD) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = (lane & 7) + 8 * i;
            Q.c[i] = c < (d >> 2) ? s4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
        float4* q4 = reinterpret_cast<float4*>(qs);
        for (int c = lane; c < (d >> 2); c += 32) q4[c] = s4[c];
        Q.q = qs;
        __syncwarp();
    }
    return Q;
}

// one row as the query of rows_delta (the values of load_query, read from the row storage in use)
template <bool SMALLD, typename RT>
__device__ __forceinline__ Query row_query(const RT* __restrict__ row, float* qs, int d, int lane) {
    Query Q;
    if constexpr (sizeof(RT) == 1) {
        const int lsh = byte_lanes_log2(d);
        const int part = lane & ((1 << lsh) - 1);
        Q.w = make_uint4(0u, 0u, 0u, 0u);
        if (part < (d >> 4)) Q.w = reinterpret_cast<const uint4*>(row)[part];
        uint32_t s = __dp4a(Q.w.x, Q.w.x, 0u);
        s = __dp4a(Q.w.y, Q.w.y, s);
        s = __dp4a(Q.w.z, Q.w.z, s);
        s = __dp4a(Q.w.w, Q.w.w, s);
        Q.q2 = row_group_sum(s, lsh);
    } else if constexpr (SMALLD) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = (lane & 7) + 8 * i;
            Q.c[i] = c < (d >> 2) ? row_chunk(row, c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
        float4* q4 = reinterpret_cast<float4*>(qs);
        for (int c = lane; c < (d >> 2); c += 32) q4[c] = row_chunk(row, c);
        Q.q = qs;
        __syncwarp();
    }
    return Q;
}

// The sums of four partials per lane over the eight lanes of a row (offsets 4, 2, 1, the last
// three levels of the butterfly), all four together: each exchange step halves the values a lane
// keeps, so lane p of row group s ends with the total of partial p / 2. Lane r then takes the total of
// row r when r is in [r0, r0 + 16): partial (r - r0) / 4, group r % 4 (r0 a multiple of 16). The additions
// are the butterfly's (each is commutative), so FP32 totals are the canonical ones.
template <typename T, typename ADD>
__device__ __forceinline__ T take_row_totals(const T (&v)[4], int r0, T mine, int lane, ADD add) {
    const bool b2 = (lane & 4) != 0, b1 = (lane & 2) != 0;
    const T h0 = add(b2 ? v[2] : v[0], __shfl_xor_sync(kFull, b2 ? v[0] : v[2], 4));
    const T h1 = add(b2 ? v[3] : v[1], __shfl_xor_sync(kFull, b2 ? v[1] : v[3], 4));
    T x = add(b1 ? h1 : h0, __shfl_xor_sync(kFull, b1 ? h0 : h1, 2));
    x = add(x, __shfl_xor_sync(kFull, x, 1));
    const T got = __shfl_sync(kFull, x, 8 * (lane & 3) + 2 * ((lane >> 2) & 3));
    return (lane & 16) == r0 ? got : mine;
}

// Canonical distance sums between the query and the U <= 32 rows base[rid[r]]; lane r receives row r's.
// FP32 rows up to 128 coordinates: eight lanes per row, four rows per warp load, eight loads in
// flight. Lane p adds the partials of chunks p, p + 16 and p + 8, p + 24 (the butterfly's offsets 16
// and 8) by itself and the eight lanes' sums go through its last three levels four rows at a time. (One
// row per warp load, its 32 x 32 partials re-added through 4 KB of shared memory, takes a third more
// instructions per row and halves the warps that fit on an SM.)
// Wider rows: eight rows at a time, one lane per chunk, two chunks of every row (16 loads) in
// flight; the eight rows' partials go through the butterfly together. The kernels are compiled for fewer
// resident warps here (16 per SM in the cross query, 12 in k_search): the gather is bound by L2 and DRAM
// latency, and loads in flight count for more than warps. Measured (d = 768 BF16, 120k): cross query
// 13.9 ms with 8 loads and 20 warps, 12.5 ms so; k_search 1.51 and 0.89 ms. On FP32 rows the eight rows' chunks
// and sums are more than the registers hold: 48 to 112 bytes spill in the cross query (128 registers), up to 36 in
// k_search (168).
// Byte rows (d <= 128, d % 16 == 0): every partial sum of the canonical FP32 value is then an
// integer below 128 * 255^2 < 2^24, so it is exact and the canonical value is the exact
// integer result. Lanes take 16 bytes each (32 / lanes-per-row rows per warp load) and form
// |q|^2 + |x|^2 - 2 q.x with four-way byte dot products, summed over the row's lanes. The loads are
// unconditional (a lane past the rows, or past a row's end, reads valid bytes again), and warp loads without a
// row are left out together: cross query of the 1M Sift-like merge 53.4 -> 51.3 ms (without the latter 53.0).
// SKIP (FP32 rows up to 128 coordinates; many warps share an SM): the loads are unconditional (past the last
// row its chunks again, past a row's end its last chunk, left out of the sum by a branch), and the second
// eight rows of a step are left out together when there are none. Loads under a lane's own condition made
// each row's a branch of its own: cross query 300k d = 96 15.1 -> 13.0 ms, d = 32 0.445 -> 0.398 ms. k_search,
// where few searches wait for each other's chain, is slower so (10,000 queries 0.86 -> 0.96 ms) and
// leaves it off, as is reading the next entry's adjacency row ahead there (held in a register 1.6 ms,
// as a prefetch 0.94).
template <int METRIC, bool SMALLD, typename RT, bool SKIP = true>
__device__ __forceinline__ float rows_delta(const RT* __restrict__ base, const int32_t* rid, int U, const Query& Q,
                                            int d, int lane) {
    const int nc4 = d >> 2;
    if constexpr (sizeof(RT) == 1) {
        const int lpr = byte_lanes(d);
        const int rpi = 32 >> byte_lanes_log2(d);   // rows per warp load
        const int lsh = byte_lanes_log2(d), rsh = 5 - lsh;   // lpr = 1 << lsh, rpi = 1 << rsh
        const int sub = lane >> lsh, part = lane & (lpr - 1);
        const bool has = part < (d >> 4);
        // rows in batches of four warp loads (all issued before the sums)
        uint32_t mine = 0u;
        for (int t0 = 0; t0 * rpi < U; t0 += 4) {
            uint4 w[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int r = (t0 + t) * rpi + sub;
                if ((t0 + t) * rpi >= U) {   // the same for every lane
                    w[t] = make_uint4(0u, 0u, 0u, 0u);
                    continue;
                }
                w[t] = *reinterpret_cast<const uint4*>(base + (long long)rid[min(r, U - 1)] * d + 16 * min(part, (d >> 4) - 1));
            }
            uint32_t sv[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                uint32_t sq = __dp4a(Q.w.x, w[t].x, 0u);
                sq = __dp4a(Q.w.y, w[t].y, sq);
                sq = __dp4a(Q.w.z, w[t].z, sq);
                sq = __dp4a(Q.w.w, w[t].w, sq);
                if (METRIC == FGIM_L2SQ) {
                    uint32_t sx = __dp4a(w[t].x, w[t].x, 0u);
                    sx = __dp4a(w[t].y, w[t].y, sx);
                    sx = __dp4a(w[t].z, w[t].z, sx);
                    sx = __dp4a(w[t].w, w[t].w, sx);
                    sv[t] = has ? sx - 2u * sq : 0u;   // modulo 2^32; the row total is exact
                } else {
                    sv[t] = sq;
                }
            }
            if (lsh == 3) {   // eight lanes per row: t0 is 0 or 4, the batch holds rows 4 t0 .. 4 t0 + 15
                mine = take_row_totals(sv, 4 * t0, mine, lane, [](uint32_t a, uint32_t b) { return a + b; });
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if ((t0 + t) * rpi < U) {
                        const uint32_t tot = row_group_sum(sv[t], lsh);
                        const uint32_t got = __shfl_sync(kFull, tot, (lane & (rpi - 1)) << lsh);
                        if ((lane >> rsh) == t0 + t) mine = got;
                    }
                }
            }
        }
        if (METRIC == FGIM_L2SQ) mine += Q.q2;
        return lane < U ? (float)mine : 0.f;
    } else if constexpr (SMALLD) {
        const int part = lane & 7, sub = lane >> 3;
        float mine = 0.f;
        for (int r0 = 0; r0 < U; r0 += 16) {
            float sv[4];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                if (SKIP && hf && r0 + 8 >= U) {
                    sv[2] = sv[3] = 0.f;
                    continue;
                }
                float4 y[2][4];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int r = r0 + 8 * hf + 4 * t + sub;
                    if (SKIP) {
                        const RT* row = base + (long long)rid[min(r, U - 1)] * d;
#pragma unroll
                        for (int i = 0; i < 4; ++i) y[t][i] = row_chunk(row, min(part + 8 * i, nc4 - 1));
                        continue;
                    }
                    const bool ok = r < U;
                    const RT* row = base + (long long)(ok ? rid[r] : 0) * d;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        y[t][i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (ok && part + 8 * i < nc4) y[t][i] = row_chunk(row, part + 8 * i);
                    }
                }
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    float pt[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (!SKIP || part + 8 * i < nc4) pt[i] = chunk_part<METRIC>(Q.c[i], y[t][i]);
                    sv[2 * hf + t] = __fadd_rn(__fadd_rn(pt[0], pt[2]), __fadd_rn(pt[1], pt[3]));
                }
            }
            mine = take_row_totals(sv, r0, mine, lane, [](float a, float b) { return __fadd_rn(a, b); });
        }
        return mine;
    } else {
        // each row keeps four accumulators per lane, in the chunk order of lane_part
        float mine = 0.f;
        for (int b = 0; b < U; b += 8) {
            const RT* rowp[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) rowp[t] = base + (long long)rid[b + t < U ? b + t : b] * d;
            float acc[8][4];
#pragma unroll
            for (int t = 0; t < 8; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll 2
            for (int c = lane; c < nc4; c += 32) {
                const float4 x = reinterpret_cast<const float4*>(Q.q)[c];
                float4 y[8];
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    y[t] = b + t < U ? row_chunk(rowp[t], c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int t = 0; t < 8; ++t) {
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
                }
            }
            // the butterfly over the eight rows together: offsets 16, 8 and 4 halve the rows a lane
            // keeps (row lane / 4 is left), offsets 2 and 1 finish it
            float v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t)
                v[t] = __fadd_rn(__fadd_rn(acc[t][0], acc[t][1]), __fadd_rn(acc[t][2], acc[t][3]));
#pragma unroll
            for (int o = 16, n = 4; o >= 4; o >>= 1, n >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (t < n)
                        v[t] = __fadd_rn(up ? v[t + n] : v[t], __shfl_xor_sync(kFull, up ? v[t] : v[t + n], o));
            }
            v[0] = __fadd_rn(v[0], __shfl_xor_sync(kFull, v[0], 2));
            v[0] = __fadd_rn(v[0], __shfl_xor_sync(kFull, v[0], 1));
            const float got = __shfl_sync(kFull, v[0], 4 * (lane & 7));
            if ((lane & 24) == b) mine = got;
        }
        return mine;
    }
}

constexpr int kPoolSlots = 4;
__host__ __device__ inline int pool_entries(int L) { return L <= 32 ? 32 : L <= 64 ? 64 : 128; }

// the id of the pool's first entry not yet expanded (slot, lane src, low word lo), or -1
template <int MAXS>
__device__ __forceinline__ int pool_next(const uint64_t (&pk)[MAXS], int& slot, int& src, uint32_t& lo) {
    slot = -1;
    unsigned open = 0u;
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
        if (slot < 0) {
            open = __ballot_sync(kFull, ((uint32_t)pk[s] & 1u) == 0u);
            if (open) slot = s;
        }
    }
    if (slot < 0) return -1;
    src = __ffs(open) - 1;
    lo = (uint32_t)pk[0];
#pragma unroll
    for (int s = 1; s < MAXS; ++s)
        if (slot == s) lo = (uint32_t)pk[s];
    return (int)(__shfl_sync(kFull, lo, src) >> 1);
}

// One candidate key per lane (the empty key: none) into the pool of beam_search: those that beat entry
// L - 1 enter together. pk and pool: the pool's registers and its copy in shared memory.
template <int MAXS>
__device__ __forceinline__ void pool_insert(uint64_t (&pk)[MAXS], uint64_t* pool, uint64_t cand, int L, int lane) {
    bool valid = cand < pool[L - 1];
    __syncwarp();
    if (__ballot_sync(kFull, valid) == 0u) return;
    // rank of the candidate among the pool's entries: halving steps over its 32, 64 or 128
    // slots (a valid candidate ranks below the last one: it beats entry L - 1). An entry
    // equal but for the mark means it is pooled already (the lossy table let it in).
    int pos = 0;
#pragma unroll
    for (int st = 16 * MAXS; st > 0; st >>= 1)
        if (pool[pos + st - 1] < cand) pos += st;
    if (valid && (pool[pos] | 1ull) == (cand | 1ull)) valid = false;
    unsigned vm = __ballot_sync(kFull, valid);
    if (vm == 0u) return;
    // the candidates are distinct: rank among them, and each pool entry's shift
    int crank = pos, shift[MAXS];
#pragma unroll
    for (int s = 0; s < MAXS; ++s) shift[s] = 0;
    do {
        const uint64_t cj = shfl64(cand, __ffs(vm) - 1);
        vm &= vm - 1;
        crank += cj < cand ? 1 : 0;
#pragma unroll
        for (int s = 0; s < MAXS; ++s) shift[s] += cj < pk[s] ? 1 : 0;
    } while (vm);
    // merged order: pool entry e goes to e + shift, a candidate to its rank among both
    __syncwarp();
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
        const int e = 32 * s + lane + shift[s];
        if (shift[s] != 0 && pk[s] != kEmptyKey && e < L) pool[e] = pk[s];
    }
    if (valid && crank < L) pool[crank] = cand;
    __syncwarp();
#pragma unroll
    for (int s = 0; s < MAXS; ++s) pk[s] = pool[32 * s + lane];
}

// Alg. 1 over one graph whose rows are Xt[v] / adj[v * M] for local ids v < nt. Keys carry
// global ids (local + id_off). The pool C (<= L <= 32 * MAXS entries, sorted by (delta, id)) lives in
// registers: entry e = 32 s + lane is pk[s] of that lane; pool[] in shared memory holds a copy. An
// entry's low word is id << 1 | expanded (ids are below 2^31), so entries of different ids order by
// (delta, id) whatever their marks, and the empty key (all ones) reads as expanded. Slots past the
// pool's size, and past L, hold the empty key, so pool[L - 1] is the key a candidate has to beat.
// The candidates of an expansion that beat it enter together: each finds its rank among the pool
// entries by a binary search of the copy, its rank among the other candidates and every pool
// entry's shift come from one loop over them, and one scatter through shared memory writes the
// merged pool. (Inserting them one by one, a ballot and a shift of all slots each, took half of the
// kernel's instructions at L = 48.)
// Returns the pool size and leaves the keys (delta, id) in pool[0 .. size).
// scratch: 32 ints of shared memory for the compacted neighbour ids.
template <int METRIC, bool SMALLD, typename RT, int MAXS, bool SKIP>
__device__ __forceinline__ int beam_search(const RT* __restrict__ Xt, const float* __restrict__ invt, const int32_t* __restrict__ adj,
                           int M, int nt, int ep, int id_off, const Query& Q, float qinv, int d, int L, uint64_t* pool,
                           uint16_t* ht, int htbits, int32_t* scratch, WarpCounters& ctr, int* status,
                           bool dedupe = true) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    if (ep < 0 || ep >= nt || L < 1 || L > 32 * MAXS) {
        if (lane == 0) atomicOr(status, kErrBounds);
        return 0;
    }
    const VisitedHash H(nt, htbits);
    ht_clear(ht, htbits, lane);
    if (lane == 0) scratch[0] = ep;
    uint64_t pk[MAXS];
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
        pk[s] = kEmptyKey;
        pool[32 * s + lane] = kEmptyKey;
    }
    __syncwarp();
    {
        const float dd = rows_delta<METRIC, SMALLD, RT, SKIP>(Xt, scratch, 1, Q, d, lane);
        if (lane == 0) {
            const float inv = (METRIC == FGIM_COSINE) ? __fmul_rn(qinv, invt[ep]) : 1.f;
            pk[0] = mkkey(delta_finish<METRIC>(dd, inv), (int32_t)((uint32_t)(ep + id_off) << 1));
            pool[0] = pk[0];
            H.add(ht, ep);
        }
        __syncwarp();
    }
    // every vertex is expanded at most once, so nt + 1 iterations always suffice; status[1],
    // when positive, is a smaller expansion budget (a test hook for the timeout path)
    bool done = false;
    const int hop_budget = status[1];
    const unsigned budget = hop_budget > 0 ? (unsigned)hop_budget : (unsigned)nt + 1u;
    unsigned it = 0, ndc = 1;
    for (; it <= (unsigned)nt; ++it) {
        int slot, src;
        uint32_t lo;
        const int id = pool_next<MAXS>(pk, slot, src, lo);
        if (id < 0) {
            done = true;
            break;
        }
        if (it >= budget) break;
        const int u = id - id_off;
        if (lane == src) {
#pragma unroll
            for (int s = 0; s < MAXS; ++s)
                if (slot == s) pk[s] |= 1ull;
            reinterpret_cast<uint32_t*>(pool)[2 * (32 * slot + lane)] = lo | 1u;   // the copy's mark
        }
        const int32_t* row = adj + (long long)u * M;
        for (int c0 = 0; c0 < M; c0 += 32) {
            int v = (c0 + lane < M) ? row[c0 + lane] : -1;
            if (v >= nt) {
                atomicOr(status, kErrBounds);
                v = -1;
            }
            // a neighbour listed twice is evaluated once (the lowest lane keeps it); skipped
            // (dedupe false) when the caller knows that no 32-entry chunk of a row repeats an id
            if (dedupe) {   // warp-uniform: every lane takes the match
                const unsigned same = __match_any_sync(kFull, v);
                if ((same & lt) != 0u) v = -1;
            }
            if (v >= 0 && H.seen(ht, v)) v = -1;
            const unsigned m = __ballot_sync(kFull, v >= 0);
            if (m == 0u) continue;
            const int U = __popc(m);
            if (v >= 0) scratch[__popc(m & lt)] = v;
            __syncwarp();
            const float dd = rows_delta<METRIC, SMALLD, RT, SKIP>(Xt, scratch, U, Q, d, lane);
            uint64_t cand = kEmptyKey;
            if (lane < U) {
                const int32_t w = scratch[lane];
                const float inv = (METRIC == FGIM_COSINE) ? __fmul_rn(qinv, invt[w]) : 1.f;
                cand = mkkey(delta_finish<METRIC>(dd, inv), (int32_t)((uint32_t)(w + id_off) << 1));
            }
            ndc += (unsigned)U;
            __syncwarp();   // scratch has been read
            pool_insert<MAXS>(pk, pool, cand, L, lane);
        }
    }
    if (!done && lane == 0) atomicOr(status, kErrTimeout);
    ctr.ndc += ndc;
    ctr.hops += it;
    int n = 0;
    __syncwarp();
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
        n += __popc(__ballot_sync(kFull, pk[s] != kEmptyKey));
        if (pk[s] != kEmptyKey) pool[32 * s + lane] = (pk[s] & 0xffffffff00000000ull) | ((uint32_t)pk[s] >> 1);
    }
    __syncwarp();
    return n;
}

__device__ __forceinline__ void warp_add_counters(const WarpCounters& c, unsigned long long* out) {
    if (lane_id() == 0 && out) {
        atomicAdd(out + 0, (unsigned long long)c.ndc);
        atomicAdd(out + 1, (unsigned long long)c.hops);
    }
}

// The items (queries, rows) of a beam-search launch: a warp starts with its own and takes further ones
// from *next, which counts the items handed out so, until it passes the last.
__device__ __forceinline__ long long first_item() {
    return (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
}
template <bool MORE>   // false: one item per warp
__device__ __forceinline__ long long next_item(unsigned long long* next) {
    if (!MORE || !next) return 0x7fffffffffffffffLL;
    unsigned long long v = 0;
    if (lane_id() == 0) v = atomicAdd(next, 1ull);
    __syncwarp();
    return (long long)shfl64(v, 0) + (long long)gridDim.x * (blockDim.x >> 5);
}

// shared-memory layout of one warp; all offsets multiples of 16 bytes
struct WarpLayout {
    int q, pool, ht, res, scratch, bytes;
};

__host__ __device__ inline int align16(int x) { return (x + 15) & ~15; }

// qrow: the query is kept in shared memory (rows wider than 128 coordinates)
__host__ __device__ inline WarpLayout warp_layout(int d, int L, int htbits, int kres, bool qrow) {
    WarpLayout w;
    int o = 0;
    w.q = o;
    if (qrow) o += align16(d * 4);
    w.pool = o;
    o += pool_entries(L) * 8;
    w.ht = o;
    o += (1 << htbits) * 2;
    w.res = o;
    o += align16(kres * 8);
    w.scratch = o;
    o += 32 * 4;
    w.bytes = o;
    return w;
}

// ---------------------------------------------------------------------------- host
// Warps per block when the autotuner has no choice for the workload. Rows of up to 128 coordinates: the
// launch keeps as many blocks as fit and every warp takes its items from a counter, so that no warp
// waits for the longest search of its block and the shape of a block does not matter (cross query of
// the 1M Sift-like merge 56.7 ms with one block of four warps per four rows, 54.6 ms with blocks of one
// warp, 52.5 ms so with one, two or four). Wider rows: one warp per block and per item; the loop over
// items costs registers that the loads in flight need there (120k, d = 768 BF16: 12.5 ms, 14.9 ms as
// resident blocks).
static inline int beam_warps(int d) { return d <= 128 ? 4 : 1; }

// Grid of a beam-search kernel over nq items of rows of d coordinates, and the counter its warps take
// their items from: *next (counters[kItemCounter], zeroed here) hands out the items after the first of every warp;
// nullptr: one item per warp (few items, wide rows).
template <typename K>
cudaError_t beam_grid(K kernel, int d, int wpb, size_t smem, long long nq, unsigned long long* counters, unsigned* blocks,
                      unsigned long long** next, cudaStream_t s) {
    const long long need = (nq + wpb - 1) / wpb;
    *blocks = (unsigned)need;
    *next = nullptr;
    if (d > 128) return cudaSuccess;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || need <= sms * 4LL) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, wpb * 32, smem)) != cudaSuccess) return e;
    if (per_sm < 1 || need <= (long long)per_sm * sms) return e;
    *blocks = (unsigned)(per_sm * sms);
    *next = counters + kItemCounter;
    return cudaMemsetAsync(*next, 0, sizeof(**next), s);
}

static inline int ht_bits_for(int L) {
    int want = 32 * L;
    int b = 9;
    while ((1 << b) < want && b < 12) ++b;
    return b;
}

#define FGIM_DISPATCH_METRIC_D(M, D, MACRO, RT, MS)                                              \
    do {                                                                                         \
        const bool small_ = (D) <= 128;                                                          \
        if ((M) == FGIM_L2SQ) {                                                                  \
            if (small_) MACRO(FGIM_L2SQ, true, RT, MS); else MACRO(FGIM_L2SQ, false, RT, MS);    \
        } else if ((M) == FGIM_IP) {                                                             \
            if (small_) MACRO(FGIM_IP, true, RT, MS); else MACRO(FGIM_IP, false, RT, MS);        \
        } else {                                                                                 \
            if (small_) MACRO(FGIM_COSINE, true, RT, MS); else MACRO(FGIM_COSINE, false, RT, MS); \
        }                                                                                        \
    } while (0)
// BF16 rows (d > 128 only: small rows gain little)
#define FGIM_DISPATCH_WIDE_MS(M, MACRO, RT, MS)                                                   \
    do {                                                                                         \
        if ((M) == FGIM_L2SQ) MACRO(FGIM_L2SQ, false, RT, MS);                                   \
        else if ((M) == FGIM_IP) MACRO(FGIM_IP, false, RT, MS);                                  \
        else MACRO(FGIM_COSINE, false, RT, MS);                                                  \
    } while (0)
#define FGIM_DISPATCH_ALL_WIDE(M, L, MACRO, RT)                                                  \
    do {                                                                                         \
        if ((L) <= 32) FGIM_DISPATCH_WIDE_MS(M, MACRO, RT, 1);                                   \
        else if ((L) <= 64) FGIM_DISPATCH_WIDE_MS(M, MACRO, RT, 2);                              \
        else FGIM_DISPATCH_WIDE_MS(M, MACRO, RT, kPoolSlots);                                    \
    } while (0)
// byte rows (d <= 128 only)
#define FGIM_DISPATCH_BYTES_MS(M, MACRO, MS)                                                     \
    do {                                                                                         \
        if ((M) == FGIM_L2SQ) MACRO(FGIM_L2SQ, true, uint8_t, MS);                               \
        else if ((M) == FGIM_IP) MACRO(FGIM_IP, true, uint8_t, MS);                              \
        else MACRO(FGIM_COSINE, true, uint8_t, MS);                                              \
    } while (0)
#define FGIM_DISPATCH_ALL_BYTES(M, L, MACRO)                                                     \
    do {                                                                                         \
        if ((L) <= 32) FGIM_DISPATCH_BYTES_MS(M, MACRO, 1);                                      \
        else if ((L) <= 64) FGIM_DISPATCH_BYTES_MS(M, MACRO, 2);                                 \
        else FGIM_DISPATCH_BYTES_MS(M, MACRO, kPoolSlots);                                       \
    } while (0)
// register pool of one slot (L <= 32), two (L <= 64) or kPoolSlots slots
#define FGIM_DISPATCH_ALL(M, D, L, MACRO, RT)                                                     \
    do {                                                                                         \
        if ((L) <= 32) FGIM_DISPATCH_METRIC_D(M, D, MACRO, RT, 1);                               \
        else if ((L) <= 64) FGIM_DISPATCH_METRIC_D(M, D, MACRO, RT, 2);                          \
        else FGIM_DISPATCH_METRIC_D(M, D, MACRO, RT, kPoolSlots);                                \
    } while (0)

}  // namespace fgim
