// Steps a1-a5 of the hot path: degrees, priority ranks, the projection
// graph G* with priority-sorted neighbour lists, the per-start orientation
// cut and exact wedge work, and the degree-binned schedule.
//
// Paper: Definition 3 (priority), Definition 4 (projection, Section 5.2),
// Section 4 (neighbour lists sorted by priority, early termination; the bin
// sort of Theorem 2's proof), Section 6.2 (workload of a start vertex and
// heaviest-first dynamic scheduling, Eq. 5).
#include <algorithm>
#include <vector>

#include "bfc_internal.cuh"

namespace bfc {

namespace {

constexpr int kT = 256;

inline unsigned blocks_for(int64_t n, int t = kT) {
    int64_t b = (n + t - 1) / t;
    if (b < 1) b = 1;
    return (unsigned)b;
}

// A prepared batch run without host synchronisation (the batch plan) checks
// the caller's CSR on the device; every later kernel of that run is given
// the error word and returns at once when the CSR failed the checks, so no
// kernel indexes with unchecked input.  Elsewhere the word is null.
__device__ __forceinline__ bool aborted(const int *guard) {
    return guard && (*(volatile const int *)guard & (kErrBadOffsets | kErrBadId));
}
// The row kernels set the word that they are guarded by (an edge to another
// graph of the batch), so threads that read it for themselves can differ.  A
// kernel whose warps or CTAs work together leaves by one decision for all of
// them: called by every thread of the warp, of the CTA.
__device__ __forceinline__ bool aborted_warp(const int *guard) {
    return __any_sync(0xffffffffu, aborted(guard));
}
__device__ __forceinline__ bool aborted_cta(const int *guard) {
    return __syncthreads_or(aborted(guard));
}

// ----- validation and a1: degrees ----------------------------------------------
// One pass over the caller's arrays (always on: every later index depends on
// it): the offsets with the U degrees, and the ids with the L degrees.  An id
// outside [0, l) is reported and counted nowhere.
__global__ void k_check_input(const int32_t *__restrict__ off, const int32_t *__restrict__ adj, int32_t r, int32_t l,
                              int64_t m, int32_t *deg_u, int32_t *deg_l, int *err) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t u = i0; u <= r; u += stride) {
        const int32_t o = off[u];
        if (u == 0 && o != 0) atomicOr(err, kErrBadOffsets);
        if (u < r) {
            const int32_t e = off[u + 1];
            if (e < o) atomicOr(err, kErrBadOffsets);
            deg_u[u] = e - o;
        }
        if (u == r && (int64_t)o != m) atomicOr(err, kErrBadOffsets);
    }
    for (int64_t k = i0; k < m; k += stride) {
        const int32_t v = adj[k];
        if (v < 0 || v >= l) atomicOr(err, kErrBadId);
        else atomicAdd(&deg_l[v], 1);
    }
}

// ----- a2: priority ranks ----------------------------------------------------
// Both layers in one sort: the key is (layer, graph of a batch, degree), the
// value the global id (L vertex v -> v, U vertex u -> l + u, ascending before the
// sort), so the stable sort's positions are the ids of G*: L first, each layer
// (each graph's part of it) by (degree, id), Definition 3's order.  A degree
// that does not fit its bits belongs to a row with duplicate edges that the
// validation rejects; it is cut off in the key only.
__device__ __forceinline__ int32_t graph_of(const int32_t *start, int32_t num_graphs, int32_t id) {
    int32_t lo = 0, hi = num_graphs;   // last g with start[g] <= id
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (start[mid] <= id) lo = mid; else hi = mid;
    }
    return lo;
}

__global__ void k_rank_keys(const int32_t *__restrict__ deg_l, const int32_t *__restrict__ deg_u, int32_t l,
                            int32_t n, const int32_t *__restrict__ gl, const int32_t *__restrict__ gu,
                            int32_t num_graphs, int bdeg, int blayer, uint64_t *keys,
    const int *guard = nullptr) {
    if (aborted(guard)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool in_u = i >= l;
    const int32_t id = in_u ? (int32_t)(i - l) : (int32_t)i;
    const uint64_t d = (uint64_t)(uint32_t)(in_u ? deg_u[id] : deg_l[id]), top = (1ull << bdeg) - 1;
    uint64_t key = (d < top ? d : top) | ((uint64_t)(in_u ? 1 : 0) << blayer);
    if (gl) key |= (uint64_t)graph_of(in_u ? gu : gl, num_graphs, id) << bdeg;
    keys[i] = key;
}

// ranks, the degree of every G* vertex (32 bits, and 64 for the offsets' scan)
// and the largest degree of each layer: top[0] L, top[1] U
__global__ void __launch_bounds__(kT) k_ranks(const int32_t *__restrict__ order, const int32_t *__restrict__ deg_l,
                                              const int32_t *__restrict__ deg_u, int32_t l, int32_t n,
                                              int32_t *rank_l, int32_t *rank_u, int32_t *deg_star, int64_t *deg64,
                                              unsigned long long *top,
    const int *guard = nullptr) {
    if (aborted_cta(guard)) return;
    __shared__ int32_t best[2];
    if (threadIdx.x < 2) best[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const int32_t id = order[i];
        const bool in_u = id >= l;
        const int32_t d = in_u ? deg_u[id - l] : deg_l[id];
        if (in_u) rank_u[id - l] = (int32_t)(i - l); else rank_l[id] = (int32_t)i;
        deg_star[i] = d;
        deg64[i] = d;
        if (d > best[in_u]) atomicMax(&best[in_u], d);
    }
    __syncthreads();
    if (threadIdx.x < 2 && best[threadIdx.x] > 0) atomicMax(top + threadIdx.x, (unsigned long long)best[threadIdx.x]);
}

// ----- a3: projection + sorted adjacency -------------------------------------
// ---- U side row by row.  Row u of the caller's CSR becomes G* row l + rank_u[u]
// (its slots start at off_star[l + rank_u[u]]); inside the row the neighbours
// go in ascending L rank.  The ranks of a row are distinct (E is a set), so
// any ordering method gives the same layout.  Tiers by degree:
//   d <= 32            one warp (eight lanes up to 8 neighbours), each lane's
//                      position = the lanes below it;
//   32 < d <= 256      one warp, bitonic sort of 32-bit (rank, index) keys in
//                      registers where the ranks have at most 24 bits;
//   256 < d            one CTA (256 threads up to 4,096 neighbours, 1,024 above),
//                      a bitmap of the L ranks of the row's graph, whose prefix
//                      popcounts are the positions, where that range is at most
//                      524,288 ranks (80 KB with the prefixes: two CTAs share an
//                      SM; wider bitmaps have not been measured) and duplicate
//                      edges are rejected anyway (a repeated bit has no position
//                      of its own).
// Otherwise:
//   32 < d <= 256      (ranges above 2^24 ranks) one warp, bitonic sort of
//                      (rank, slot) in its shared memory;
//   256 < d <= 4,096   (ranges above 524,288, validate = 0) one CTA, bitonic sort
//                      of (rank, slot) in shared memory;
//   d > 4,096          (likewise; a few hundred rows) one radix sort of their
//                      edges.  A plan, which cannot read their number, takes the
//                      bitmap with validate = 0 too.
// Each tier also writes the swapped key (rank_l, rank_u) at the U-side
// position; U-side order is ascending in rank_u, so the stable sort of those
// keys on the rank_l bits yields the L side.  The sort carries each key's
// U-side position (its index before the sort).
constexpr int kRowWarpMax = 32;
constexpr int kRowWarpSortMax = 256;
constexpr int kRowCtaMax = 4096;
constexpr int kRowCtaThreads = 256;
constexpr int32_t kRowBitmapMax = 1 << 19;   // L ranks of one bitmap
constexpr int kRowTiers = 5;   // warp sort, bitmap (256 threads), bitmap (1,024), CTA sort, radix
constexpr int kRedWords = 12 + 4;   // statistics, two queue and five tier counters

struct URowOut {
    int64_t m;
    int32_t l;
    int bu;
    const int64_t *off_star;
    int32_t *adj_star, *eid_star, *rows_star;
    uint64_t *keys2;
    int *err;
    int dup_bit;     // what a duplicate edge sets: kErrDuplicate (validate) or kErrParallel
    __device__ __forceinline__ void put(int32_t ru, int64_t pos, int32_t rl, int32_t slot) const {
        const int64_t k = off_star[l + ru] - m + pos;   // U-side position
        adj_star[m + k] = rl;
        eid_star[m + k] = slot;
        rows_star[m + k] = l + ru;
        keys2[k] = ((uint64_t)(uint32_t)rl << bu) | (uint64_t)(uint32_t)ru;
    }
};

// A warp takes `span` rows (their offsets and ranks are one load per lane; 32
// where there are enough rows for every warp of the device, else down to 4),
// then four rows of at most 8 neighbours at a time, then the longer ones one by
// one.  With 32 rows a warp, 2,000 rows were 63 warps walking 32 rows in turn.
__global__ void k_u_rows_warp(const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
                              const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
                              int32_t r, int span, const int32_t *__restrict__ gl,
                              const int32_t *__restrict__ gu, int32_t num_graphs, URowOut o,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 3, j = lane & 7;
    bool cross = false;   // a batch: an L rank outside the row's graph
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u0 = w0 * span; u0 < r; u0 += nw * span) {
        const int64_t u = u0 + lane;
        int32_t b = 0, d = 0, ru = 0, lo = 0, hi = o.l;
        if (u < r && lane < span) {
            b = off_u[u];
            d = off_u[u + 1] - b;
            if (d > 0 && d <= kRowWarpMax) {
                ru = rank_u[u];
                if (gl) {
                    const int32_t gg = graph_of(gu, num_graphs, (int32_t)u);
                    lo = gl[gg];
                    hi = gl[gg + 1];
                }
            }
        }
        uint32_t left = __ballot_sync(0xffffffffu, d > 0 && d <= 8);
        while (left) {   // four short rows, one per group of eight lanes
            int src = 32;
            for (int k = 0; k < 4; ++k) {
                if (k == g && left) src = __ffs((int)left) - 1;
                left &= left - 1;
            }
            const int32_t bk = __shfl_sync(0xffffffffu, b, src & 31), rk = __shfl_sync(0xffffffffu, ru, src & 31);
            int32_t dk = __shfl_sync(0xffffffffu, d, src & 31);
            if (src > 31) dk = 0;
            const int32_t lok = __shfl_sync(0xffffffffu, lo, src & 31), hik = __shfl_sync(0xffffffffu, hi, src & 31);
            const int32_t rl = j < dk ? rank_l[adj_u[bk + j]] : 0x7fffffff;
            cross |= j < dk && (rl < lok || rl >= hik);
            int pos = 0;
            bool dup = false;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int32_t ok = __shfl_sync(0xffffffffu, rl, (g << 3) + k);
                // ties (duplicate edges) are broken by lane, so positions stay distinct
                pos += (ok < rl || (ok == rl && k < j)) ? 1 : 0;
                dup |= ok == rl && k != j;
            }
            if (j < dk) {
                if (dup) atomicOr(o.err, o.dup_bit);
                o.put(rk, pos, rl, bk + j);
            }
        }
        left = __ballot_sync(0xffffffffu, d > 8 && d <= kRowWarpMax);
        while (left) {
            const int src = __ffs((int)left) - 1;
            left &= left - 1;
            const int32_t bk = __shfl_sync(0xffffffffu, b, src), dk = __shfl_sync(0xffffffffu, d, src);
            const int32_t rk = __shfl_sync(0xffffffffu, ru, src);
            const int32_t lok = __shfl_sync(0xffffffffu, lo, src), hik = __shfl_sync(0xffffffffu, hi, src);
            const int32_t rl = lane < dk ? rank_l[adj_u[bk + lane]] : 0x7fffffff;
            cross |= lane < dk && (rl < lok || rl >= hik);
            int pos = 0;
            bool dup = false;
            for (int k = 0; k < dk; ++k) {
                const int32_t ok = __shfl_sync(0xffffffffu, rl, k);
                pos += (ok < rl || (ok == rl && k < lane)) ? 1 : 0;
                dup |= ok == rl && k != lane;
            }
            if (lane < dk) {
                if (dup) atomicOr(o.err, o.dup_bit);
                o.put(rk, pos, rl, bk + lane);
            }
        }
    }
    if (cross) atomicOr(o.err, kErrBadId);
}

// Ascending bitonic sort of 32 * R keys held by a warp, key lane * R + r in
// register r: strides below R are exchanges inside a lane, the others one
// shuffle per key.
template <int R>
__device__ __forceinline__ void warp_sort(uint32_t (&key)[R], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= R) {
                // ascending where bit k of the index is clear; the lower of a
                // pair keeps the smaller key there
                const bool keep_min = ((lane * R) & k) == 0 ? ((lane * R) & j) == 0 : ((lane * R) & j) != 0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, key[r], j / R);
                    key[r] = keep_min ? min(key[r], o) : max(key[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if ((r & j) == 0) {
                        const bool up = k < R ? (r & k) == 0 : ((lane * R) & k) == 0;
                        const uint32_t a = key[r], c = key[r | j];
                        key[r] = up ? min(a, c) : max(a, c);
                        key[r | j] = up ? max(a, c) : min(a, c);
                    }
                }
            }
        }
    }
}

// one row of at most 32 * R neighbours; `buf` (32 * R keys of this warp) turns
// the sorted order back into consecutive lanes for the stores
template <int R>
__device__ __forceinline__ void warp_sort_row(const int32_t *adj_u, const int32_t *rank_l, int32_t b, int32_t d,
                                              int32_t ru, int32_t base, int32_t len, uint32_t *buf, int lane,
                                              const URowOut &o) {
    uint32_t key[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * 32 + lane;
        const uint32_t k = i < d ? (uint32_t)(rank_l[adj_u[b + i]] - base) : 0xffffffu;
        if (i < d && k >= (uint32_t)len) atomicOr(o.err, kErrBadId);   // an edge to another graph of the batch
        key[r] = i < d ? (k << 8) | (uint32_t)i : 0xffffffffu;
    }
    warp_sort<R>(key, lane);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) buf[lane * R + r] = key[r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = r * 32 + lane;
        if (i < d) {
            const uint32_t k = buf[i];
            if (i > 0 && (buf[i - 1] >> 8) == (k >> 8)) atomicOr(o.err, o.dup_bit);
            o.put(ru, i, base + (int32_t)(k >> 8), b + (int32_t)(k & 0xffu));
        }
    }
}

// rows of 33 to 256 neighbours, L ranks (within a batch's graph) of at most 24
// bits (a rank of all ones in 24 bits with index 255 equals the padding key, and
// then no key is padding)
__global__ void __launch_bounds__(kRowCtaThreads) k_u_rows_warp_reg(
    const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
    const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
    const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev,
    const int32_t *__restrict__ gl, const int32_t *__restrict__ gu, int32_t num_graphs, URowOut o,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    __shared__ uint32_t buf[kRowCtaThreads / 32][kRowWarpSortMax];
    const int lane = threadIdx.x & 31;
    uint32_t *wb = buf[threadIdx.x >> 5];
    const int32_t nrows = *nrows_dev;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = w0; i0 < nrows; i0 += nw) {
        const int32_t u = rows[i0];
        const int32_t b = off_u[u], d = off_u[u + 1] - b, ru = rank_u[u];
        int32_t base = 0, len = o.l;
        if (gl) {
            const int32_t g = graph_of(gu, num_graphs, u);
            base = gl[g];
            len = gl[g + 1] - base;
        }
        if (d <= 64) warp_sort_row<2>(adj_u, rank_l, b, d, ru, base, len, wb, lane, o);
        else if (d <= 128) warp_sort_row<4>(adj_u, rank_l, b, d, ru, base, len, wb, lane, o);
        else warp_sort_row<8>(adj_u, rank_l, b, d, ru, base, len, wb, lane, o);
    }
}

// ascending bitonic sort of np (a power of two) values by the calling warp
__device__ __forceinline__ void warp_bitonic(uint64_t *buf, int np, int lane) {
    for (int k = 2; k <= np; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < np; i += 32) {
                const int ij = i ^ j;
                if (ij > i) {
                    const uint64_t a = buf[i], c = buf[ij];
                    if ((a > c) == ((i & k) == 0)) { buf[i] = c; buf[ij] = a; }
                }
            }
            __syncwarp();
        }
    }
}

__global__ void __launch_bounds__(kRowCtaThreads) k_u_rows_warp_sort(
    const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
    const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
    const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev, URowOut o,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    const int32_t nrows = *nrows_dev;
    __shared__ uint64_t buf[kRowCtaThreads / 32][kRowWarpSortMax];
    const int lane = threadIdx.x & 31;
    uint64_t *wb = buf[threadIdx.x >> 5];
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i0 = w0; i0 < nrows; i0 += nw) {
        const int32_t u = rows[i0];
        const int32_t b = off_u[u], d = off_u[u + 1] - b;
        int np = 64;
        while (np < d) np <<= 1;
        for (int i = lane; i < np; i += 32)
            wb[i] = i < d ? ((uint64_t)(uint32_t)rank_l[adj_u[b + i]] << 32) | (uint32_t)(b + i) : ~0ull;
        __syncwarp();
        warp_bitonic(wb, np, lane);
        const int32_t ru = rank_u[u];
        for (int i = lane; i < d; i += 32) {
            const uint64_t vv = wb[i];
            const int32_t rl = (int32_t)(vv >> 32);
            if (i > 0 && (int32_t)(wb[i - 1] >> 32) == rl) atomicOr(o.err, o.dup_bit);
            o.put(ru, i, rl, (int32_t)(uint32_t)vv);
        }
        __syncwarp();   // the buffer is reused by the warp's next row
    }
}

__global__ void __launch_bounds__(kRowCtaThreads) k_u_rows_cta(
    const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
    const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
    const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev, URowOut o,
    const int *guard = nullptr) {
    if (aborted_cta(guard)) return;
    const int32_t nrows = *nrows_dev;
    __shared__ uint64_t buf[kRowCtaMax];
    for (int64_t i0 = blockIdx.x; i0 < nrows; i0 += gridDim.x) {
        const int32_t u = rows[i0];
        const int32_t b = off_u[u], d = off_u[u + 1] - b;
        int np = 64;
        while (np < d) np <<= 1;
        // (rank, slot): slots are distinct, so the sort has no ties
        for (int i = threadIdx.x; i < np; i += kRowCtaThreads)
            buf[i] = i < d ? ((uint64_t)(uint32_t)rank_l[adj_u[b + i]] << 32) | (uint32_t)(b + i) : ~0ull;
        __syncthreads();
        for (int k = 2; k <= np; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < np; i += kRowCtaThreads) {
                    const int ij = i ^ j;
                    if (ij > i) {
                        const uint64_t a = buf[i], c = buf[ij];
                        if ((a > c) == ((i & k) == 0)) { buf[i] = c; buf[ij] = a; }
                    }
                }
                __syncthreads();
            }
        }
        const int32_t ru = rank_u[u];
        for (int i = threadIdx.x; i < d; i += kRowCtaThreads) {
            const uint64_t vv = buf[i];
            const int32_t rl = (int32_t)(vv >> 32);
            if (i > 0 && (int32_t)(buf[i - 1] >> 32) == rl) atomicOr(o.err, o.dup_bit);
            o.put(ru, i, rl, (int32_t)(uint32_t)vv);
        }
        __syncthreads();   // buf is reused by the next row
    }
}

// lists of the rows of every tier above 32 neighbours (any order: every row
// is written to its own slots); one atomic per warp and list.  lists[t * r ...]:
// tier 0 warp sort, 1 and 2 bitmap, 3 CTA sort, 4 radix.  `range`: the L ranks of
// a single graph (a batch's row: its graph's); bitmaps only where `bitmaps`
// (2: above 4,096 neighbours only), and tier 2 only where `wide_tier`.
__global__ void k_row_tiers(const int32_t *__restrict__ off_u, int32_t r, int32_t range,
                            const int32_t *__restrict__ gu, const int32_t *__restrict__ gl, int32_t num_graphs,
                            int bitmaps, int wide_tier, int32_t *lists, int32_t *counts,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (int64_t u0 = (int64_t)blockIdx.x * blockDim.x; u0 < r; u0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = u0 + threadIdx.x;
        const int32_t d = u < r ? off_u[u + 1] - off_u[u] : 0;
        int tier = d <= kRowWarpMax ? -1 : 0;
        if (d > kRowWarpSortMax) {
            int32_t len = range;
            if (gl) {
                const int32_t g = graph_of(gu, num_graphs, (int32_t)u);
                len = gl[g + 1] - gl[g];
            }
            tier = (bitmaps && len <= kRowBitmapMax) ? (d <= kRowCtaMax && bitmaps == 2 ? 3 : (d <= kRowCtaMax || !wide_tier ? 1 : 2))
                                                     : (d <= kRowCtaMax ? 3 : 4);
        }
        if (!__any_sync(0xffffffffu, tier >= 0)) continue;
#pragma unroll
        for (int t = 0; t < kRowTiers; ++t) {
            const uint32_t bm = __ballot_sync(0xffffffffu, tier == t);
            int32_t o = 0;
            if (lane == 0 && bm) o = atomicAdd(counts + t, __popc(bm));
            o = __shfl_sync(0xffffffffu, o, 0);
            if (tier == t) lists[(int64_t)t * r + o + __popc(bm & lt)] = (int32_t)u;
        }
    }
}

// U rows of more than 256 neighbours, one CTA per row: one bit per neighbour's
// L rank in a bitmap of its graph's L rank range (all L ranks of a single
// graph); a neighbour's position is the number of set bits below its rank.  A
// bit that is already set is a duplicate edge: it is reported, and one of the
// positions past the distinct ranks is written for it, so that every position
// of the row holds a valid id.  Replaces a bitonic sort (78 stages with a barrier each at 4,096
// neighbours) and, above 4,096, a radix sort of all such rows' edges.
template <int kThreads>
__global__ void __launch_bounds__(kThreads) k_u_rows_bitmap(
    const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
    const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
    const int32_t *__restrict__ rows, const int32_t *__restrict__ nrows_dev, int32_t range,
    const int32_t *__restrict__ gl, const int32_t *__restrict__ gu, int32_t num_graphs, URowOut o,
    const int *guard = nullptr) {
    if (aborted_cta(guard)) return;
    extern __shared__ __align__(16) uint32_t bm_smem[];   // bits[words], then prefix of each 4 words
    __shared__ int32_t part[kThreads / 32];
    __shared__ int32_t n_dup;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t nrows = *nrows_dev;
    for (int64_t i0 = blockIdx.x; i0 < nrows; i0 += gridDim.x) {
        const int32_t u = rows[i0];
        const int32_t b = off_u[u], d = off_u[u + 1] - b, ru = rank_u[u];
        int32_t base = 0, len = range;
        if (gl) {
            const int32_t g = graph_of(gu, num_graphs, u);
            base = gl[g];   // the graph's L ranks: [gl[g], gl[g + 1])
            len = gl[g + 1] - base;
        }
        const int quads = (len + 127) / 128;   // 16-byte units of the bitmap
        uint4 *const q4 = reinterpret_cast<uint4 *>(bm_smem);
        int32_t *const qpre = reinterpret_cast<int32_t *>(q4 + quads);
        for (int i = tid; i < quads; i += kThreads) q4[i] = make_uint4(0, 0, 0, 0);
        if (tid == 0) n_dup = 0;
        __syncthreads();
#pragma unroll 4
        for (int32_t i = tid; i < d; i += kThreads) {
            const int32_t rl = rank_l[adj_u[b + i]], k = rl - base;
            if ((uint32_t)k >= (uint32_t)len) {   // an edge to another graph of the batch
                atomicOr(o.err, kErrBadId);
                continue;
            }
            const uint32_t bit = 1u << (k & 31);
            if (atomicOr(&bm_smem[k >> 5], bit) & bit) {
                atomicOr(o.err, o.dup_bit);
                o.put(ru, d - 1 - atomicAdd(&n_dup, 1), rl, b + i);
            }
        }
        __syncthreads();
        // exclusive prefix of the quads' popcounts: a contiguous share per thread
        const int per = (quads + kThreads - 1) / kThreads;
        const int f = min(tid * per, quads), e = min(f + per, quads);
        int32_t sum = 0;
        for (int i = f; i < e; ++i) {
            const uint4 q = q4[i];
            qpre[i] = sum;
            sum += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
        }
        int32_t incl = sum;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, incl, dd);
            if (lane >= dd) incl += t;
        }
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        int32_t before = incl - sum;
        for (int w = 0; w < warp; ++w) before += part[w];
        for (int i = f; i < e; ++i) qpre[i] += before;
        __syncthreads();
#pragma unroll 4
        for (int32_t i = tid; i < d; i += kThreads) {
            const int32_t rl = rank_l[adj_u[b + i]], k = rl - base;
            if ((uint32_t)k >= (uint32_t)len) continue;
            const uint4 q = q4[k >> 7];
            const int w = (k >> 5) & 3;
            const uint32_t mine = w == 0 ? q.x : (w == 1 ? q.y : (w == 2 ? q.z : q.w));
            int32_t pos = qpre[k >> 7] + __popc(mine & ((1u << (k & 31)) - 1u));
            if (w > 0) pos += __popc(q.x);
            if (w > 1) pos += __popc(q.y);
            if (w > 2) pos += __popc(q.z);
            o.put(ru, pos, rl, b + i);
        }
        __syncthreads();   // the bitmap is reused by the next row
    }
}

__global__ void k_large_deg(const int32_t *__restrict__ off_u, const int32_t *__restrict__ large,
                            int32_t nlarge, int64_t *ldeg) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nlarge) return;
    ldeg[i] = off_u[large[i] + 1] - off_u[large[i]];
}

// one CTA per large row copies its edges with composite keys (rank_u, rank_l)
__global__ void k_large_keys(const int32_t *__restrict__ off_u, const int32_t *__restrict__ adj_u,
                             const int32_t *__restrict__ rank_u, const int32_t *__restrict__ rank_l,
                             const int32_t *__restrict__ large, const int64_t *__restrict__ loff,
                             int32_t nlarge, int bl, uint64_t *keys, int32_t *vals) {
    for (int64_t i0 = blockIdx.x; i0 < nlarge; i0 += gridDim.x) {
        const int32_t u = large[i0];
        const int64_t o = loff[i0], d = loff[i0 + 1] - o;
        const int32_t b = off_u[u];
        const uint64_t hi = (uint64_t)(uint32_t)rank_u[u] << bl;
        for (int64_t i = threadIdx.x; i < d; i += blockDim.x) {
            keys[o + i] = hi | (uint64_t)(uint32_t)rank_l[adj_u[b + i]];
            vals[o + i] = b + (int32_t)i;
        }
    }
}

__global__ void k_large_heads(const uint64_t *__restrict__ keys, int64_t n, int bl, int32_t *heads) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        heads[i] = (i == 0 || (keys[i] >> bl) != (keys[i - 1] >> bl)) ? (int32_t)i : 0;
}

__global__ void k_large_emit(const uint64_t *__restrict__ keys, const int32_t *__restrict__ vals,
                             const int32_t *__restrict__ row_first, int64_t n, int bl, URowOut o) {
    const uint64_t mask_l = (1ull << bl) - 1ull;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = keys[i];
        if (i > 0 && keys[i - 1] == key) atomicOr(o.err, o.dup_bit);
        o.put((int32_t)(key >> bl), i - row_first[i], (int32_t)(key & mask_l), vals[i]);
    }
}

// L-side slot i = (v, u): v's list in ascending U rank, with the edge's
// U-side position k.  Algorithm 2's runs come from the two positions of the
// edge, with no search: where v is the start (u has fewer neighbours than v) the
// run through u is the prefix of N(u) before v, which is as long as v's position
// in that list; where u is the start the run through v is as long as u's
// position in N(v).  The second kind is scattered to the U-side slot, whose
// plen the caller has set to zero (the row kernels' scattered stores would cost
// more than the clear).  Reads `off` at random (L2-resident: 8 bytes
// per vertex), writes 4 bytes at random for the U starts' middles only; a
// binary search of the middle's list per slot took 15.8 ms on a 300M-edge
// shopping graph.
// `dups` (validate = 0, where the caller answers for them): the edges of a
// duplicate group are neighbours on both sides, and each takes the first one's
// positions.
template <bool kRuns>
__global__ void k_emit_l_side(const uint64_t *__restrict__ keys2, const int32_t *__restrict__ vals2,
                              int64_t m, int bu, int32_t l, const int64_t *__restrict__ off, int32_t *adj_star,
                              int32_t *eid_star, int32_t *rows_star, int32_t *plen, int64_t *sbeg, int dups,
    const int *guard = nullptr) {
    if (aborted(guard)) return;
    const uint64_t mask_u = (1ull << bu) - 1ull;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = keys2[i];
        const int32_t k = vals2[i], v = (int32_t)(key >> bu), u = l + (int32_t)(key & mask_u);
        adj_star[i] = u;
        eid_star[i] = k;
        rows_star[i] = v;
        if (kRuns) {
            const int64_t bv = off[v], bu0 = off[u];
            int64_t first = i;
            if (dups && i > bv && keys2[i - 1] == key) {   // v's keys ascend from bv on
                int64_t lo = bv;
                while (lo < first) {
                    const int64_t mid = (lo + first) >> 1;
                    if (keys2[mid] < key) lo = mid + 1; else first = mid;
                }
            }
            // equal degrees: the U vertex has the higher priority
            if (off[u + 1] - bu0 < off[v + 1] - bv) {
                plen[i] = (int32_t)(m + vals2[first] - bu0);
                sbeg[i] = bu0;
            } else {
                plen[i] = 0;
                plen[m + k] = (int32_t)(first - bv);
            }
        }
    }
}

// ----- a4: orientation cut and per-start work ---------------------------------
// cut[x] = |{y in N(x): p(y) < p(x)}|.  Lists are ascending in priority and
// the degree of G* ids is non-decreasing inside a layer, so the cut is a
// lower bound on degree: for x in L a U neighbour of equal degree has higher
// priority (U ids > L ids); for x in U an L neighbour of equal degree is lower.
__device__ __forceinline__ int32_t cut_of(const int32_t *__restrict__ adj, const int32_t *__restrict__ deg_star,
                                          int64_t b, int32_t d, int32_t dx, bool in_u) {
    int32_t lo = 0, hi = d;
    while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1), dy = deg_star[adj[b + mid]];
        if (in_u ? dy <= dx : dy < dx) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// (Algorithm 3's run lengths need every cut first; Algorithm 2's k_work finds
// them as it goes.)
__global__ void k_cut(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                      const int32_t *__restrict__ deg_star, int32_t n, int32_t l, int32_t *cut, const int *guard) {
    if (aborted(guard)) return;
    int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const int64_t b = off[x];
    cut[x] = cut_of(adj, deg_star, b, (int32_t)(off[x + 1] - b), deg_star[x], x >= l);
}

// Algorithm 3: for slot e = (x, v) the ends are the w in N(v) with
// p(w) > p(x) and p(w) > p(v).  N(v) ascends in priority, so they form the
// suffix that starts after both x (x is in N(v)) and v's cut.
__global__ void k_slen(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                       const int32_t *__restrict__ rows, const int32_t *__restrict__ cut,
                       int64_t slots, int32_t *slen, int64_t *sbeg, const int *guard) {
    if (aborted(guard)) return;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < slots;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = rows[e];
        const int32_t v = adj[e];
        const int64_t b = off[v], d = off[v + 1] - b;
        int64_t lo = 0, hi = d;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (adj[b + mid] <= x) lo = mid + 1; else hi = mid;
        }
        const int64_t a = lo > cut[v] ? lo : (int64_t)cut[v];
        slen[e] = (int32_t)(d - a);
        sbeg[e] = b + a;
    }
}

// work[x] = Σ plen over x's middle slots (the first cut[x] slots for
// Algorithm 2, every slot for Algorithm 3).  For Algorithm 2 the U-side middle
// slots (at or past `fill_from`) also get the start of their run, off[middle].
// A warp takes 32 starts and each lane walks its own where there are at most
// 24 slots (neighbouring lists share their sectors); the longer ones go to two
// queues for k_work_long, one per warp up to 4,096 slots and one per CTA above.
// (Ranks are by degree, so the long lists are neighbours: whatever takes several
// in a row has them all.)  With one warp per start the millions of one-slot
// starts of a sparse batch and the longest list of a skewed graph each took 2.5 ms.
constexpr int kWorkLane = 24;
constexpr int kWorkWarp = 4096;

__device__ __forceinline__ unsigned slot_work(const int64_t *off, const int32_t *adj, const int32_t *plen,
                                              int64_t e, bool fill, int64_t *sbeg) {
    if (fill) sbeg[e] = off[adj[e]];
    return (unsigned)plen[e];
}

__global__ void k_work(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                       const int32_t *__restrict__ deg_star, int32_t l, int32_t *cut,
                       const int32_t *__restrict__ plen, int32_t n, int all_slots, int64_t fill_from, int64_t *sbeg, uint64_t *work, int32_t *queue, int32_t *queued,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x0 = warp * 32; x0 < n; x0 += nwarps * 32) {
        const int64_t x = x0 + lane;
        int64_t b = 0;
        int32_t c = 0;
        if (x < n) {
            b = off[x];
            c = (int32_t)(off[x + 1] - b);
            if (!all_slots) {
                c = cut_of(adj, deg_star, b, c, deg_star[x], x >= l);
                cut[x] = c;
            }
        }
        unsigned long long s = 0;
        if (c <= kWorkLane) {
            const bool fill = b >= fill_from;
            for (int32_t j = 0; j < c; ++j) s += slot_work(off, adj, plen, b + j, fill, sbeg);
            if (x < n) work[x] = s;
        }
        // queue[0, n): the warps' from the front, the CTAs' from the back
        const uint32_t by_warp = __ballot_sync(0xffffffffu, c > kWorkLane && c <= kWorkWarp);
        const uint32_t by_cta = __ballot_sync(0xffffffffu, c > kWorkWarp);
        int32_t at = 0;
        if (lane == 0 && by_warp) at = atomicAdd(queued, __popc(by_warp));
        if (lane == 1 && by_cta) at = atomicAdd(queued + 1, __popc(by_cta));
        const int32_t at_w = __shfl_sync(0xffffffffu, at, 0), at_c = __shfl_sync(0xffffffffu, at, 1);
        const uint32_t lt = (1u << lane) - 1u;
        if (c > kWorkWarp) queue[n - 1 - at_c - __popc(by_cta & lt)] = (int32_t)x;
        else if (c > kWorkLane) queue[at_w + __popc(by_warp & lt)] = (int32_t)x;
    }
}

// Σ plen over slots b + j, b + j + W, ... of a list's first c, four loads at a
// time, and the runs' starts where `fill`
template <int W>
__device__ __forceinline__ unsigned long long walk_slots(const int64_t *__restrict__ off,
                                                         const int32_t *__restrict__ adj,
                                                         const int32_t *__restrict__ plen, int64_t b, int32_t j,
                                                         int32_t c, bool fill, int64_t *__restrict__ sbeg) {
    unsigned long long t = 0;
    for (; j < c; j += 4 * W) {
        unsigned len[4];
        int32_t mid[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = j + u * W < c;
            len[u] = in ? (unsigned)plen[b + j + u * W] : 0u;
            mid[u] = in && fill ? adj[b + j + u * W] : -1;
        }
        if (fill) {
            int64_t at[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) at[u] = mid[u] >= 0 ? off[mid[u]] : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (mid[u] >= 0) sbeg[b + j + u * W] = at[u];
        }
        t += (unsigned long long)len[0] + len[1] + len[2] + len[3];
    }
    return t;
}

constexpr int kWorkThreads = 512;
__global__ void __launch_bounds__(kWorkThreads) k_work_long(
    const int64_t *__restrict__ off, const int32_t *__restrict__ adj, const int32_t *__restrict__ cut,
    const int32_t *__restrict__ plen, int32_t n, int all_slots, int64_t fill_from, int64_t *sbeg, uint64_t *work,
    const int32_t *__restrict__ queue, const int32_t *__restrict__ queued,
    const int *guard = nullptr) {
    if (aborted_cta(guard)) return;
    __shared__ unsigned long long part[kWorkThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_warp = queued[0], n_cta = queued[1];
    for (int i = blockIdx.x; i < n_cta; i += gridDim.x) {
        const int32_t x = queue[n - 1 - i];
        const int64_t b = off[x];
        const int32_t c = all_slots ? (int32_t)(off[x + 1] - b) : cut[x];
        const bool fill = b >= fill_from;
        unsigned long long t = walk_slots<kWorkThreads>(off, adj, plen, b, (int32_t)threadIdx.x, c, fill, sbeg);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
        if (lane == 0) part[warp] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            t = 0;
            for (int w = 0; w < kWorkThreads / 32; ++w) t += part[w];
            work[x] = t;
        }
        __syncthreads();
    }
    for (int i = blockIdx.x * (kWorkThreads / 32) + warp; i < n_warp; i += gridDim.x * (kWorkThreads / 32)) {
        const int32_t x = queue[i];
        const int64_t b = off[x];
        const int32_t c = all_slots ? (int32_t)(off[x + 1] - b) : cut[x];
        const bool fill = b >= fill_from;
        unsigned long long t = walk_slots<32>(off, adj, plen, b, lane, c, fill, sbeg);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
        if (lane == 0) work[x] = t;
    }
}

// ----- a5: bins and schedule ---------------------------------------------------
// A core start (dense-core hybrid) with wedges is always a dense item: only
// dense items skip the core wedges and add the core pairs after the walk.
__device__ __forceinline__ bool forced_dense(int32_t x, int32_t l, int32_t core_lo_u, int32_t core_lo_l,
                                             uint64_t w) {
    return w > 0 && (x >= l ? x >= core_lo_u : x >= core_lo_l);
}

// Bins of a6: 0 dense (work > hash_max), 1 CTA hash (team_max < work <=
// hash_max), 2 team (warp_max < work <= team_max), 3 warp (0 < work <= warp_max).
// 5: of the warp bin, the starts of at most 32 wedges and 32 middles
// (Algorithm 2), which take one window and no table.
struct BinBounds {
    uint64_t warp_max, team_max, hash_max;
    int32_t l, core_lo_u, core_lo_l;
    const int32_t *cut;   // null: no bin 5
    __device__ __forceinline__ int of(int32_t x, uint64_t w) const {
        if (w > hash_max || forced_dense(x, l, core_lo_u, core_lo_l, w)) return 0;
        if (w > warp_max) return w > team_max ? 1 : 2;
        if (w == 0) return 4;
        return cut && w <= (uint64_t)kTinyMax && cut[x] <= kTinyMax ? 5 : 3;
    }
};

// The starts of each bin: counts[b] (and [4]: bins 0 to 2 together), bin 3 from
// the front of warp_items[n], bin 5 from its back, and the others in `heavy` (in
// no order; only the heavy ones, a few per cent of the starts with work, are
// then sorted).  A CTA takes 2,048 starts and reserves
// their room with one addition per list.
// With `stats` also: stats[0] += Σ work, stats[1] = max work, stats[2] +=
// starts above heavy_work, stats[11] = the error word, and of a batch gwork[g] +=
// the work of graph g (one addition per warp where its vertices lie in one
// graph, which all but a few warps' do).
constexpr int kBinTile = 8 * kT;
__global__ void __launch_bounds__(kT) k_bin_starts(const uint64_t *__restrict__ work, int32_t n, BinBounds bb,
                                                   unsigned long long *counts, int32_t *heavy, int32_t *warp_items,
                                                   unsigned long long *stats, uint64_t heavy_work,
                                                   const int32_t *__restrict__ gstar, unsigned long long *gwork,
    const int *guard = nullptr) {
    if (stats && guard && blockIdx.x == 0 && threadIdx.x == 0) stats[11] = (unsigned long long)*(volatile const int *)guard;
    if (aborted_cta(guard)) return;
    unsigned long long sum = 0, top = 0, above = 0;
    __shared__ int32_t cnt[6], at[3];   // at: this tile's room in heavy, warp front, warp back
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (int64_t x0 = (int64_t)blockIdx.x * kBinTile; x0 < n; x0 += (int64_t)gridDim.x * kBinTile) {
        if (threadIdx.x < 6) cnt[threadIdx.x] = 0;
        __syncthreads();
        int bin[8], place[8];   // place: among the tile's starts of the same list
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int64_t x = x0 + i * kT + threadIdx.x;
            const uint64_t w = x < n ? work[x] : 0;
            bin[i] = w > 0 ? bb.of((int32_t)x, w) : 4;
            sum += w;
            top = w > top ? w : top;
            above += w > heavy_work ? 1 : 0;
            if (gwork) {
                const int32_t g = x < n ? gstar[x] : -1;
                const int32_t g0 = __shfl_sync(0xffffffffu, g, 0);
                if (__all_sync(0xffffffffu, g == g0)) {
                    unsigned long long t = w;
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
                    if (lane == 0 && t) atomicAdd(gwork + g0, t);
                } else if (w) {
                    atomicAdd(gwork + g, (unsigned long long)w);
                }
            }
        }
        // cnt[0..2]: bins; cnt[3], cnt[5]: lists of their own; cnt[4]: the heavy list
#pragma unroll
        for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const uint32_t m = __ballot_sync(0xffffffffu, bin[i] == b);
                if (lane == 0 && m) atomicAdd(&cnt[b], __popc(m));
            }
            const uint32_t mh = __ballot_sync(0xffffffffu, bin[i] < 3), mw = __ballot_sync(0xffffffffu, bin[i] == 3),
                           mt = __ballot_sync(0xffffffffu, bin[i] == 5);
            int o = 0;
            if (lane == 0 && mh) o = atomicAdd(&cnt[4], __popc(mh));
            if (lane == 1 && mw) o = atomicAdd(&cnt[3], __popc(mw));
            if (lane == 2 && mt) o = atomicAdd(&cnt[5], __popc(mt));
            const int oh = __shfl_sync(0xffffffffu, o, 0), ow = __shfl_sync(0xffffffffu, o, 1),
                      ot = __shfl_sync(0xffffffffu, o, 2);
            place[i] = bin[i] < 3 ? oh + __popc(mh & lt) : (bin[i] == 3 ? ow + __popc(mw & lt) : ot + __popc(mt & lt));
        }
        __syncthreads();
        if (threadIdx.x < 6 && cnt[threadIdx.x] > 0) {
            const int32_t o = (int32_t)atomicAdd(counts + threadIdx.x, (unsigned long long)cnt[threadIdx.x]);
            if (threadIdx.x >= 3) at[threadIdx.x == 4 ? 0 : (threadIdx.x == 3 ? 1 : 2)] = o;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int32_t x = (int32_t)(x0 + i * kT + threadIdx.x);
            if (bin[i] < 3) heavy[at[0] + place[i]] = x;
            else if (bin[i] == 3) warp_items[at[1] + place[i]] = x;
            else if (bin[i] == 5) warp_items[n - 1 - at[2] - place[i]] = x;
        }
        __syncthreads();
    }
    if (stats) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, d);
            above += __shfl_xor_sync(0xffffffffu, above, d);
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, top, d);
            top = o > top ? o : top;
        }
        if (lane == 0) {
            if (sum) atomicAdd(stats, sum);
            if (top) atomicMax(stats + 1, top);
            if (above) atomicAdd(stats + 2, above);
        }
    }
}

// ascending key = descending work; forced dense starts first
__global__ void k_sched_keys(const uint64_t *__restrict__ work, const int32_t *__restrict__ heavy, int64_t n_heavy,
                             uint64_t maxw, int32_t l, int32_t core_lo_u, int32_t core_lo_l, uint64_t *keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_heavy) return;
    const int32_t x = heavy[i];
    keys[i] = forced_dense(x, l, core_lo_u, core_lo_l, work[x]) ? 0 : maxw - work[x];
}

// The same order for at most 4,096 heavy starts, by one CTA: a bitonic sort of
// (key, place) words in shared memory, one launch for the ten of a radix sort
// over so few keys.  A pair of elements less than 32 apart is one warp's, so only
// the wider strides need the CTA's barrier.
constexpr int kSchedSmall = 4096;
constexpr int kSchedPlaceBits = 12;
__global__ void __launch_bounds__(1024) k_sched_small(const uint64_t *__restrict__ work,
                                                      const int32_t *__restrict__ heavy, int n_heavy, uint64_t maxw,
                                                      int32_t l, int32_t core_lo_u, int32_t core_lo_l, int32_t *order) {
    __shared__ uint64_t buf[kSchedSmall];
    int np = 64;
    while (np < n_heavy) np <<= 1;
    for (int i = threadIdx.x; i < np; i += 1024) {
        uint64_t key = ~0ull;
        if (i < n_heavy) {
            const int32_t x = heavy[i];
            key = (forced_dense(x, l, core_lo_u, core_lo_l, work[x]) ? 0 : maxw - work[x]) << kSchedPlaceBits | (uint64_t)i;
        }
        buf[i] = key;
    }
    __syncthreads();
    for (int k = 2; k <= np; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < np; i += 1024) {
                const int ij = i ^ j;
                if (ij > i) {
                    const uint64_t a = buf[i], c = buf[ij];
                    if ((a > c) == ((i & k) == 0)) { buf[i] = c; buf[ij] = a; }
                }
            }
            // this stride, or the first of the next k, crosses warps
            if (j >= 32 || (j == 1 && k >= 32)) __syncthreads(); else __syncwarp();
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_heavy; i += 1024) order[i] = heavy[buf[i] & ((1u << kSchedPlaceBits) - 1u)];
}

// the dense chunks of start x (dense_chunk_end from offset 0 up); with `out`,
// each chunk's item is written there
__device__ __forceinline__ int32_t dense_chunks(int32_t x, int32_t l, int32_t cut, const int64_t *off,
                                                const int32_t *vbase, int2 *out = nullptr) {
    const int32_t lb = vbase ? vbase[x] : (x >= l ? l : 0);
    const int32_t R = x - lb;
    int32_t k = 0;
    for (int32_t lo = 0; lo < R; ++k) {
        int bits;
        const int32_t hi = dense_chunk_end(lo, R, cut, off, lb, &bits);
        if (out) out[k] = make_int2(x, dense_item_y(lo, bits));
        lo = hi;
    }
    return k;
}

// the only dense chunk of a start whose layer is no larger than one
__device__ __forceinline__ int2 one_dense_item(int32_t x, int32_t l, int32_t cut, const int64_t *off,
                                               const int32_t *vbase) {
    const int32_t lb = vbase ? vbase[x] : (x >= l ? l : 0);
    int bits = 4;
    if (x > lb) dense_chunk_end(0, x - lb, cut, off, lb, &bits);
    return make_int2(x, dense_item_y(0, bits));
}

__global__ void k_chunk_counts(const int32_t *__restrict__ order, int64_t n_dense, int32_t l,
                               const int32_t *__restrict__ cut, const int64_t *__restrict__ off,
                               const int32_t *__restrict__ vbase, int64_t *nch) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_dense) return;
    int32_t x = order[i];
    nch[i] = dense_chunks(x, l, cut[x], off, vbase);
}

// A start of the CTA-hash bin whose whole end range is one chunk of dense
// counters gets those instead of a table (Algorithm 2 only): clearing at most
// 192 KB costs a CTA about 1,500 clocks, a table with as many wedges 70 clocks
// per 32 of them against about 10.
__device__ __forceinline__ int2 hash_or_dense_item(int32_t x, int32_t l, int32_t cut, const int64_t *off,
                                                   const int32_t *vbase) {
    const int32_t lb = vbase ? vbase[x] : (x >= l ? l : 0);
    int bits;
    return make_int2(x, dense_chunk_end(0, x - lb, cut, off, lb, &bits) == x - lb ? dense_item_y(0, bits) : -1);
}

// starts in descending work order: dense (chunked; nch_scan null: one chunk
// each), CTA hash, team.  Here and above `cut` and `off` are the graph's bcut and boff.
__global__ void k_emit_items(const int32_t *__restrict__ order, int64_t n_dense, int64_t n_hash,
                             int64_t n_team, const int64_t *__restrict__ nch_scan,
                             int32_t l, const int32_t *__restrict__ cut, const int64_t *__restrict__ off,
                             const int32_t *__restrict__ vbase, int ends_above, int2 *cta_items,
                             int32_t *team_items) {
    const int64_t total_dense = nch_scan ? nch_scan[n_dense] : n_dense;
    const int64_t all = n_dense + n_hash + n_team;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < all;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t x = order[i];
        if (i < n_dense) {
            if (nch_scan) dense_chunks(x, l, cut[x], off, vbase, cta_items + nch_scan[i]);
            else cta_items[i] = one_dense_item(x, l, cut[x], off, vbase);
        } else if (i < n_dense + n_hash) {
            cta_items[total_dense + (i - n_dense)] =
                ends_above ? make_int2(x, -1) : hash_or_dense_item(x, l, cut[x], off, vbase);
        } else {
            team_items[i - n_dense - n_hash] = x;
        }
    }
}

// bcut and boff (see Graph).  With `err` only where the word tells of parallel
// edges, else copies of cut and off; `most` caps bcut.
__global__ void k_count_bounds(const uint64_t *__restrict__ work, const int32_t *__restrict__ cut,
                               const int64_t *__restrict__ off, int32_t n, int32_t most, const int *err,
                               int32_t *bcut, int64_t *boff) {
    const bool parallel = !err || (*err & kErrParallel);
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x <= n; x += (int64_t)gridDim.x * blockDim.x) {
        boff[x] = parallel ? x << 31 : off[x];
        if (x < n) bcut[x] = parallel ? (int32_t)(work[x] < (uint64_t)most ? work[x] : (uint64_t)most) : cut[x];
    }
}

// retry entries -(x+1): counted with dense chunks
__global__ void k_items_to_dense_retries(const int2 *__restrict__ items, int64_t n, int32_t *starts) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) starts[i] = -(items[i].x + 1);
}

// ----- chunk-boundary table for the dense bin ----------------------------------
__device__ __forceinline__ int64_t coff_base(int32_t v, int32_t l, int32_t u1, int32_t l1) {
    return v < l ? (int64_t)v * u1 : (int64_t)l * u1 + (int64_t)(v - l) * l1;
}

__global__ void k_coff_fill(const int64_t *__restrict__ off, int32_t l, int32_t u1, int32_t l1,
                            int64_t entries, int32_t *coff) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < entries;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t split = (int64_t)l * u1;
        const int32_t v = i < split ? (int32_t)(i / u1) : l + (int32_t)((i - split) / l1);
        coff[i] = (int32_t)(off[v + 1] - off[v]);
    }
}

// entry c of v = first position in N(v) whose neighbour rank is >= c * unit
__global__ void k_coff_slots(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                             const int32_t *__restrict__ rows, int64_t slots, int32_t l,
                             int32_t u1, int32_t l1, int32_t *coff) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < slots;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = rows[p];
        const int32_t lbe = v < l ? l : 0;
        const int64_t b = off[v];
        const int32_t cp = (adj[p] - lbe) / kChunkUnit;
        const int32_t cprev = p == b ? -1 : (adj[p - 1] - lbe) / kChunkUnit;
        const int64_t tb = coff_base(v, l, u1, l1);
        for (int32_t c = cprev + 1; c <= cp; ++c) coff[tb + c] = (int32_t)(p - b);
    }
}

// A batch's table.  The middles of every dense start with several chunks
// (one warp per start: its cut[x] lower-priority neighbours).
__global__ void k_coff_mark(const int32_t *__restrict__ order, int64_t n_dense, const int64_t *__restrict__ nch,
                            const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                            const int32_t *__restrict__ cut, int32_t *mark) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < n_dense; i += nw) {
        if (nch[i] <= 1) continue;
        const int32_t x = order[i];
        const int64_t e0 = off[x];
        for (int64_t e = e0 + lane; e < e0 + cut[x]; e += 32) mark[adj[e]] = 1;
    }
}

// entries of a marked v: the chunks of its graph's neighbour layer, plus one
// (the neighbours' layer range is that of any neighbour w: vend[w] - vbase[w])
__global__ void k_coff_sizes(const int32_t *__restrict__ mark, const int64_t *__restrict__ off,
                             const int32_t *__restrict__ adj, const int32_t *__restrict__ vbase,
                             const int32_t *__restrict__ vend, int32_t n, int64_t *cnt) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        int64_t c = 0;
        if (mark[v] && off[v + 1] > off[v]) {
            const int32_t w = adj[off[v]];
            c = (int64_t)(vend[w] - vbase[w] + kChunkUnit - 1) / kChunkUnit + 1;
        }
        cnt[v] = c;
    }
}

// every entry of v starts at "past the end of N(v)"
__global__ void k_coff_fill_var(const int64_t *__restrict__ off, const int64_t *__restrict__ cstart, int32_t n,
                                int32_t *coff) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = (int32_t)(off[v + 1] - off[v]);
        for (int64_t c = cstart[v]; c < cstart[v + 1]; ++c) coff[c] = d;
    }
}

// entry c of a marked v = first position in N(v) whose neighbour id is at
// least (first id of the neighbours' graph range) + c * unit
__global__ void k_coff_slots_var(const int64_t *__restrict__ off, const int32_t *__restrict__ adj,
                                 const int32_t *__restrict__ rows, int64_t slots,
                                 const int32_t *__restrict__ vbase, const int64_t *__restrict__ cstart,
                                 int32_t *coff) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < slots;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = rows[p];
        const int64_t tb = cstart[v], te = cstart[v + 1];
        if (te == tb) continue;
        const int64_t b = off[v];
        const int32_t lbe = vbase[adj[b]];
        const int32_t cp = (adj[p] - lbe) / kChunkUnit;
        const int32_t cprev = p == b ? -1 : (adj[p - 1] - lbe) / kChunkUnit;
        for (int32_t c = cprev + 1; c <= cp && tb + c < te; ++c) coff[tb + c] = (int32_t)(p - b);
    }
}

// the first entry of each middle of those starts, at the middle's slot
__global__ void k_coff_slot_bases(const int32_t *__restrict__ order, int64_t n_dense,
                                  const int64_t *__restrict__ nch, const int64_t *__restrict__ off,
                                  const int32_t *__restrict__ adj, const int32_t *__restrict__ cut,
                                  const int64_t *__restrict__ cstart, int32_t *ctb) {
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < n_dense; i += nw) {
        if (nch[i] <= 1) continue;
        const int32_t x = order[i];
        const int64_t e0 = off[x];
        for (int64_t e = e0 + lane; e < e0 + cut[x]; e += 32) ctb[e] = (int32_t)cstart[adj[e]];
    }
}

unsigned grid_stride_blocks(int64_t n) {
    int64_t b = (n + kT - 1) / kT;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return (unsigned)b;
}

// ----- batches prepared as one disjoint union ------------------------------------
__global__ void k_check_starts(const int32_t *__restrict__ start, int32_t num_graphs,
                               int32_t total, int *err, int32_t max_len = 0x7fffffff,
                               int *longest = nullptr) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= num_graphs;
         g += (int64_t)gridDim.x * blockDim.x) {
        if (g == 0 && start[0] != 0) atomicOr(err, kErrBadOffsets);
        if (g < num_graphs && (start[g + 1] < start[g] || start[g + 1] - start[g] > max_len))
            atomicOr(err, kErrBadOffsets);
        if (longest && g < num_graphs) atomicMax(longest, start[g + 1] - start[g]);
        if (g == num_graphs && start[g] != total) atomicOr(err, kErrBadOffsets);
    }
}

// Every edge must join a U and an L vertex of the same graph.  The row kernels
// that know their row's graph check its L ranks as they read them; this pass is
// for the tiers that do not (ranges above 524,288 ranks, validate = 0): one
// lookup of the row's graph, then its L ids against that graph's range.  A warp
// takes 32 rows (lanes on their own up to 24 neighbours, the warp together above).
__global__ void k_check_batch_rows(const int32_t *__restrict__ off, const int32_t *__restrict__ adj, int32_t r,
                                   const int32_t *__restrict__ gu, const int32_t *__restrict__ gl,
                                   int32_t num_graphs, int *err,
    const int *guard = nullptr) {
    if (aborted_warp(guard)) return;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int64_t u0 = warp * 32; u0 < r; u0 += nwarps * 32) {
        const int64_t u = u0 + lane;
        int32_t b = 0, d = 0, lo = 0, hi = 0;
        if (u < r) {
            b = off[u];
            d = off[u + 1] - b;
            const int32_t g = graph_of(gu, num_graphs, (int32_t)u);
            lo = gl[g];
            hi = gl[g + 1];
        }
        if (d <= kWorkLane)
            for (int32_t j = 0; j < d; ++j) { const int32_t v = adj[b + j]; bad |= v < lo || v >= hi; }
        uint32_t todo = __ballot_sync(0xffffffffu, d > kWorkLane);
        while (todo) {
            const int k = __ffs((int)todo) - 1;
            todo &= todo - 1;
            const int32_t bk = __shfl_sync(0xffffffffu, b, k), dk = __shfl_sync(0xffffffffu, d, k);
            const int32_t lk = __shfl_sync(0xffffffffu, lo, k), hk = __shfl_sync(0xffffffffu, hi, k);
#pragma unroll 8
            for (int32_t j = lane; j < dk; j += 32) { const int32_t v = adj[bk + j]; bad |= v < lk || v >= hk; }
        }
    }
    if (bad) atomicOr(err, kErrBadId);
}

// graph-major ranks: vertex x of G* belongs to the graph whose rank range
// holds it; vbase[x] = the first G* id of that graph in x's layer
__global__ void k_graph_star(int32_t r, int32_t l, const int32_t *__restrict__ gu,
                             const int32_t *__restrict__ gl, int32_t num_graphs, int32_t *gstar,
                             int32_t *vbase, int32_t *vend,
    const int *guard = nullptr) {
    if (aborted(guard)) return;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < (int64_t)r + l;
         x += (int64_t)gridDim.x * blockDim.x) {
        if (x < l) {
            const int32_t gg = graph_of(gl, num_graphs, (int32_t)x);
            gstar[x] = gg;
            vbase[x] = gl[gg];
            vend[x] = gl[gg + 1];
        } else {
            const int32_t gg = graph_of(gu, num_graphs, (int32_t)(x - l));
            gstar[x] = gg;
            vbase[x] = l + gu[gg];
            vend[x] = l + gu[gg + 1];
        }
    }
}

// slot -> owning vertex of G*, one warp per vertex
__global__ void k_rows_from_off(const int64_t *__restrict__ off, int32_t n, int32_t *rows) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = w; x < n; x += nw)
        for (int64_t p = off[x] + lane; p < off[x + 1]; p += 32) rows[p] = (int32_t)x;
}

}  // namespace

// the bin bounds that a schedule's three limits stand for
static BinBounds bin_bounds(const Graph *g, int32_t warp_max_work, int32_t team_max_work, int32_t hash_max_work) {
    const bool vpp = g->opt.orientation == 1;
    BinBounds bb;
    bb.warp_max = (uint64_t)warp_max_work;
    // Algorithm 3: ends concentrate on few high-priority vertices, so no start
    // gets dense counters up front; every start beyond the warp bin gets a
    // team or CTA hash table and one whose table fills up is re-queued
    bb.hash_max = vpp ? ~0ull : (uint64_t)hash_max_work;
    const int32_t team_req = team_max_work >= 0 ? team_max_work : (vpp ? kTeamMaxWork : kTeamFitWork);
    bb.team_max = std::max<uint64_t>((uint64_t)team_req, bb.warp_max);
    if (!vpp) bb.team_max = std::min<uint64_t>(bb.team_max, bb.hash_max);
    if (vpp && hash_max_work == 0) bb.team_max = bb.warp_max;   // all of them to the dense pass
    // without a core the bounds lie past every id
    bb.l = g->l;
    bb.core_lo_u = g->core_u > 0 ? g->core_lo_u : g->n;
    bb.core_lo_l = g->core_l > 0 ? g->core_lo_l : g->n;
    bb.cut = vpp ? nullptr : g->cut;
    return bb;
}

// Starts the binning of all starts on s: counts[0..5] (zeroed here) = dense,
// hash, team, warp, the first three together, tiny; g->warp_items is filled.
// With `stats` (zeroed by the caller, counts at stats + 3) the graph's statistics too.
static int bin_starts(Graph *g, cudaStream_t s, const BinBounds &bb, unsigned long long *counts, int32_t *heavy,
                      unsigned long long *stats, const int *guard) {
    if (!stats) BFC_CUDA(cudaMemsetAsync(counts, 0, 6 * sizeof(unsigned long long), s));
    if (g->n == 0) return BFC_OK;
    k_bin_starts<<<(unsigned)std::min<int64_t>(((int64_t)g->n + kBinTile - 1) / kBinTile, 152 * 8), kT, 0, s>>>(
        g->work, g->n, bb, counts, heavy, g->warp_items, stats, (uint64_t)g->opt.hash_max_work, g->gstar,
        stats && g->num_graphs > 0 ? g->gwork : nullptr, guard); note_launch();
    BFC_CUDA(cudaGetLastError());
    return BFC_OK;
}

// Room for a schedule's lists in one allocation: CTA items, team items and one
// place per start that can be re-queued (each at most once per launch): the rest
// of the first slab where they fit (the one schedule that most graphs have), else
// an allocation of its own.  Another rebinning takes it over where it is large
// enough, else replaces it.
static int schedule_lists(Graph *g, int64_t n_items, int64_t n_team, int64_t retry_cap) {
    n_items = std::max<int64_t>(n_items, 1);
    n_team = std::max<int64_t>(n_team, 1);
    retry_cap = std::max<int64_t>(retry_cap, 1);
    const size_t need = (size_t)n_items * sizeof(int2) + (size_t)(n_team + retry_cap) * sizeof(int32_t);
    if (need > g->lists_bytes) {
        const bool first = !g->lists;
        if (g->lists_own) g->mem.drop(g->lists);
        g->lists = nullptr;
        g->lists_bytes = 0;
        g->lists_own = !(first && g->mem.carve(&g->lists, need));
        if (g->lists_own && g->mem.get_own(&g->lists, need) != cudaSuccess) {
            g->lists = nullptr;
            g->lists_own = false;
            set_last_error("device allocation failed: schedule lists");
            return BFC_ERR_OUT_OF_MEMORY;
        }
        g->lists_bytes = need;
    }
    g->cta_items = reinterpret_cast<int2 *>(g->lists);
    g->team_items = reinterpret_cast<int32_t *>(g->cta_items + n_items);
    g->retry = g->team_items + n_team;
    g->retry_cap = retry_cap;
    return BFC_OK;
}

// Step a5: order the starts by descending exact work and split them into the
// warp, CTA-hash and CTA-dense bins (dense starts into end-range chunks);
// builds the chunk-boundary table when a dense start has several chunks.
// `rows_star` (slot -> vertex of G*) may be null; it is rebuilt when needed.
// hc[0..5] and `heavy` are bin_starts' results with the bounds bb.  Only reads
// memory of the library.
static int schedule_graph(Graph *g, cudaStream_t s, int32_t warp_max_work, int32_t team_max_work,
                          int32_t hash_max_work, const int32_t *rows_star, const BinBounds &bb,
                          const unsigned long long *hc, int32_t *heavy) {
    const int32_t r = g->r, l = g->l, n = g->n;
    const int64_t m = g->m;
    const bool vpp = g->opt.orientation == 1;
    Allocs tmp;
    tmp.stream = s;
    struct TmpGuard { Allocs *a; ~TmpGuard() { a->release(); } } guard{&tmp};
#define GET(allocs, ptr, cnt)                                                         \
    do {                                                                              \
        cudaError_t e_ = (allocs).get(&(ptr), (size_t)(cnt));                         \
        if (e_ != cudaSuccess) {                                                      \
            set_last_error(std::string("device allocation failed: ") + #ptr);         \
            return BFC_ERR_OUT_OF_MEMORY;                                             \
        }                                                                             \
    } while (0)
    const uint64_t maxw = g->info.max_start_work, team_max = bb.team_max;
    int64_t n_dense = 0, n_hash = 0, n_team = 0, n_warp = 0, n_tiny = 0, n_items = 0, h_dense_items = 0;
    if (n > 0 && g->info.wedges > 0) {
        n_dense = (int64_t)hc[0]; n_hash = (int64_t)hc[1]; n_team = (int64_t)hc[2]; n_warp = (int64_t)hc[3];
        n_tiny = (int64_t)hc[5];
        const int64_t n_heavy = n_dense + n_hash + n_team;
        uint64_t *k0 = nullptr, *k1 = nullptr;
        int32_t *v1 = nullptr;
        uint32_t *hist, *hist_tmp;
        int64_t *scan64_tmp = nullptr, *nch = nullptr;
        const int32_t *order = heavy;
        if (n_heavy > 0) GET(tmp, scan64_tmp, scan_tmp_elems<int64_t>(std::max<int64_t>(n_dense, n) + 1));
        if (n_heavy > 1 && n_heavy <= kSchedSmall && maxw < 1ull << (64 - kSchedPlaceBits - 1)) {
            GET(tmp, v1, n_heavy);
            k_sched_small<<<1, 1024, 0, s>>>(g->work, heavy, (int)n_heavy, maxw, l, bb.core_lo_u,
                                                            bb.core_lo_l, v1); note_launch();
            BFC_CUDA(cudaGetLastError());
            order = v1;
        } else if (n_heavy > 1) {
            GET(tmp, k0, n_heavy + 1); GET(tmp, k1, n_heavy + 1); GET(tmp, v1, n_heavy);
            GET(tmp, hist, radix_hist_elems(n_heavy));
            GET(tmp, hist_tmp, scan_tmp_elems<uint32_t>((int64_t)radix_hist_elems(n_heavy)));
            int which = 0;
            k_sched_keys<<<blocks_for(n_heavy), kT, 0, s>>>(g->work, heavy, n_heavy, maxw, l, bb.core_lo_u,
                                                            bb.core_lo_l, k0); note_launch();
            BFC_CUDA(cudaGetLastError());
            BFC_CUDA(radix_sort_pairs(k0, heavy, k1, v1, n_heavy, 0, bits_for(maxw), hist, hist_tmp, s, &which));
            order = which ? v1 : heavy;
        }
        // a layer (a batch's graph's) this small is one chunk of any counters,
        // or of 16-bit ones where no degree can pass 65,535
        const bool one_chunk = g->max_range <= kDense32 ||
                               (!g->parallel && g->max_range <= kDense16 && g->max_range <= (int32_t)kNarrowMaxCut);
        int64_t *nch_scan = nullptr;
        h_dense_items = n_dense;
        if (n_dense > 0 && !one_chunk) {
            GET(tmp, nch, n_dense + 1);
            GET(tmp, nch_scan, n_dense + 1);
            k_chunk_counts<<<blocks_for(n_dense), kT, 0, s>>>(order, n_dense, l, g->bcut, g->boff, g->vbase, nch); note_launch();
            BFC_CUDA(cudaGetLastError());
            BFC_CUDA(scan_exclusive<int64_t>(nch, nch_scan, n_dense, scan64_tmp, s));
            BFC_CUDA(cudaMemcpyAsync(&h_dense_items, nch_scan + n_dense, sizeof(int64_t),
                                     cudaMemcpyDeviceToHost, s));
            BFC_CUDA(cudaStreamSynchronize(s));
        }
        n_items = h_dense_items + n_hash;
        if (int rc = schedule_lists(g, n_items, n_team, n_hash + n_team)) return rc;
        if (n_heavy > 0) {
            k_emit_items<<<grid_stride_blocks(n_heavy), kT, 0, s>>>(
                order, n_dense, n_hash, n_team, nch_scan, l, g->bcut, g->boff, g->vbase, vpp ? 1 : 0, g->cta_items,
                g->team_items); note_launch();
            BFC_CUDA(cudaGetLastError());
        }
        // chunk boundaries of every list, so dense items read them instead of searching
        const int32_t u1 = (int32_t)((r + kChunkUnit - 1) / kChunkUnit) + 1;
        const int32_t l1 = (int32_t)((l + kChunkUnit - 1) / kChunkUnit) + 1;
        const int64_t entries = (int64_t)l * u1 + (int64_t)r * l1;
        if (!g->coff && g->num_graphs > 0 && h_dense_items > n_dense) {
            // a batch: entries only for the middles of starts with several
            // chunks, as many as the chunks of their graph's neighbour layer
            // (+1), found through a per-vertex start array
            int32_t *mark;
            int64_t *ecnt, *cstart;   // cstart: first entry of each vertex
            GET(tmp, mark, n);
            GET(tmp, ecnt, (int64_t)n + 1);
            GET(tmp, cstart, (int64_t)n + 1);
            BFC_CUDA(cudaMemsetAsync(mark, 0, sizeof(int32_t) * (size_t)n, s));
            k_coff_mark<<<grid_stride_blocks(n_dense * 32), kT, 0, s>>>(order, n_dense, nch, g->off, g->adj,
                                                                         g->cut, mark); note_launch();
            k_coff_sizes<<<grid_stride_blocks(n), kT, 0, s>>>(mark, g->off, g->adj, g->vbase, g->vend, n, ecnt); note_launch();
            BFC_CUDA(cudaGetLastError());
            BFC_CUDA(scan_exclusive<int64_t>(ecnt, cstart, n, scan64_tmp, s));
            int64_t ventries = 0;
            BFC_CUDA(cudaMemcpyAsync(&ventries, cstart + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
            BFC_CUDA(cudaStreamSynchronize(s));
            if (ventries <= kChunkTableMaxEntries) {   // else searches
                if (!rows_star) {
                    int32_t *rs;
                    GET(tmp, rs, 2 * m);
                    k_rows_from_off<<<grid_stride_blocks((int64_t)n * 32), kT, 0, s>>>(g->off, n, rs); note_launch();
                    BFC_CUDA(cudaGetLastError());
                    rows_star = rs;
                }
                // each middle slot of those starts holds its middle's first
                // entry (-1 elsewhere), read with the slot's other arrays
                int32_t *coff, *ctb;
                GET(g->mem, coff, std::max<int64_t>(ventries, 1));
                GET(g->mem, ctb, 2 * m);
                k_coff_fill_var<<<grid_stride_blocks(n), kT, 0, s>>>(g->off, cstart, n, coff); note_launch();
                BFC_CUDA(cudaGetLastError());
                k_coff_slots_var<<<grid_stride_blocks(2 * m), kT, 0, s>>>(g->off, g->adj, rows_star, 2 * m,
                                                                          g->vbase, cstart, coff); note_launch();
                BFC_CUDA(cudaGetLastError());
                BFC_CUDA(cudaMemsetAsync(ctb, 0xff, sizeof(int32_t) * (size_t)(2 * m), s));
                k_coff_slot_bases<<<grid_stride_blocks(n_dense * 32), kT, 0, s>>>(order, n_dense, nch, g->off, g->adj,
                                                                                   g->cut, cstart, ctb); note_launch();
                BFC_CUDA(cudaGetLastError());
                g->coff = coff;   // the two only together
                g->ctb = ctb;
            }
        }
        if (!g->coff && g->num_graphs == 0 && h_dense_items > n_dense && entries <= kChunkTableMaxEntries) {
            if (!rows_star) {
                int32_t *rs;
                GET(tmp, rs, 2 * m);
                k_rows_from_off<<<grid_stride_blocks((int64_t)n * 32), kT, 0, s>>>(g->off, n, rs); note_launch();
                BFC_CUDA(cudaGetLastError());
                rows_star = rs;
            }
            GET(g->mem, g->coff, entries);
            g->coff_u1 = u1;
            g->coff_l1 = l1;
            k_coff_fill<<<grid_stride_blocks(entries), kT, 0, s>>>(g->off, l, u1, l1, entries, g->coff); note_launch();
            BFC_CUDA(cudaGetLastError());
            k_coff_slots<<<grid_stride_blocks(2 * m), kT, 0, s>>>(g->off, g->adj, rows_star, 2 * m, l, u1, l1,
                                                                  g->coff); note_launch();
            BFC_CUDA(cudaGetLastError());
        }
    } else if (int rc = schedule_lists(g, 0, 0, 0)) {
        return rc;
    }
    g->n_cta_items = n_items;
    g->n_team_items = n_team;
    g->n_warp_items = n_warp;
    g->n_tiny_items = n_tiny;
    g->team_max = (int32_t)std::min<uint64_t>(team_max, (uint64_t)kTeamMaxWork);
    g->retry_static = 0;
    if (vpp && hash_max_work == 0 && n_hash > 0) {
        // every start beyond the warp bin goes to the dense pass directly
        k_items_to_dense_retries<<<blocks_for(n_hash), kT, 0, s>>>(g->cta_items, n_hash, g->retry); note_launch();
        BFC_CUDA(cudaGetLastError());
        g->retry_static = n_hash;
        g->n_cta_items = 0;
    }
    // Algorithm 2's tables always fit when a team start has at most 3,072
    // wedges (4,096 slots) and a CTA start at most 24,576 (32,768 slots)
    g->may_retry = vpp ? (n_hash + n_team > 0) : (n_team > 0 && team_max > (uint64_t)kTeamFitWork);
    g->info.dense_items = h_dense_items;
    g->info.starts_with_work = n_dense + n_hash + n_team + n_warp + n_tiny;
    g->info.dense_starts = n_dense;
    g->info.hash_starts = n_hash;
    g->info.team_starts = n_team;
    g->info.warp_starts = n_warp + n_tiny;
    g->opt.warp_max_work = warp_max_work;
    g->opt.team_max_work = team_max_work;
    g->opt.hash_max_work = hash_max_work;
#undef GET
    g->schedule_rc = BFC_OK;
    return BFC_OK;
}

int rebin_graph(Graph *g, cudaStream_t s, int32_t warp_max_work, int32_t team_max_work,
                int32_t hash_max_work) {
    // no schedule until the new one is whole: a count after a failure reports it
    // and launches nothing
    g->schedule_rc = BFC_ERR_OUT_OF_MEMORY;
    g->mem.stream = s;
    Allocs tmp;
    tmp.stream = s;
    struct TmpGuard { Allocs *a; ~TmpGuard() { a->release(); } } guard{&tmp};
    int32_t *heavy;
    unsigned long long *counts, hc[6] = {0, 0, 0, 0, 0, 0};
    if (tmp.get(&heavy, (size_t)std::max(g->n, 1)) || tmp.get(&counts, 6)) {
        set_last_error("device allocation failed: bins");
        return BFC_ERR_OUT_OF_MEMORY;
    }
    const BinBounds bb = bin_bounds(g, warp_max_work, team_max_work, hash_max_work);
    int rc = bin_starts(g, s, bb, counts, heavy, nullptr, nullptr);
    if (rc) return rc;
    BFC_CUDA(cudaMemcpyAsync(hc, counts, sizeof(hc), cudaMemcpyDeviceToHost, s));
    BFC_CUDA(cudaStreamSynchronize(s));
    rc = schedule_graph(g, s, warp_max_work, team_max_work, hash_max_work, nullptr, bb, hc, heavy);
    if (rc != BFC_OK) g->schedule_rc = rc;
    g->info.device_bytes = (int64_t)g->mem.total;
    if (rc == BFC_OK) BFC_CUDA(cudaStreamSynchronize(s));
    return rc;
}

// what an error word says about the caller's arrays (BFC_OK: nothing)
static int input_error(int err, int32_t num_graphs) {
    if (err & kErrBadOffsets) { set_last_error("off_u is not a CSR offset array of num_edges entries"); return BFC_ERR_INVALID_GRAPH; }
    if (err & kErrBadId) {
        set_last_error(num_graphs > 0 ? "an L id lies outside [0, num_l), or an edge joins vertices of two different "
                                        "graphs of the batch"
                                      : "adj_u holds an id outside [0, num_l)");
        return BFC_ERR_INVALID_GRAPH;
    }
    if (err & kErrDuplicate) { set_last_error("duplicate edge"); return BFC_ERR_INVALID_GRAPH; }
    return BFC_OK;
}

// The largest degree that the rank keys have to tell apart: no larger than the
// largest layer (of one graph) where duplicate edges are rejected; otherwise
// every edge can be the same one.
static int64_t degree_bound(const bfc_options *opt, int32_t max_range, int64_t m) {
    return opt->validate ? max_range : std::max<int64_t>(max_range, m);
}

// Step a2: one sort of both layers' vertices.
static int launch_ranks(Graph *g, const int32_t *deg_l, const int32_t *deg_u, const int32_t *gl, const int32_t *gu,
                        int64_t max_degree, uint64_t *k0, int32_t *v0, uint64_t *k1, int32_t *v1, uint32_t *hist,
                        uint32_t *hist_tmp, int32_t *deg_star, int64_t *deg64, unsigned long long *top,
                        cudaStream_t s, const int *guard) {
    const int32_t n = g->n;
    if (n == 0) return BFC_OK;
    const int bdeg = bits_for((uint64_t)max_degree);
    const int blayer = bdeg + (g->num_graphs > 0 ? bits_for((uint64_t)(g->num_graphs - 1)) : 0);
    k_rank_keys<<<blocks_for(n), kT, 0, s>>>(deg_l, deg_u, g->l, n, gl, gu, g->num_graphs, bdeg, blayer, k0, guard); note_launch();
    BFC_CUDA(cudaGetLastError());
    int which = 0;
    BFC_CUDA(radix_sort_pairs(k0, v0, k1, v1, n, 0, blayer + (g->r > 0 && g->l > 0 ? 1 : 0), hist, hist_tmp, s, &which,
                              true));
    k_ranks<<<blocks_for(n), kT, 0, s>>>(which ? v1 : v0, deg_l, deg_u, g->l, n, g->rank_l, g->rank_u, deg_star, deg64,
                                         top, guard); note_launch();
    BFC_CUDA(cudaGetLastError());
    return BFC_OK;
}

// shared memory of a bitmap over `range` L ranks
static int bitmap_bytes(int32_t range) { return (std::min(range, kRowBitmapMax) + 127) / 128 * 20; }

static int rows_smem_setup(int device) {
    static bool done[64] = {false};
    if (device < 0 || device >= 64) return BFC_ERR_INVALID_ARGUMENT;
    if (done[device]) return BFC_OK;
    BFC_CUDA(cudaFuncSetAttribute(k_u_rows_bitmap<kRowCtaThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  bitmap_bytes(kRowBitmapMax)));
    BFC_CUDA(cudaFuncSetAttribute(k_u_rows_bitmap<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  bitmap_bytes(kRowBitmapMax)));
    done[device] = true;
    return BFC_OK;
}

// The U side of G*: every tier that needs no size on the host (tier_n is zero).  `range`: the L
// ranks of a single graph, or of a batch's largest graph.
static int launch_u_rows(const int32_t *off_u, const int32_t *adj_u, Graph *g, int32_t range, const int32_t *gu,
                         const int32_t *gl, int32_t num_graphs, int bitmaps, const URowOut &uo,
                         int32_t *tier_rows, int32_t *tier_n, cudaStream_t s, const int *guard) {
    const int32_t r = g->r;
    const int64_t m = g->m;
    int rc = rows_smem_setup(g->device);
    if (rc) return rc;
    const int span = (int)std::min<int64_t>(std::max<int64_t>(r / (152 * 64), 4), 32);
    k_u_rows_warp<<<grid_stride_blocks((int64_t)(r + span - 1) / span * 32), kT, 0, s>>>(
        off_u, adj_u, g->rank_u, g->rank_l, r, span, gl, gu, num_graphs, uo, guard); note_launch();
    BFC_CUDA(cudaGetLastError());
    if (m <= kRowWarpMax) return BFC_OK;
    const int wide_tier = range > kRowCtaMax ? 1 : 0;   // a valid row is no longer than the range
    k_row_tiers<<<grid_stride_blocks(r), kT, 0, s>>>(off_u, r, range, gu, gl, num_graphs, bitmaps, wide_tier, tier_rows,
                                                     tier_n,
                                                     guard); note_launch();
    const unsigned wg = (unsigned)std::min<int64_t>(m / (kRowWarpMax + 1) * 32 / kRowCtaThreads + 1, 152 * 8);
    if (range <= 1 << 24) {
        k_u_rows_warp_reg<<<wg, kRowCtaThreads, 0, s>>>(off_u, adj_u, g->rank_u, g->rank_l, tier_rows, tier_n, gl, gu,
                                                        num_graphs, uo, guard); note_launch();
    } else {
        k_u_rows_warp_sort<<<wg, kRowCtaThreads, 0, s>>>(off_u, adj_u, g->rank_u, g->rank_l, tier_rows, tier_n, uo,
                                                         guard); note_launch();
    }
    if (bitmaps && m > kRowWarpSortMax) {
        k_u_rows_bitmap<kRowCtaThreads>
            <<<(unsigned)std::min<int64_t>(m / kRowWarpSortMax, 152 * 8), kRowCtaThreads, bitmap_bytes(range), s>>>(
                off_u, adj_u, g->rank_u, g->rank_l, tier_rows + r, tier_n + 1, range, gl, gu, num_graphs, uo, guard);
        note_launch();
    }
    if (bitmaps == 2 && m > kRowWarpSortMax) {
        k_u_rows_cta<<<(unsigned)std::min<int64_t>(m / kRowWarpSortMax, 152 * 16), kRowCtaThreads, 0, s>>>(
            off_u, adj_u, g->rank_u, g->rank_l, tier_rows + 3 * (int64_t)r, tier_n + 3, uo, guard); note_launch();
    }
    if (bitmaps && wide_tier && m > kRowCtaMax) {
        k_u_rows_bitmap<1024>
            <<<(unsigned)std::min<int64_t>(m / kRowCtaMax, 152 * 2), 1024, bitmap_bytes(range), s>>>(
                off_u, adj_u, g->rank_u, g->rank_l, tier_rows + 2 * (int64_t)r, tier_n + 2, range, gl, gu, num_graphs, uo,
                guard);
        note_launch();
    }
    BFC_CUDA(cudaGetLastError());
    return BFC_OK;
}

// cut (Algorithm 2) and work per start, and the runs of the U-side middle slots
// (`queued` is zero)
static void launch_work(Graph *g, const int32_t *deg_star, int32_t *queue, int32_t *queued, cudaStream_t s,
                        const int *guard) {
    const int vpp = g->opt.orientation;
    const int64_t fill_from = vpp ? 2 * g->m + 1 : g->m;
    k_work<<<grid_stride_blocks(g->n), kT, 0, s>>>(g->off, g->adj, deg_star, g->l, g->cut, g->plen, g->n, vpp,
                                                   fill_from, g->sbeg, g->work, queue, queued, guard); note_launch();
    if (2 * g->m > kWorkLane) {
        k_work_long<<<(unsigned)std::min<int64_t>(2 * g->m / kWorkLane / (kWorkThreads / 32) + 1, 152 * 4), kWorkThreads, 0, s>>>(
            g->off, g->adj, g->cut, g->plen, g->n, vpp, fill_from, g->sbeg, g->work, queue, queued, guard); note_launch();
    }
}

int prepare_graph(const bfc_csr *csr, const bfc_options *opt, cudaStream_t s, Graph *g,
                  int32_t num_graphs, const int32_t *graph_u_start, const int32_t *graph_l_start) {
    const int32_t r = csr->num_u, l = csr->num_l;
    const int64_t m = csr->num_edges;
    const int32_t n = r + l;
    g->r = r; g->l = l; g->n = n; g->m = m;
    g->opt = *opt;
    g->stream = s;
    g->mem.stream = s;
    {
        // many small graphs may be kept: one slab that just holds a small graph's arrays
        auto small = [](size_t bytes) { return bytes <= Allocs::kCarve ? Allocs::rounded(bytes) : 0; };
        const size_t nn = (size_t)n, mm = (size_t)m, per_n = num_graphs > 0 ? 6 : 3;
        const size_t sum = small(4 * (size_t)r) + small(4 * (size_t)l) + 2 * small(8 * nn) + small(8 * (nn + 1)) +
                           per_n * small(4 * nn) + 3 * small(8 * mm) + small(16 * mm) +
                           (num_graphs > 0 ? small(8 * (size_t)num_graphs) : 0) + 2 * 256 +
                           small(4 * nn);   // the schedule's lists, where few starts are heavy
        g->mem.slab_next = std::min(sum, Allocs::kSlab);
    }

    Allocs tmp;
    tmp.stream = s;
    struct TmpGuard { Allocs *a; ~TmpGuard() { a->release(); } } guard{&tmp};

#define GET(allocs, ptr, cnt)                                                         \
    do {                                                                              \
        cudaError_t e_ = (allocs).get(&(ptr), (size_t)(cnt));                         \
        if (e_ != cudaSuccess) {                                                      \
            set_last_error(std::string("device allocation failed: ") + #ptr);         \
            return BFC_ERR_OUT_OF_MEMORY;                                             \
        }                                                                             \
    } while (0)

    // ---- kept arrays
    GET(g->mem, g->err, 4);
    GET(g->mem, g->rank_u, r);
    GET(g->mem, g->rank_l, l);
    GET(g->mem, g->off, (int64_t)n + 1);
    GET(g->mem, g->adj, 2 * m);
    GET(g->mem, g->eid, 2 * m);
    GET(g->mem, g->plen, 2 * m);
    GET(g->mem, g->sbeg, std::max<int64_t>(2 * m, 1));
    GET(g->mem, g->cut, n);
    GET(g->mem, g->work, n);
    GET(g->mem, g->cursors, 8 + 4);
    g->acc = reinterpret_cast<unsigned long long *>(g->cursors + 8);   // cleared together
    GET(g->mem, g->pv, n);
    GET(g->mem, g->warp_items, std::max(n, 1));
    g->bcut = g->cut;
    g->boff = g->off;
    BFC_CUDA(cudaMemsetAsync(g->err, 0, 4 * sizeof(int), s));

    // A batch's start arrays are checked first: its largest layers size what
    // follows.  Everything else about the caller's arrays is checked by kernels
    // whose error word stops every later kernel that would index with them, and
    // reported at the one round trip after the work is known.
    int herr = 0;
    int32_t l_range = l;
    g->max_range = std::max(r, l);
    if (num_graphs > 0) {
        k_check_starts<<<blocks_for((int64_t)num_graphs + 1), kT, 0, s>>>(graph_u_start, num_graphs, r, g->err, 0x7fffffff, g->err + 2); note_launch();
        k_check_starts<<<blocks_for((int64_t)num_graphs + 1), kT, 0, s>>>(graph_l_start, num_graphs, l, g->err, 0x7fffffff, g->err + 1); note_launch();
        BFC_CUDA(cudaGetLastError());
        int hstart[3] = {0, 0, 0};
        BFC_CUDA(cudaMemcpyAsync(hstart, g->err, 3 * sizeof(int), cudaMemcpyDeviceToHost, s));
        BFC_CUDA(cudaStreamSynchronize(s));
        if (hstart[0]) { set_last_error("graph start arrays are not prefix sums of the layer sizes"); return BFC_ERR_INVALID_GRAPH; }
        l_range = hstart[1];   // the largest L layer of one graph
        g->max_range = std::max(hstart[1], hstart[2]);
        g->num_graphs = num_graphs;
        GET(g->mem, g->gstar, std::max<int64_t>(n, 1));
        GET(g->mem, g->vbase, std::max<int64_t>(n, 1));
        GET(g->mem, g->vend, std::max<int64_t>(n, 1));
        GET(g->mem, g->gwork, num_graphs);
        BFC_CUDA(cudaMemsetAsync(g->gwork, 0, sizeof(unsigned long long) * num_graphs, s));
    }
    const int *guard_err = g->err;

    // ---- temporaries
    const int64_t nsort = std::max<int64_t>({(int64_t)r, (int64_t)l, m, (int64_t)n, 1});
    uint64_t *k0, *k1;
    int32_t *v0, *v1, *deg_u, *deg_l, *deg_star, *rows_star, *heads, *big, *n_big, *heavy;
    uint32_t *hist, *hist_tmp;
    int64_t *scan64_tmp, *deg64;
    // [0] W, [1] heaviest start, [2] starts beyond the CTA-hash bin, [3..9) bin
    // counts, [9] / [10] largest L / U degree, [11] the error word, then the work
    // queues' and the row tiers' counters: cleared together
    unsigned long long *red;
    GET(tmp, k0, nsort + 1); GET(tmp, k1, nsort + 1);
    GET(tmp, v0, nsort); GET(tmp, v1, nsort);
    GET(tmp, deg_u, r); GET(tmp, deg_l, l); GET(tmp, deg_star, n);
    GET(tmp, rows_star, 2 * m);
    GET(tmp, big, n);
    GET(tmp, hist, radix_hist_elems(nsort));
    GET(tmp, hist_tmp, scan_tmp_elems<uint32_t>((int64_t)radix_hist_elems(nsort)));
    GET(tmp, scan64_tmp, std::max(scan_tmp_elems<int64_t>((int64_t)n + 1),
                                  max_scan_tmp_elems(m)));
    GET(tmp, deg64, (int64_t)n + 1);
    GET(tmp, red, kRedWords);
    n_big = reinterpret_cast<int32_t *>(red + 12);
    GET(tmp, heavy, std::max(n, 1));
    BFC_CUDA(cudaMemsetAsync(red, 0, kRedWords * sizeof(unsigned long long), s));

    // ---- a1: degrees, and the check of the caller's offsets and L ids
    BFC_CUDA(cudaMemsetAsync(deg_l, 0, sizeof(int32_t) * std::max<int64_t>(l, 1), s));
    k_check_input<<<grid_stride_blocks(std::max<int64_t>(m, (int64_t)r + 1)), kT, 0, s>>>(
        csr->off_u, csr->adj_u, r, l, m, deg_u, deg_l, g->err); note_launch();
    BFC_CUDA(cudaGetLastError());

    // ---- a2: per-layer priority ranks by a stable sort on (layer, graph, degree)
    {
        int rc = launch_ranks(g, deg_l, deg_u, graph_l_start, graph_u_start, degree_bound(opt, g->max_range, m), k0, v0, k1, v1, hist,
                              hist_tmp, deg_star, deg64, red + 9, s, guard_err);
        if (rc) return rc;
    }

    if (num_graphs > 0 && n > 0) {
        k_graph_star<<<grid_stride_blocks(n), kT, 0, s>>>(r, l, graph_u_start, graph_l_start,
                                                         num_graphs, g->gstar, g->vbase, g->vend, guard_err); note_launch();
        BFC_CUDA(cudaGetLastError());
    }

    // ---- a3: G* offsets and priority-sorted lists
    BFC_CUDA(scan_exclusive<int64_t>(deg64, g->off, n, scan64_tmp, s));
    const int bu = bits_for(r > 0 ? (uint64_t)(r - 1) : 0);
    const int bl = bits_for(l > 0 ? (uint64_t)(l - 1) : 0);
    if (m > 0) {
        if (num_graphs > 0 && (!opt->validate || l_range > kRowBitmapMax)) {
            k_check_batch_rows<<<grid_stride_blocks(r), kT, 0, s>>>(csr->off_u, csr->adj_u, r, graph_u_start,
                                                                    graph_l_start, num_graphs, g->err, guard_err); note_launch();
            BFC_CUDA(cudaGetLastError());
        }
        // U side row by row (warp / CTA tiers, radix sort for the largest rows);
        // the swapped keys for the L side land in k1
        const URowOut uo{m, l, bu, g->off, g->adj, g->eid, rows_star, k1, g->err, opt->validate ? kErrDuplicate : kErrParallel};
        int32_t *tier_rows = nullptr, *const tier_n = n_big + 2;
        GET(tmp, tier_rows, kRowTiers * std::max<int64_t>(r, 1));
        {
            int rc = launch_u_rows(csr->off_u, csr->adj_u, g, l_range, graph_u_start, graph_l_start, num_graphs,
                                   opt->validate, uo, tier_rows, tier_n, s, guard_err);
            if (rc) return rc;
        }
        // rows that no bitmap takes (see the tiers): CTA sorts, and a radix sort
        // of the largest rows' edges
        if (m > kRowWarpSortMax && (!opt->validate || l_range > kRowBitmapMax)) {
            int32_t hn[2] = {0, 0};
            BFC_CUDA(cudaMemcpyAsync(hn, tier_n + 3, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
            BFC_CUDA(cudaMemcpyAsync(&herr, g->err, sizeof(int), cudaMemcpyDeviceToHost, s));
            BFC_CUDA(cudaStreamSynchronize(s));
            if (int rc = input_error(herr, num_graphs)) return rc;
            if (hn[0] > 0) {
                k_u_rows_cta<<<(unsigned)std::min<int32_t>(hn[0], 152 * 16), kRowCtaThreads, 0, s>>>(
                    csr->off_u, csr->adj_u, g->rank_u, g->rank_l, tier_rows + 3 * (int64_t)r, tier_n + 3,
                    uo, guard_err); note_launch();
                BFC_CUDA(cudaGetLastError());
            }
            const int32_t *large_rows = tier_rows + 4 * (int64_t)r;
            const int32_t nl = hn[1];
            int64_t *ldeg, *loff;
            GET(tmp, ldeg, (int64_t)nl + 1);
            GET(tmp, loff, (int64_t)nl + 1);
            int64_t nlarge = 0;
            if (nl > 0) {
                k_large_deg<<<blocks_for(nl), kT, 0, s>>>(csr->off_u, large_rows, nl, ldeg); note_launch();
                BFC_CUDA(cudaGetLastError());
                BFC_CUDA(scan_exclusive<int64_t>(ldeg, loff, nl, scan64_tmp, s));
                BFC_CUDA(cudaMemcpyAsync(&nlarge, loff + nl, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
                BFC_CUDA(cudaStreamSynchronize(s));
            }
            if (nlarge > 0) {
                uint64_t *ka;
                int32_t *va, *rowf;
                GET(tmp, ka, nlarge); GET(tmp, va, nlarge); GET(tmp, rowf, nlarge); GET(tmp, heads, nlarge);
                k_large_keys<<<(unsigned)std::min<int32_t>(nl, 1024), kT, 0, s>>>(csr->off_u, csr->adj_u, g->rank_u,
                                                                                   g->rank_l, large_rows, loff, nl, bl,
                                                                                   k0, v0); note_launch();
                BFC_CUDA(cudaGetLastError());
                int wl = 0;
                BFC_CUDA(radix_sort_pairs(k0, v0, ka, va, nlarge, 0, bu + bl, hist, hist_tmp, s, &wl));
                const uint64_t *kl = wl ? ka : k0;
                const int32_t *vl = wl ? va : v0;
                k_large_heads<<<grid_stride_blocks(nlarge), kT, 0, s>>>(kl, nlarge, bl, heads); note_launch();
                BFC_CUDA(cudaGetLastError());
                BFC_CUDA(max_scan_inclusive(heads, rowf, nlarge, (int32_t *)scan64_tmp, s));
                k_large_emit<<<grid_stride_blocks(nlarge), kT, 0, s>>>(kl, vl, rowf, nlarge, bl, uo); note_launch();
                BFC_CUDA(cudaGetLastError());
            }
        }
        uint64_t *ks = k0;
        int32_t *vs = v0;
        uint64_t *ko = k1;
        int32_t *vo = v1;
        // stable sort of the (rank_l, rank_u) keys on the rank_l bits only:
        // the input is already ascending in rank_u within each rank_l
        int which2 = 0;
        BFC_CUDA(radix_sort_pairs(ko, vo, ks, vs, m, bu, bu + bl, hist, hist_tmp, s, &which2, true));
        const uint64_t *k2 = which2 ? ks : ko;
        const int32_t *v2 = which2 ? vs : vo;
        if (opt->orientation == 0) {
            BFC_CUDA(cudaMemsetAsync(g->plen + m, 0, sizeof(int32_t) * (size_t)m, s));
            k_emit_l_side<true><<<grid_stride_blocks(m), kT, 0, s>>>(k2, v2, m, bu, l, g->off, g->adj, g->eid,
                                                                      rows_star, g->plen, g->sbeg, !opt->validate,
                                                                      guard_err); note_launch();
        } else {
            k_emit_l_side<false><<<grid_stride_blocks(m), kT, 0, s>>>(k2, v2, m, bu, l, g->off, g->adj, g->eid,
                                                                       rows_star, nullptr, nullptr, 0, guard_err); note_launch();
        }
        BFC_CUDA(cudaGetLastError());
    }

    // ---- a4: cut, per-middle prefix lengths, per-start work, W
    if (n > 0 && opt->orientation == 1) {
        k_cut<<<blocks_for(n), kT, 0, s>>>(g->off, g->adj, deg_star, n, l, g->cut, guard_err); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    if (m > 0 && opt->orientation == 1) {
        k_slen<<<grid_stride_blocks(2 * m), kT, 0, s>>>(g->off, g->adj, rows_star, g->cut, 2 * m,
                                                         g->plen, g->sbeg, guard_err); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    const bool core_auto = opt->core_vertices < 0 && opt->orientation == 0 && num_graphs == 0;
    if (n > 0) {
        launch_work(g, deg_star, big, n_big, s, guard_err);
        BFC_CUDA(cudaGetLastError());
    }
    // the bins without a core, before the round trip (a core, which only large
    // graphs get, moves its starts to the dense bin: those are binned again)
    BinBounds bb = bin_bounds(g, opt->warp_max_work, opt->team_max_work, opt->hash_max_work);
    {
        int rc = bin_starts(g, s, bb, red + 3, heavy, red, guard_err);
        if (rc) return rc;
    }
    unsigned long long hred[12] = {0};
    // without a vertex no kernel has copied the error word
    BFC_CUDA(n > 0 ? cudaMemcpyAsync(hred, red, sizeof(hred), cudaMemcpyDeviceToHost, s)
                   : cudaMemcpyAsync(&herr, g->err, sizeof(int), cudaMemcpyDeviceToHost, s));
    BFC_CUDA(cudaStreamSynchronize(s));
    if (int rc = input_error(n > 0 ? (int)hred[11] : herr, num_graphs)) return rc;
    g->info.wedges = hred[0];
    g->info.max_start_work = hred[1];
    g->info.max_deg_l = (int32_t)hred[9];
    g->info.max_deg_u = (int32_t)hred[10];
    if (n > 0 && ((int)hred[11] & kErrParallel)) {   // known from here on: no error of a later count
        g->parallel = true;
        BFC_CUDA(cudaMemsetAsync(g->err, 0, sizeof(int), s));
        int32_t *bcut;
        int64_t *boff;
        GET(g->mem, bcut, n);
        GET(g->mem, boff, (int64_t)n + 1);
        k_count_bounds<<<grid_stride_blocks((int64_t)n + 1), kT, 0, s>>>(g->work, g->cut, g->off, n, 0x7fffffff,
                                                                         nullptr, bcut, boff); note_launch();
        BFC_CUDA(cudaGetLastError());
        g->bcut = bcut;
        g->boff = boff;
    }

    // ---- dense-core hybrid (Algorithm 2 single graphs): the requested core
    // size, or (core_vertices = -1) as many vertices as starts heavier than
    // the CTA-hash bin, at most kCoreAutoMax
    // (an automatic core below 2 x kCoreAutoMinLayer vertices cannot hold
    // both layers: nothing is launched for it)
    // (the product of 0/1 matrices knows no parallel edges)
    if (opt->core_vertices != 0 && opt->orientation == 0 && num_graphs == 0 && !g->parallel &&
        !(core_auto && hred[2] < 2ull * kCoreAutoMinLayer)) {
        const int32_t k = core_auto ? (int32_t)std::min<unsigned long long>(hred[2], (unsigned long long)kCoreAutoMax)
                                    : opt->core_vertices;
        int rc = core_prepare(g, s, deg_star, k, core_auto);
        if (rc) return rc;
    }
    g->info.core_u = g->core_u;
    g->info.core_l = g->core_l;

    // ---- a5: heaviest-first order and bins
    if (g->core_u + g->core_l > 0) {
        bb = bin_bounds(g, opt->warp_max_work, opt->team_max_work, opt->hash_max_work);
        int rc = bin_starts(g, s, bb, red + 3, heavy, nullptr, nullptr);
        if (rc) return rc;
        BFC_CUDA(cudaMemcpyAsync(hred + 3, red + 3, 6 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
        BFC_CUDA(cudaStreamSynchronize(s));
    }
    {
        int rc = schedule_graph(g, s, opt->warp_max_work, opt->team_max_work, opt->hash_max_work, rows_star, bb,
                                hred + 3, heavy);
        if (rc) return rc;
    }
    g->info.num_u = r; g->info.num_l = l; g->info.num_edges = m;
    g->info.device_bytes = (int64_t)g->mem.total;
    BFC_CUDA(cudaStreamSynchronize(s));
#undef GET
    return BFC_OK;
}

// ----------------------------------------------------------------------------
// Batch plan: a batch of a fixed shape prepared and counted with no host
// synchronisation and no allocation, so the whole step can be captured in a
// CUDA graph and replayed on new contents.  Sizes that prepare_graph reads
// back to the host come from the shape instead: the degree bits of the rank
// keys from the largest layer of one graph, the row tiers and the bin sizes
// from counts in device memory that the kernels read themselves, and every
// dense start is one end-range chunk (a graph's layer holds at most 65,535
// vertices, so counts fit 16 bits and the end range one chunk).
// ----------------------------------------------------------------------------
namespace {

// One byte per heavy start, heaviest first inside its bin: the three bins take
// codes 0..., by quarter octaves of the work (dense starts) or octaves.  Places
// past the heavy ones get 255.
__global__ void k_sched_keys_plan(const uint64_t *__restrict__ work, const int32_t *__restrict__ heavy, int32_t n,
                                  BinBounds bb, const unsigned long long *__restrict__ counts, uint64_t *keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t key = 255;
    if (i < (int64_t)counts[4]) {
        const uint64_t w = work[heavy[i]];
        const int oct = 63 - __clzll((long long)w);
        const int bin = bb.of(heavy[i], w);
        if (bin == 0) {
            const int q = oct >= 2 ? 4 * oct + (int)((w >> (oct - 2)) & 3) : 4 * oct;
            key = q < 160 ? 160 - q : 0;          // 1..160; from 2^40 wedges up 0
        } else {
            key = (bin == 1 ? 161 : 193) + (31 - min(oct, 31));
        }
    }
    keys[i] = key;
}

// the item lists from the sorted order and the bin sizes on the device: a
// dense start is one chunk (and so is one of the CTA-hash bin, which gets dense
// counters too), so the lists follow the order directly
__global__ void k_emit_items_plan(const int32_t *__restrict__ order,
                                  const unsigned long long *__restrict__ counts, const int32_t *__restrict__ cut,
                                  const int64_t *__restrict__ off, const int32_t *__restrict__ vbase, int2 *cta_items,
                                  int32_t *team_items, const int *guard) {
    if (aborted(guard)) return;
    const int64_t nd = (int64_t)counts[0], nh = (int64_t)counts[1], nt = (int64_t)counts[2];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nd + nh + nt;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = order[i];
        if (i < nd + nh) cta_items[i] = one_dense_item(x, 0, cut[x], off, vbase);
        else team_items[i - nd - nh] = x;
    }
}

__global__ void k_plan_status(const int *__restrict__ err, int check_dup, int32_t *status) {
    const int e = *err;
    int32_t st = BFC_OK;
    if (e & (kErrBadOffsets | kErrBadId)) st = BFC_ERR_INVALID_GRAPH;
    else if ((e & kErrDuplicate) && check_dup) st = BFC_ERR_INVALID_GRAPH;
    else if (e & kErrTimeout) st = BFC_ERR_TIMEOUT;
    else if (e & (kErrHashFull | kErrBounds)) st = BFC_ERR_INTERNAL;
    *status = st;
}

}  // namespace

int batch_plan_create(BatchPlan *pl, cudaStream_t s) {
    Graph *g = &pl->g;
    const int32_t r = pl->r, l = pl->l, n = r + l, G = pl->num_graphs;
    const int64_t m = pl->m;
    g->r = r; g->l = l; g->n = n; g->m = m;
    g->num_graphs = G;
    g->stream = s;
    g->mem.stream = s;
#define GET(ptr, cnt)                                                                 \
    do {                                                                              \
        cudaError_t e_ = g->mem.get(&(ptr), (size_t)std::max<int64_t>((int64_t)(cnt), 1)); \
        if (e_ != cudaSuccess) {                                                      \
            set_last_error(std::string("device allocation failed: ") + #ptr);         \
            return BFC_ERR_OUT_OF_MEMORY;                                             \
        }                                                                             \
    } while (0)
    // kept arrays (those of prepare_graph for a batch)
    GET(g->err, 4); GET(g->rank_u, r); GET(g->rank_l, l); GET(g->off, (int64_t)n + 1);
    GET(g->adj, 2 * m); GET(g->eid, 2 * m); GET(g->plen, 2 * m); GET(g->cut, n); GET(g->work, n);
    GET(g->cursors, 8 + 4); GET(g->pv, 1); GET(g->sbeg, 2 * m);
    g->acc = reinterpret_cast<unsigned long long *>(g->cursors + 8);   // cleared together
    GET(g->gstar, n); GET(g->vbase, n); GET(g->vend, n); GET(g->gwork, G);
    g->bcut = g->cut;
    g->boff = g->off;
    if (!g->opt.validate) {
        GET(pl->bcut, n); GET(pl->boff, (int64_t)n + 1);
        g->bcut = pl->bcut;
        g->boff = pl->boff;
    }
    GET(g->cta_items, n); GET(g->team_items, n); GET(g->warp_items, n); GET(g->retry, 1);
    // temporaries, kept with the plan
    const int64_t nsort = std::max<int64_t>({(int64_t)r, (int64_t)l, m, (int64_t)n, 1});
    GET(pl->k0, nsort + 1); GET(pl->k1, nsort + 1); GET(pl->v0, nsort); GET(pl->v1, nsort);
    GET(pl->deg_u, r); GET(pl->deg_l, l); GET(pl->deg_star, n);
    GET(pl->rows_star, 2 * m); GET(pl->big, n);
    GET(pl->tier_rows, kRowTiers * (int64_t)std::max(r, 1));
    GET(pl->hist, radix_hist_elems(nsort));
    GET(pl->hist_tmp, scan_tmp_elems<uint32_t>((int64_t)radix_hist_elems(nsort)));
    GET(pl->scan64_tmp, std::max(scan_tmp_elems<int64_t>((int64_t)n + 1), max_scan_tmp_elems(m)));
    GET(pl->deg64, (int64_t)n + 1); GET(pl->red, kRedWords); GET(pl->heavy, n);
    pl->n_big = reinterpret_cast<int32_t *>(pl->red + 12);
    pl->tier_n = pl->n_big + 2;
#undef GET
    // every kept array starts zeroed: a run that stops at the checks leaves
    // arrays that later kernels can still index safely
    for (int i = 0; i < g->mem.n; ++i) BFC_CUDA(cudaMemsetAsync(g->mem.ptr[i], 0, g->mem.bytes[i], s));
    g->n_cta_items = 0; g->n_team_items = 0; g->n_warp_items = 0;   // a run's are in device memory
    g->schedule_rc = BFC_OK;
    g->retry_static = 0; g->retry_cap = 1; g->may_retry = false;
    g->info.num_u = r; g->info.num_l = l; g->info.num_edges = m;
    g->info.device_bytes = (int64_t)g->mem.total;
    // the radix sort's and the count's kernel attributes are set here, outside
    // any capture: a two-key sort and the count's per-device setup
    int which = 0;
    BFC_CUDA(radix_sort_pairs(pl->k0, pl->v0, pl->k1, pl->v1, 2, 0, 8, pl->hist, pl->hist_tmp, s, &which));
    int rc = count_smem_setup(g->device);
    if (rc == BFC_OK) rc = rows_smem_setup(g->device);
    if (rc) return rc;
    BFC_CUDA(cudaStreamSynchronize(s));
    return BFC_OK;
}

int batch_plan_run(BatchPlan *pl, const int32_t *off_u, const int32_t *adj_u, const int32_t *gu,
                   const int32_t *gl, cudaStream_t s, unsigned long long *totals, int32_t *status) {
    Graph *g = &pl->g;
    const int32_t r = pl->r, l = pl->l, n = r + l, G = pl->num_graphs;
    const int64_t m = pl->m;
    const int *guard = g->err;
    g->stream = s;
    const bfc_options *opt = &g->opt;
    BFC_CUDA(cudaMemsetAsync(g->err, 0, 4 * sizeof(int), s));
    // ---- checks: the CSR, the graph start arrays, edges inside their graph
    k_check_starts<<<blocks_for((int64_t)G + 1), kT, 0, s>>>(gu, G, r, g->err, pl->max_layer); note_launch();
    k_check_starts<<<blocks_for((int64_t)G + 1), kT, 0, s>>>(gl, G, l, g->err, pl->max_layer); note_launch();
    BFC_CUDA(cudaGetLastError());
    // ---- a1: degrees (and the check of the L ids)
    BFC_CUDA(cudaMemsetAsync(pl->deg_l, 0, sizeof(int32_t) * std::max<int64_t>(l, 1), s));
    k_check_input<<<grid_stride_blocks(std::max<int64_t>(m, (int64_t)r + 1)), kT, 0, s>>>(
        off_u, adj_u, r, l, m, pl->deg_u, pl->deg_l, g->err); note_launch();
    BFC_CUDA(cudaGetLastError());
    BFC_CUDA(cudaMemsetAsync(pl->red, 0, kRedWords * sizeof(unsigned long long), s));
    // ---- a2: graph-major ranks; without duplicates a degree is below 2^16 (at most the other layer)
    int rc = launch_ranks(g, pl->deg_l, pl->deg_u, gl, gu, degree_bound(opt, pl->max_layer, m), pl->k0, pl->v0, pl->k1, pl->v1, pl->hist,
                          pl->hist_tmp, pl->deg_star, pl->deg64, pl->red + 9, s, guard);
    if (rc) return rc;
    if (n > 0) {
        k_graph_star<<<grid_stride_blocks(n), kT, 0, s>>>(r, l, gu, gl, G, g->gstar, g->vbase, g->vend, guard); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    BFC_CUDA(scan_exclusive<int64_t>(pl->deg64, g->off, n, pl->scan64_tmp, s));
    // ---- a3: G*
    const int bu = bits_for(r > 0 ? (uint64_t)(r - 1) : 0);
    const int bl = bits_for(l > 0 ? (uint64_t)(l - 1) : 0);
    if (m > 0) {
        const URowOut uo{m, l, bu, g->off, g->adj, g->eid, pl->rows_star, pl->k1, g->err,
                         opt->validate ? kErrDuplicate : kErrParallel};
        // duplicate edges that the caller answers for keep their order in every row
        // but the longest
        if (!opt->validate) { k_check_batch_rows<<<grid_stride_blocks(r), kT, 0, s>>>(off_u, adj_u, r, gu, gl, G, g->err, guard); note_launch(); }
        rc = launch_u_rows(off_u, adj_u, g, pl->max_layer, gu, gl, G, opt->validate ? 1 : 2, uo, pl->tier_rows, pl->tier_n,
                           s, guard);
        if (rc) return rc;
        // L side: stable sort of the swapped keys on their rank_l bits
        int which2 = 0;
        BFC_CUDA(radix_sort_pairs(pl->k1, pl->v1, pl->k0, pl->v0, m, bu, bu + bl, pl->hist, pl->hist_tmp, s, &which2, true));
        const uint64_t *k2 = which2 ? pl->k0 : pl->k1;
        const int32_t *v2 = which2 ? pl->v0 : pl->v1;
        BFC_CUDA(cudaMemsetAsync(g->plen + m, 0, sizeof(int32_t) * (size_t)m, s));
        k_emit_l_side<true><<<grid_stride_blocks(m), kT, 0, s>>>(k2, v2, m, bu, l, g->off, g->adj, g->eid,
                                                                  pl->rows_star, g->plen, g->sbeg, !opt->validate, guard); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    // ---- a4: cut, runs, work
    if (n > 0) {
        BFC_CUDA(cudaMemsetAsync(g->gwork, 0, sizeof(unsigned long long) * G, s));
        launch_work(g, pl->deg_star, pl->big, pl->n_big, s, guard);
        BFC_CUDA(cudaGetLastError());
    }
    // ---- a5: heaviest first, bins from device counts
    // bins by compaction, then the heavy starts heaviest first: how many there
    // are is not known here, so the sort covers n keys of one byte (the rest
    // hold the largest key and stay behind), which order them to a quarter octave
    unsigned long long *bins = pl->red + 3;
    if (n > 0) {
        const BinBounds bb{(uint64_t)opt->warp_max_work, pl->team_max, (uint64_t)opt->hash_max_work, l, n, n, g->cut};
        rc = bin_starts(g, s, bb, bins, pl->heavy, pl->red, guard);
        if (rc) return rc;
        k_sched_keys_plan<<<blocks_for(n), kT, 0, s>>>(g->work, pl->heavy, n, bb, bins, pl->k0); note_launch();
        BFC_CUDA(cudaGetLastError());
        int which = 0;
        BFC_CUDA(radix_sort_pairs(pl->k0, pl->heavy, pl->k1, pl->v1, n, 0, 8, pl->hist, pl->hist_tmp, s, &which));
        if (!opt->validate) {
            // a dense start is one chunk of up to 65,535 ends, so of 16-bit counters
            k_count_bounds<<<grid_stride_blocks((int64_t)n + 1), kT, 0, s>>>(
                g->work, g->cut, g->off, n, (int32_t)kNarrowMaxCut, g->err, pl->bcut, pl->boff); note_launch();
            BFC_CUDA(cudaGetLastError());
        }
        k_emit_items_plan<<<grid_stride_blocks(n), kT, 0, s>>>(which ? pl->v1 : pl->heavy, bins, g->bcut, g->boff,
                                                               g->vbase, g->cta_items, g->team_items, guard); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    // ---- a6-a7: one persistent count; per-graph totals
    BFC_CUDA(cudaMemsetAsync(totals, 0, sizeof(unsigned long long) * G, s));
    g->item_counts = bins;
    rc = launch_count(g, s, kModeBatch, nullptr, nullptr, totals);
    if (rc) return rc;
    if (status) {
        k_plan_status<<<1, 1, 0, s>>>(g->err, opt->validate, status); note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    return BFC_OK;
}

}  // namespace bfc
