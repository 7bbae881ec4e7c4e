// bfc_count_small_noalloc: an exact butterfly count for small graphs that
// allocates nothing.
//
// Who needs it: code that may not call cudaMalloc or any allocating routine
// at the point where it counts -- for example a caller whose memory is fully
// reserved up front by its own allocator and that may not grow the device
// footprint, or a real-time loop that must not hit the driver's allocator
// (which can synchronise the device).  The regular entry points
// (bfc_prepare and friends) allocate the renumbered graph from a pool, so
// they are not usable there.
//
// How: every byte of working memory this entry point needs lives in one
// file-scope __device__ array of fixed size (below), which every GPU that
// loads the library holds until the process exits.  The caller passes only
// inputs and outputs.  The whole count is one cooperative kernel: it clears
// the scratch it uses, checks the CSR, ranks all vertices by Definition 3,
// writes both sides' lists as 16-bit ranks (the filter p(w) < p(x) is then one
// comparison, with no degree lookup per wedge) and counts with Algorithm 2:
// a start with at most 768 possible wedges by one warp with a hash table, a
// heavier one by a CTA with dense 16-bit counters.  A count of a simple graph
// is at most 49,152; edges that occur more than once can take one past 16 bits,
// which the counter's own increments show: the heavy starts are then counted
// again with 32-bit counters over halves of the ranks.
#include <cooperative_groups.h>

#include <mutex>

#include "bfc_internal.cuh"

namespace cg = cooperative_groups;

namespace bfc {
namespace {

constexpr int kNaThreads = 1024;                  // one CTA of 32 warps per SM
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaSmemBytes = 192 * 1024;          // dynamic shared memory: counters, tables, sorts
constexpr int32_t kNaMaxVertices = 65536;         // |U| + |L|: ranks fit 16 bits
constexpr int32_t kNaMaxLayer = 49152;
constexpr int64_t kNaMaxEdges = 1 << 20;          // 1,048,576 edges
constexpr int kNaTiles = kNaMaxVertices / kNaThreads;
constexpr int kNaDigits = 256;                    // rank classes: degrees 0..254 and "255 or more"
// the degrees add up to 2m, so at most 2m / 255 vertices are in the last class
constexpr int kNaMaxHigh = 8224;
static_assert(2 * kNaMaxEdges / 255 <= kNaMaxHigh, "high-degree list too small");
constexpr int kNaSlots = 1024;                    // hash slots per warp
constexpr int32_t kNaLightWork = kNaSlots / 4 * 3;
constexpr int kNaBigList = 512;                   // a middle's list above this is read by the whole CTA
constexpr int kNaMaxBig = (int)(2 * kNaMaxEdges / kNaBigList);
constexpr int kNaCntBytes = kNaMaxVertices * 2;   // 16-bit counters by rank
constexpr int32_t kNaWide = kNaCntBytes / 4;      // ranks per 32-bit pass
static_assert(kNaCntBytes + kNaMaxBig * 2 <= kNaSmemBytes, "counters and big-list queue");
static_assert(kNaWarps * kNaSlots * 4 <= kNaSmemBytes, "warp tables");
static_assert(16384 * 8 <= kNaSmemBytes && kNaMaxHigh <= 16384, "high-degree sort");
static_assert(kNaWarps * kNaDigits * 4 <= kNaSmemBytes, "per-warp digit counts");
// words: header | deg[n] | rank[n] | vstart[n] | vdeg[n] | items[n] | lpos[l] |
// tile histograms | high-degree list | lists as 16-bit ranks [2m]
constexpr int kNaHeader = 16;
constexpr int64_t kNaWords = kNaHeader + 5ll * kNaMaxVertices + kNaMaxLayer + kNaTiles * kNaDigits + kNaMaxHigh +
                             kNaMaxEdges;

}  // namespace
}  // namespace bfc

// The shared scratch of bfc_count_small_noalloc (about 5.8 MB).
static __device__ __align__(256) int32_t g_noalloc_scratch[bfc::kNaWords];

namespace bfc {
namespace {

// Where the scratch's parts begin.
struct NaScratch {
    unsigned long long *acc;
    int32_t *err, *cursor, *n_heavy, *n_light, *q_heavy, *q_light, *q_again;
    int32_t *deg;      // [n] by global id (L vertex v -> v, U vertex u -> l + u)
    int32_t *rank;     // [n] by global id: position in Definition 3's order
    int32_t *vstart;   // [n] by rank: where the vertex's list starts in `adj`
    int32_t *vdeg;     // [n] by rank: its length
    int32_t *items;    // [n] heavy starts from the front, light ones from the back
    int32_t *lpos;     // [l] next free position of each L list
    int32_t *thist;    // [tiles][256]
    int32_t *high;     // vertices of degree 255 or more, ascending global id
    uint16_t *adj;     // [2m] neighbours' ranks: L lists, then U lists at m + off_u
    __device__ NaScratch(int32_t *s, int32_t n, int32_t l) {
        acc = reinterpret_cast<unsigned long long *>(s);   // [4]: light starts, heavy ones, the same again, -
        err = s + 8; cursor = s + 9; n_heavy = s + 10; n_light = s + 11; q_heavy = s + 12; q_light = s + 13; q_again = s + 14;
        deg = s + kNaHeader;
        rank = deg + n;
        vstart = rank + n;
        vdeg = vstart + n;
        items = vdeg + n;
        lpos = items + n;
        thist = lpos + l;
        high = thist + kNaTiles * kNaDigits;
        adj = reinterpret_cast<uint16_t *>(high + kNaMaxHigh);
    }
};

// The wedges through up to 32 middles, lane i's being the list [s, s + d)
// (d = 0: none): eight lanes per middle, four middles at a time; op(w) for
// every end rank w below rx.  Called by whole warps.
template <class Op>
__device__ __forceinline__ void na_middles(const uint16_t *adj, int32_t s, int32_t d, int32_t rx,
                                           int lane, Op op) {
    const int g = lane >> 3, j = lane & 7;
    uint32_t left = __ballot_sync(0xffffffffu, d > 0);
    while (left) {
        // the four lowest lanes still to do, one per group
        int src = -1;
        uint32_t m = left;
        for (int k = 0; k < 4; ++k) {
            const int f = __ffs((int)m) - 1;   // -1 when none is left
            if (k == g) src = f;
            m &= m - 1;
        }
        left = m;
        const int32_t gs = __shfl_sync(0xffffffffu, s, src & 31);
        int32_t gd = __shfl_sync(0xffffffffu, d, src & 31);
        if (src < 0) gd = 0;
        for (int32_t k = j; __any_sync(0xffffffffu, k < gd); k += 32) {
            int32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = k + 8 * u < gd ? (int32_t)adj[gs + k + 8 * u] : 0x7fffffff;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (w[u] < rx) op(w[u]);
        }
    }
}

// What bounds it: latency.  A small graph is a chain of dependent passes over a
// few hundred KB with a grid barrier between them, then starts of a few
// microseconds each.  On 12,007 x 8,001 vertices with 150,001 edges 132 us; 521 us
// when each row's list was built by one thread and every start took a CTA.
__global__ void __launch_bounds__(kNaThreads, 1)
k_count_noalloc(int32_t r, int32_t l, int32_t m, const int32_t *__restrict__ off_u,
                const int32_t *__restrict__ adj_u, int32_t *scratch,
                unsigned long long *total_out, int32_t *status_out) {
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long red[64];
    __shared__ int32_t sh_item, sh_nbig, sh_part[32], sh_base[kNaDigits];

    const int32_t n = r + l;
    const NaScratch S(scratch, n, l);
    const int32_t gtid = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
    const int32_t gstride = (int32_t)(gridDim.x * blockDim.x);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t gwarp = gtid >> 5, gwarps = gstride >> 5;
    const uint32_t lt = (1u << lane) - 1u;

    // clear what must start at zero (the scratch keeps the previous call's contents)
    if (gtid < kNaHeader) scratch[gtid] = 0;
    for (int32_t i = gtid; i < l; i += gstride) S.deg[i] = 0;
    grid.sync();

    // the CSR must be a CSR before anything indexes with it; degrees
    for (int32_t u = gtid; u <= r; u += gstride) {
        const int32_t o = off_u[u];
        if (u == 0 && o != 0) atomicOr(S.err, 1);
        if (u == r && o != m) atomicOr(S.err, 1);
        if (u < r) {
            const int32_t d = off_u[u + 1] - o;
            if (off_u[u + 1] < o) atomicOr(S.err, 1);
            S.deg[l + u] = d;
        }
    }
    for (int32_t k = gtid; k < m; k += gstride) {
        const int32_t v = adj_u[k];
        if (v < 0 || v >= l) atomicOr(S.err, 2);
        else atomicAdd(&S.deg[v], 1);
    }
    grid.sync();
    if (*((volatile int32_t *)S.err) != 0) {   // the same in every thread of the grid
        if (gtid == 0) {
            *total_out = 0ull;
            if (status_out) *status_out = BFC_ERR_INVALID_GRAPH;
        }
        return;
    }

    // ranks: vertices in (degree, global id) order.  One stable counting pass
    // over 256 classes (degrees 0..254 exactly, the rest in the last class),
    // in tiles of 1,024 vertices, one per CTA where there are 64 CTAs; then the
    // few vertices of the last class are sorted by one CTA.
    uint32_t *const wcnt = reinterpret_cast<uint32_t *>(smem_raw);   // [32 warps][256]
    const int tiles = (n + kNaThreads - 1) / kNaThreads;
    int32_t digit = 0, before = 0, id = 0;   // this thread's class and its place among its warp's, its vertex
    // wcnt[w][c] = how many of class c the tile's warps before w hold; returns
    // (for c = tid) how many the tile holds
    auto tile_classes = [&](int tile) {
        id = tile * kNaThreads + tid;
        uint32_t run = 0;
        __syncthreads();
        for (int i = tid; i < kNaWarps * kNaDigits; i += kNaThreads) wcnt[i] = 0;
        __syncthreads();
        digit = id < n ? min(S.deg[id], kNaDigits - 1) : kNaDigits;
        const uint32_t peers = __match_any_sync(0xffffffffu, digit);
        before = __popc(peers & lt);
        if (id < n && before == 0) wcnt[warp * kNaDigits + digit] = __popc(peers);
        __syncthreads();
        if (tid < kNaDigits) {
            for (int w = 0; w < kNaWarps; ++w) {
                const uint32_t c = wcnt[w * kNaDigits + tid];
                wcnt[w * kNaDigits + tid] = run;
                run += c;
            }
        }
        return run;
    };
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const uint32_t run = tile_classes(tile);
        if (tid < kNaDigits) S.thist[tile * kNaDigits + tid] = (int32_t)run;
    }
    // L lists: 32 at a time take their room from one cursor (any order)
    for (int32_t v0 = gwarp * 32; v0 < l; v0 += gwarps * 32) {
        const int32_t v = v0 + lane, d = v < l ? S.deg[v] : 0;
        int32_t incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        int32_t at = 0;
        if (lane == 31) at = atomicAdd(S.cursor, incl);
        at = __shfl_sync(0xffffffffu, at, 31) + incl - d;
        if (v < l) S.lpos[v] = at;
    }
    grid.sync();
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        if (tiles > (int)gridDim.x) tile_classes(tile);   // a CTA's only tile keeps what it counted
        // class starts: all tiles of the lower classes, and the lower tiles of this one
        int32_t all = 0, mine = 0;
        if (tid < kNaDigits)
            for (int t = 0; t < tiles; ++t) {
                const int32_t c = S.thist[t * kNaDigits + tid];
                if (t < tile) mine += c;
                all += c;
            }
        int32_t incl = all;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sh_part[warp] = incl;
        __syncthreads();
        if (tid < kNaDigits) {
            int32_t lower = 0;
            for (int w = 0; w < warp; ++w) lower += sh_part[w];
            sh_base[tid] = lower + incl - all + mine;
            if (tid == kNaDigits - 1) sh_item = lower + incl - all;   // first rank of the last class
        }
        __syncthreads();
        if (id < n) {
            const int32_t rk = sh_base[digit] + (int32_t)wcnt[warp * kNaDigits + digit] + before;
            if (digit == kNaDigits - 1) {
                S.high[rk - sh_item] = id;
            } else {
                S.rank[id] = rk;
                S.vstart[rk] = id < l ? S.lpos[id] : m + off_u[id - l];
                S.vdeg[rk] = S.deg[id];
            }
        }
    }
    grid.sync();
    if (blockIdx.x == 0) {   // the last class: ascending (degree, id) by a bitonic sort
        const int32_t first = n > 0 ? sh_item : 0, nh = n - first;
        uint64_t *const buf = reinterpret_cast<uint64_t *>(smem_raw);
        int np = 1;
        while (np < nh) np <<= 1;
        if (nh > 0) {
            for (int i = tid; i < np; i += kNaThreads)
                buf[i] = i < nh ? ((uint64_t)(uint32_t)S.deg[S.high[i]] << 32) | (uint32_t)S.high[i] : ~0ull;
            __syncthreads();
            for (int k = 2; k <= np; k <<= 1)
                for (int j = k >> 1; j > 0; j >>= 1) {
                    for (int i = tid; i < np; i += kNaThreads) {
                        const int ij = i ^ j;
                        if (ij > i) {
                            const uint64_t a = buf[i], c = buf[ij];
                            if ((a > c) == ((i & k) == 0)) { buf[i] = c; buf[ij] = a; }
                        }
                    }
                    __syncthreads();
                }
            for (int i = tid; i < nh; i += kNaThreads) {
                const int32_t v = (int32_t)(uint32_t)buf[i], rk = first + i;
                S.rank[v] = rk;
                S.vstart[rk] = v < l ? S.lpos[v] : m + off_u[v - l];
                S.vdeg[rk] = S.deg[v];
            }
        }
    }
    grid.sync();

    // both sides' lists as ranks; an edge finds its row by a binary search
    for (int32_t k = gtid; k < m; k += gstride) {
        const int32_t v = adj_u[k];
        int32_t lo = 0, hi = r;   // last u with off_u[u] <= k (the one with a non-empty row)
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (off_u[mid] <= k) lo = mid; else hi = mid;
        }
        S.adj[m + k] = (uint16_t)S.rank[v];
        S.adj[atomicAdd(&S.lpos[v], 1)] = (uint16_t)S.rank[l + lo];
    }
    grid.sync();

    // starts: one with at most one possible wedge closes no butterfly; a light
    // one has at most 768
    for (int32_t i = gwarp; i < n; i += gwarps) {
        const int32_t x = n - 1 - i, s = S.vstart[x], d = S.vdeg[x];
        if (d < 2) continue;
        int32_t bound = 0;
        bool heavy = d > 1024;
        for (int32_t j = lane; !heavy && j - lane < d; j += 32) {
            const int32_t v = j < d ? (int32_t)S.adj[s + j] : 0x7fffffff;
            const int32_t b = v < x ? min(S.vdeg[v] - 1, kNaLightWork + 1) : 0;
            bound += (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)b);
            heavy = bound > kNaLightWork;   // the same in every lane
        }
        if (!heavy && bound < 2) continue;
        if (lane == 0) {
            if (heavy) S.items[atomicAdd(S.n_heavy, 1)] = x;
            else S.items[n - 1 - atomicAdd(S.n_light, 1)] = x;
        }
    }
    grid.sync();

    // Algorithm 2: Σ old over the increments of count_wedge(w) = Σ C(count, 2),
    // the heavy starts' apart from the light ones'
    unsigned long long acc = 0, acc_light = 0;
    const int32_t n_heavy = *((volatile int32_t *)S.n_heavy), n_light = *((volatile int32_t *)S.n_light);
    // the wedges of heavy start x, by the whole CTA (sh_nbig is zero); flush()
    // follows at most 1,024 calls of op(w) by a thread, unless more long lists
    // are met than a simple graph has
    auto heavy_walk = [&](int32_t x, auto op, auto flush) {
        uint16_t *const big = reinterpret_cast<uint16_t *>(smem_raw + kNaCntBytes);
        const int32_t s = S.vstart[x], d = S.vdeg[x];
        for (int32_t j0 = warp * 32; j0 < d; j0 += kNaThreads) {
            const int32_t v = j0 + lane < d ? (int32_t)S.adj[s + j0 + lane] : 0x7fffffff;
            int32_t vs = 0, vd = 0;
            if (v < x) { vs = S.vstart[v]; vd = S.vdeg[v]; }
            if (vd > kNaBigList) {
                const int at = atomicAdd(&sh_nbig, 1);
                if (at < kNaMaxBig) { big[at] = (uint16_t)v; vd = 0; }   // else this warp reads it
            }
            na_middles(S.adj, vs, vd, x, lane, op);
            flush();
        }
        __syncthreads();
        const int nbig = min(sh_nbig, kNaMaxBig);
        for (int b = 0; b < nbig; ++b) {
            const int32_t v = big[b], vs = S.vstart[v], vd = S.vdeg[v];
            for (int32_t k = tid; k < vd; k += kNaThreads) {
                const int32_t w = S.adj[vs + k];
                if (w < x) op(w);
            }
            flush();
        }
    };
    uint32_t *const cnt = reinterpret_cast<uint32_t *>(smem_raw);
    auto clear = [&](int32_t words) {
        uint4 *const c4 = reinterpret_cast<uint4 *>(smem_raw);
        for (int32_t i = tid; i < (words + 3) / 4; i += kNaThreads) c4[i] = make_uint4(0, 0, 0, 0);
    };
    {
        uint32_t sum = 0;   // Σ old since the last flush: below 2^26
        uint32_t top = 0;   // the largest count that this thread has added to
        for (;;) {          // 16-bit counters, two per word
            __syncthreads();
            if (tid == 0) { sh_item = atomicAdd(S.q_heavy, 1); sh_nbig = 0; }
            __syncthreads();
            const int32_t it = sh_item;
            if (it >= n_heavy) break;
            const int32_t x = S.items[it];
            clear((x + 1) / 2);
            __syncthreads();
            heavy_walk(x, [&](int32_t w) {
                const uint32_t sh = (uint32_t)(w & 1) << 4;
                const uint32_t old = (atomicAdd(cnt + (w >> 1), 1u << sh) >> sh) & 0xffffu;
                top = max(top, old);
                sum += old;
            }, [&]() { acc += sum; sum = 0; });
            if (sh_nbig > kNaMaxBig) top = 0xffffu;   // those lists were read by one warp each
        }
        if (top == 0xffffu) atomicOr(S.err, 8);   // a counter wrapped, or a sum may have
    }
    {
        // light starts: a table of (rank, count) words per warp; a rank below
        // x is never 65,535, so all ones marks an empty slot
        uint32_t *const tab = reinterpret_cast<uint32_t *>(smem_raw) + warp * kNaSlots;
        for (;;) {
            int32_t it = 0;
            if (lane == 0) it = atomicAdd(S.q_light, 1);
            it = __shfl_sync(0xffffffffu, it, 0);
            if (it >= n_light) break;
            const int32_t x = S.items[n - 1 - it], s = S.vstart[x], d = S.vdeg[x];
            uint4 *const t4 = reinterpret_cast<uint4 *>(tab);
            for (int i = lane; i < kNaSlots / 4; i += 32) t4[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
            __syncwarp();
            auto op = [&](int32_t w) {
                uint32_t h = ((uint32_t)w * 0x9E3779B1u) >> 22;   // 10 bits
                static_assert(kNaSlots == 1024, "ten hash bits");
                for (int probe = 0; probe < kNaSlots; ++probe) {
                    uint32_t e = *((volatile uint32_t *)(tab + h));
                    if (e == ~0u) {
                        e = atomicCAS(tab + h, ~0u, ((uint32_t)w << 16) | 1u);
                        if (e == ~0u) return;
                    }
                    if ((e >> 16) == (uint32_t)w) {
                        acc_light += atomicAdd(tab + h, 1u) & 0xffffu;
                        return;
                    }
                    h = (h + 1) & (kNaSlots - 1);
                }
                atomicOr(S.err, 4);   // cannot happen: at most 768 distinct ends
            };
            for (int32_t j0 = 0; j0 < d; j0 += 32) {
                const int32_t v = j0 + lane < d ? (int32_t)S.adj[s + j0 + lane] : 0x7fffffff;
                int32_t vs = 0, vd = 0;
                if (v < x) { vs = S.vstart[v]; vd = S.vdeg[v]; }
                na_middles(S.adj, vs, vd, x, lane, op);
            }
            __syncwarp();
        }
    }
    // two sums over the grid, added to to[0] and to[1]
    auto grid_sums = [&](unsigned long long v, unsigned long long v1, unsigned long long *to) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            v += __shfl_xor_sync(0xffffffffu, v, d);
            v1 += __shfl_xor_sync(0xffffffffu, v1, d);
        }
        if (lane == 0) { red[warp] = v; red[32 + warp] = v1; }
        __syncthreads();
        if (warp < 2) {
            unsigned long long t = red[32 * warp + lane];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
            if (lane == 0 && t) atomicAdd(to + warp, t);
        }
    };
    grid_sums(acc_light, acc, S.acc);
    grid.sync();
    const bool again = (*((volatile int32_t *)S.err) & 8) != 0;   // the same in every thread of the grid
    if (again) {   // the heavy starts with 32-bit counters, kNaWide ranks at a time
        acc = 0;
        for (;;) {
            __syncthreads();
            if (tid == 0) sh_item = atomicAdd(S.q_again, 1);
            __syncthreads();
            const int32_t it = sh_item;
            if (it >= n_heavy) break;
            const int32_t x = S.items[it];
            for (int32_t lo = 0; lo < x; lo += kNaWide) {
                __syncthreads();
                if (tid == 0) sh_nbig = 0;
                clear(min(x - lo, kNaWide));
                __syncthreads();
                heavy_walk(x, [&](int32_t w) {
                    if ((uint32_t)(w - lo) < (uint32_t)kNaWide) acc += atomicAdd(cnt + (w - lo), 1u);
                }, []() {});
            }
        }
        grid_sums(acc, 0, S.acc + 2);
        grid.sync();
    }
    if (gtid == 0) {
        const bool full = (*((volatile int32_t *)S.err) & 4) != 0;
        *total_out = *((volatile unsigned long long *)S.acc) + *((volatile unsigned long long *)(S.acc + (again ? 2 : 1)));
        if (status_out) *status_out = full ? BFC_ERR_INTERNAL : BFC_OK;
    }
}

std::mutex g_na_mutex;
int32_t *g_na_ptr[64] = {};
int g_na_grid[64] = {};

// Once per device, with that device current: the device address of the
// scratch array (the host-side name is only a stand-in), the kernel's shared
// memory attribute and the co-resident grid size.
int noalloc_setup(int dev, int32_t **ptr, int *grid) {
    std::lock_guard<std::mutex> lk(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        e = cudaFuncSetAttribute(k_count_noalloc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kNaSmemBytes);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(k_count_noalloc)");
        int sms = 0, per_sm = 0, coop = 0;
        e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        if (!coop) { set_last_error("device cannot launch cooperative kernels"); return BFC_ERR_CUDA; }
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_count_noalloc, kNaThreads,
                                                          kNaSmemBytes);
        if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
        if (per_sm < 1) { set_last_error("k_count_noalloc does not fit on an SM"); return BFC_ERR_CUDA; }
        g_na_grid[dev] = sms * per_sm;
        g_na_ptr[dev] = static_cast<int32_t *>(p);
    }
    *ptr = g_na_ptr[dev];
    *grid = g_na_grid[dev];
    return BFC_OK;
}

}  // namespace
}  // namespace bfc

extern "C" int bfc_count_small_noalloc(int32_t num_u, int32_t num_l, int64_t num_edges,
                                       const int32_t *off_u_dev, const int32_t *adj_u_dev,
                                       void *stream, uint64_t *total_dev, int32_t *status_dev) {
    bfc::set_last_error("");
    if (!off_u_dev || !total_dev || (num_edges > 0 && !adj_u_dev) || num_u < 0 || num_l < 0 ||
        num_edges < 0) {
        bfc::set_last_error("bfc_count_small_noalloc: null pointer or negative size");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    if ((int64_t)num_u + num_l > bfc::kNaMaxVertices || num_u > bfc::kNaMaxLayer ||
        num_l > bfc::kNaMaxLayer || num_edges > bfc::kNaMaxEdges) {
        bfc::set_last_error("bfc_count_small_noalloc: graph too large (limits: |U|, |L| <= 49152, "
                            "|U| + |L| <= 65536, edges <= 1048576)");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    int dev = 0;
    BFC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) { bfc::set_last_error("device index out of range"); return BFC_ERR_CUDA; }
    int32_t *scratch = nullptr;
    int grid = 0;
    int rc = bfc::noalloc_setup(dev, &scratch, &grid);
    if (rc) return rc;
    int32_t r = num_u, l = num_l, m = (int32_t)num_edges;
    unsigned long long *tot = reinterpret_cast<unsigned long long *>(total_dev);
    void *args[] = {&r, &l, &m, (void *)&off_u_dev, (void *)&adj_u_dev, &scratch, &tot, &status_dev};
    BFC_CUDA(cudaLaunchCooperativeKernel((const void *)bfc::k_count_noalloc, dim3(grid),
                                         dim3(bfc::kNaThreads), args, bfc::kNaSmemBytes,
                                         static_cast<cudaStream_t>(stream)));
    bfc::note_launch();
    return BFC_OK;
}
