// Approximate counting by edge sparsification (Section 7: the exact counter
// is the inner block of a sampling estimator, run on sampled graphs).
//
// Every sample keeps each edge independently with probability p.  A
// butterfly survives a sample iff its four edges do, so E[⋈(G_j)] = p^4 ⋈(G)
// and the mean of the samples' exact counts divided by p^4 estimates ⋈(G).
//
// The samples are built side by side as one disjoint union (sample j's U
// vertices at j·|U|.., its L vertices at j·|L|..), which is then prepared and
// counted as a batch: one set of sorts and scans for all samples and one
// persistent count launch with a total per sample.
//
// Keep rule (the same on every platform): sample j keeps the edge at U-side
// slot e iff the (j·m + e + 1)-th output of SplitMix64 seeded with `seed` is
// below floor(p · 2^64); p = 1 keeps every edge.  SplitMix64 is the generator
// of Steele, Lea and Flood (OOPSLA 2014).
#include <algorithm>
#include <cmath>

#include "bfc_internal.cuh"

namespace bfc {
namespace {

constexpr int kT = 256;

unsigned grid_for(int64_t threads) {
    return (unsigned)std::min<int64_t>(std::max<int64_t>((threads + kT - 1) / kT, 1), 152 * 32);
}

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t k) {
    uint64_t z = seed + k * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

struct SampleRule {
    uint64_t seed, threshold;
    int keep_all;
};

// offsets of a CSR: off[0] = 0, off[r] = m, non-decreasing (bit 0 of *bad)
__global__ void k_sp_check_offsets(const int32_t *__restrict__ off, int32_t r, int64_t m, int *bad) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u <= r;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int32_t o = off[u];
        const bool ok = (u == 0 ? o == 0 : o >= off[u - 1]) && (u < r || o == m);
        if (!ok) atomicOr(bad, 1);
    }
}

// The union's edges in order are the kept slots of sample 0, then of sample
// 1, ...: a stream compaction over the linear index (sample, slot), with no row
// in it.  Slots are taken 32 at a time: sample j has m / 32 + 1 words, bit i of
// word w = slot 32 w + i is kept (the last word reaches past slot m - 1, so that
// every row offset lies in a word of its sample).  The masks and their prefixes
// (8 bytes per word) are held for as many samples at a time as fit 2 GB; when
// that is not all of them the masks are drawn twice.
// Before: two passes of one warp per (sample, row), whose rows average 20 slots,
// 5.7 ms for 16 samples of a 20M-edge graph.
constexpr int kSpWords = kT;   // words per CTA: 32 per warp
constexpr int64_t kSpGroupBytes = 1ll << 31;

// Pass 1: the keep masks and the kept slots per CTA (and, for sample 0, a
// check of the L ids, bit 1 of *bad).  Bound by the draws' 64-bit integer
// multiplications.
__global__ void __launch_bounds__(kT) k_sp_masks(const int32_t *__restrict__ adj, int32_t l, int64_t m,
                                                 int32_t j0, int64_t words, int64_t all_words, SampleRule rule,
                                                 uint32_t *__restrict__ mask, int64_t *__restrict__ cnt, int *bad) {
    __shared__ int32_t part[kT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * kSpWords + warp * 32;
    uint32_t mine = 0;
    int64_t j = j0 + w0 / words, wj = w0 % words;   // sample, word of it
    for (int k = 0; k < 32 && w0 + k < all_words; ++k) {   // warp-uniform
        const int64_t e = wj * 32 + lane;
        const bool in = e < m;
        if (j == 0 && in) {
            const int32_t v = adj[e];
            if (v < 0 || v >= l) atomicOr(bad, 2);
        }
        const bool keep = in && (rule.keep_all ||
                                 splitmix64_at(rule.seed, (uint64_t)j * (uint64_t)m + 1 + (uint64_t)e) < rule.threshold);
        const uint32_t b = __ballot_sync(0xffffffffu, keep);
        if (k == lane) mine = b;
        if (++wj == words) { wj = 0; ++j; }
    }
    if (w0 + lane < all_words) mask[w0 + lane] = mine;
    const int32_t c = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)__popc(mine));
    if (lane == 0) part[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t t = 0;
        for (int w = 0; w < kT / 32; ++w) t += part[w];
        cnt[blockIdx.x] = t;
    }
}

// Pass 2: the kept L ids, shifted to their sample's range, in order; per word
// the kept slots before it.  The id check has passed, the union fits 32 bits.
__global__ void __launch_bounds__(kT) k_sp_compact(const int32_t *__restrict__ adj, int32_t l, int32_t j0,
                                                   int64_t words, int64_t all_words, const uint32_t *__restrict__ mask,
                                                   const int64_t *__restrict__ cnt_scan,
                                                   int32_t *__restrict__ wpre, int32_t *__restrict__ uadj) {
    __shared__ int32_t part[kT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)blockIdx.x * kSpWords + warp * 32;
    const uint32_t mine = w0 + lane < all_words ? mask[w0 + lane] : 0;
    const int32_t c = __popc(mine);
    int32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    int32_t at = (int32_t)cnt_scan[blockIdx.x] + incl - c;
    for (int w = 0; w < warp; ++w) at += part[w];
    if (w0 + lane < all_words) wpre[w0 + lane] = at;
    const uint32_t lt = (1u << lane) - 1u;
    int64_t j = j0 + w0 / words, wj = w0 % words;
    for (int k = 0; k < 32 && w0 + k < all_words; ++k) {   // warp-uniform
        const uint32_t b = __shfl_sync(0xffffffffu, mine, k);
        const int32_t p = __shfl_sync(0xffffffffu, at, k);
        if ((b >> lane) & 1u) uadj[p + __popc(b & lt)] = adj[wj * 32 + lane] + (int32_t)(j * l);
        if (++wj == words) { wj = 0; ++j; }
    }
}

// Pass 3: the union's row offsets: row (j, u) starts after the kept slots
// of sample j below off[u] (and all of the samples before it); and where each
// sample starts.
__global__ void k_sp_offsets(const int32_t *__restrict__ off, int32_t r, int32_t j0, int32_t group, int64_t words,
                             const uint32_t *__restrict__ mask, const int32_t *__restrict__ wpre,
                             int32_t *__restrict__ uoff, int32_t *__restrict__ sstart) {
    const int64_t rows = (int64_t)group * r;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows + group;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i >= rows) {
            sstart[j0 + (i - rows)] = wpre[(i - rows) * words];
            continue;
        }
        const int64_t j = i / r;
        const int32_t e = off[i - j * r];
        const int64_t w = j * words + (e >> 5);
        uoff[(int64_t)j0 * r + i] = wpre[w] + __popc(mask[w] & ((1u << (e & 31)) - 1u));
    }
}

// the union's last offset, the sample ranges and the kept edges per sample
__global__ void k_sp_ranges(const int32_t *__restrict__ sstart, int32_t kept, int32_t r, int32_t l,
                            int32_t samples, int32_t *uoff, int32_t *us, int32_t *ls, uint64_t *sample_edges) {
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j <= samples; j += gridDim.x * blockDim.x) {
        us[j] = (int32_t)((int64_t)j * r);
        ls[j] = (int32_t)((int64_t)j * l);
        if (j == samples) uoff[(int64_t)samples * r] = kept;
        if (sample_edges && j < samples)
            sample_edges[j] = (uint64_t)((j + 1 < samples ? sstart[j + 1] : kept) - sstart[j]);
    }
}

// estimate = Σ c_j / (samples · p^4); standard error = sd(c_j) / p^4 / sqrt(samples)
__global__ void k_sp_estimate(const uint64_t *__restrict__ counts, int32_t samples, double p, double *out) {
    __shared__ unsigned long long s_sum[kT];
    __shared__ double s_sq[kT];
    unsigned long long acc = 0;
    for (int32_t j = threadIdx.x; j < samples; j += blockDim.x) acc += counts[j];
    s_sum[threadIdx.x] = acc;
    __syncthreads();
    for (int d = kT / 2; d > 0; d >>= 1) {
        if (threadIdx.x < d) s_sum[threadIdx.x] += s_sum[threadIdx.x + d];
        __syncthreads();
    }
    const unsigned long long total = s_sum[0];
    const double mean = (double)total / (double)samples;
    double sq = 0.0;
    for (int32_t j = threadIdx.x; j < samples; j += blockDim.x) {
        const double d = (double)counts[j] - mean;
        sq += d * d;
    }
    s_sq[threadIdx.x] = sq;
    __syncthreads();
    for (int d = kT / 2; d > 0; d >>= 1) {
        if (threadIdx.x < d) s_sq[threadIdx.x] += s_sq[threadIdx.x + d];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double p4 = (p * p) * (p * p);
        out[0] = (double)total / ((double)samples * p4);
        out[1] = samples > 1 ? sqrt(s_sq[0] / (double)(samples - 1) / (double)samples) / p4 : (double)NAN;
    }
}

}  // namespace
}  // namespace bfc

extern "C" int bfc_prepare_sparsified(int32_t num_u, int32_t num_l, int64_t num_edges,
                                      const int32_t *off_u_dev, const int32_t *adj_u_dev, double p,
                                      uint64_t seed, int32_t num_samples, const bfc_options *opt,
                                      void *stream, uint64_t *sample_edges_dev, bfc_graph **out) {
    bfc::set_last_error("");
    if (!out) { bfc::set_last_error("null argument"); return BFC_ERR_INVALID_ARGUMENT; }
    *out = nullptr;
    if (num_u < 0 || num_l < 0 || num_edges < 0 || num_edges > 2147483647LL || !off_u_dev ||
        (num_edges > 0 && !adj_u_dev)) {
        bfc::set_last_error("invalid CSR arguments");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    if (!(p > 0.0 && p <= 1.0)) { bfc::set_last_error("keep probability must lie in (0, 1]"); return BFC_ERR_INVALID_ARGUMENT; }
    if (num_samples < 1 || (int64_t)num_samples * ((int64_t)num_u + num_l) > 2147483646LL) {
        bfc::set_last_error("num_samples must be >= 1 with num_samples * (|U| + |L|) below 2^31 - 1");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // p · 2^64 is exact in binary floating point; the conversion truncates
    const bfc::SampleRule rule{seed, p < 1.0 ? (uint64_t)std::ldexp(p, 64) : 0ull, p == 1.0 ? 1 : 0};
    bfc::Allocs a;
    a.stream = s;
    struct Guard { bfc::Allocs *a; ~Guard() { a->release(); } } guard{&a};
    const int64_t rows = (int64_t)num_samples * num_u;
    const int64_t words = num_edges / 32 + 1;
    const int32_t group = (int32_t)std::min<int64_t>(num_samples, std::max<int64_t>(bfc::kSpGroupBytes / (8 * words), 1));
    const int32_t groups = (num_samples + group - 1) / group;
    const int64_t gctas = (group * words + bfc::kSpWords - 1) / bfc::kSpWords;   // per group
    int *bad;
    int64_t *cnt, *cnt_scan, *scan_tmp;
    uint32_t *mask;
    int32_t *wpre, *uoff, *us, *ls, *sstart;
    if (a.get(&bad, 1) || a.get(&cnt, gctas * groups) || a.get(&cnt_scan, gctas * groups + 1) ||
        a.get(&scan_tmp, bfc::scan_tmp_elems<int64_t>(gctas * groups)) || a.get(&mask, group * words) ||
        a.get(&wpre, group * words) || a.get(&uoff, rows + 1) || a.get(&us, (size_t)num_samples + 1) ||
        a.get(&ls, (size_t)num_samples + 1) || a.get(&sstart, num_samples)) {
        bfc::set_last_error("device allocation failed: sample offsets");
        return BFC_ERR_OUT_OF_MEMORY;
    }
    // the masks of group g (every group but the last is full; a CTA past the
    // last one's words counts 0)
    auto draw = [&](int32_t g) {
        const int64_t all = std::min(group, num_samples - g * group) * words;
        bfc::k_sp_masks<<<(unsigned)gctas, bfc::kT, 0, s>>>(adj_u_dev, num_l, num_edges, g * group, words, all, rule,
                                                             mask, cnt + g * gctas, bad);
        bfc::note_launch();
        return cudaGetLastError();
    };
    BFC_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), s));
    bfc::k_sp_check_offsets<<<bfc::grid_for((int64_t)num_u + 1), bfc::kT, 0, s>>>(off_u_dev, num_u, num_edges, bad);
    bfc::note_launch();
    BFC_CUDA(cudaGetLastError());
    int hbad = 0;
    BFC_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    BFC_CUDA(cudaStreamSynchronize(s));
    if (hbad) { bfc::set_last_error("offsets are not a CSR of num_edges slots"); return BFC_ERR_INVALID_GRAPH; }
    for (int32_t g = 0; g < groups; ++g) BFC_CUDA(draw(g));
    BFC_CUDA(bfc::scan_exclusive<int64_t>(cnt, cnt_scan, gctas * groups, scan_tmp, s));
    int64_t kept = 0;
    BFC_CUDA(cudaMemcpyAsync(&kept, cnt_scan + gctas * groups, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    BFC_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    BFC_CUDA(cudaStreamSynchronize(s));
    if (hbad) { bfc::set_last_error("an L id lies outside [0, num_l)"); return BFC_ERR_INVALID_GRAPH; }
    if (kept > 2147483647LL) {
        bfc::set_last_error("the samples hold more than 2^31 - 1 edges together: use fewer samples");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    int32_t *uadj;
    if (a.get(&uadj, (size_t)std::max<int64_t>(kept, 1))) {
        bfc::set_last_error("device allocation failed: sampled edges");
        return BFC_ERR_OUT_OF_MEMORY;
    }
    for (int32_t g = 0; g < groups; ++g) {
        const int32_t j0 = g * group, gs = std::min(group, num_samples - j0);
        if (groups > 1) BFC_CUDA(draw(g));
        bfc::k_sp_compact<<<(unsigned)gctas, bfc::kT, 0, s>>>(adj_u_dev, num_l, j0, words, gs * words, mask,
                                                               cnt_scan + g * gctas, wpre, uadj);
        bfc::note_launch();
        BFC_CUDA(cudaGetLastError());
        bfc::k_sp_offsets<<<bfc::grid_for((int64_t)gs * num_u + gs), bfc::kT, 0, s>>>(off_u_dev, num_u, j0, gs, words,
                                                                                       mask, wpre, uoff, sstart);
        bfc::note_launch();
        BFC_CUDA(cudaGetLastError());
    }
    bfc::k_sp_ranges<<<bfc::grid_for((int64_t)num_samples + 1), bfc::kT, 0, s>>>(
        sstart, (int32_t)kept, num_u, num_l, num_samples, uoff, us, ls, sample_edges_dev);
    bfc::note_launch();
    BFC_CUDA(cudaGetLastError());
    const bfc_csr u{(int32_t)rows, (int32_t)((int64_t)num_samples * num_l), kept, uoff, uadj};
    const bfc_batch b{num_samples, us, ls};
    // the union's arrays go back to the pool in stream order after the prepare
    return bfc_prepare_batch(&u, &b, opt, stream, out);
}

extern "C" int bfc_sparsified_estimate(const uint64_t *sample_counts_dev, int32_t num_samples, double p,
                                       void *stream, double *estimate_dev) {
    bfc::set_last_error("");
    if (!sample_counts_dev || !estimate_dev || num_samples < 1) {
        bfc::set_last_error("null argument or num_samples < 1");
        return BFC_ERR_INVALID_ARGUMENT;
    }
    if (!(p > 0.0 && p <= 1.0)) { bfc::set_last_error("keep probability must lie in (0, 1]"); return BFC_ERR_INVALID_ARGUMENT; }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    bfc::k_sp_estimate<<<1, bfc::kT, 0, s>>>(sample_counts_dev, num_samples, p, estimate_dev);
    bfc::note_launch();
    BFC_CUDA(cudaGetLastError());
    return BFC_OK;
}

extern "C" int bfc_estimate_sparsified(int32_t num_u, int32_t num_l, int64_t num_edges,
                                       const int32_t *off_u_dev, const int32_t *adj_u_dev, double p,
                                       uint64_t seed, int32_t num_samples, const bfc_options *opt,
                                       void *stream, uint64_t *sample_counts_dev, double *estimate_dev) {
    bfc::set_last_error("");
    if (!sample_counts_dev) { bfc::set_last_error("null argument"); return BFC_ERR_INVALID_ARGUMENT; }
    bfc_graph *g = nullptr;
    int rc = bfc_prepare_sparsified(num_u, num_l, num_edges, off_u_dev, adj_u_dev, p, seed, num_samples, opt,
                                    stream, nullptr, &g);
    if (rc != BFC_OK) return rc;
    rc = bfc_count_batch(g, stream, sample_counts_dev, nullptr);
    if (rc == BFC_OK && estimate_dev) rc = bfc_sparsified_estimate(sample_counts_dev, num_samples, p, stream, estimate_dev);
    const int rs = bfc_sync(g, stream);
    bfc_release(g);
    return rc != BFC_OK ? rc : rs;
}
