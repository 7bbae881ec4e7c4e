"""The list of pool allocations behind a prepared graph: pieces carved from slabs,
allocations of their own that a rebinning replaces, and the pool's refusal.  The list
is host code; it is compiled here against a pool that counts what it gave out.
Then one graph tuned again and again on the GPU.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from bfc_inputs import generators as G

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "bfc_internal.cuh"

static std::map<char *, size_t> live;
static size_t limit = ~size_t(0), in_use = 0;
static int failures = 0;
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); ++failures; } } while (0)

namespace bfc {
cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t) {
    if (in_use + bytes > limit) return cudaErrorMemoryAllocation;
    *p = aligned_alloc(256, (bytes + 255) / 256 * 256);
    live[(char *)*p] = bytes;
    in_use += bytes;
    return cudaSuccess;
}
void pool_free(void *p, cudaStream_t) {
    CHECK(live.count((char *)p) == 1);
    in_use -= live[(char *)p];
    live.erase((char *)p);
    free(p);
}
}  // namespace bfc

// whether [p, p + b) lies in one block of the pool
static bool inside(const void *p, size_t b) {
    auto it = live.upper_bound((char *)p);
    if (it == live.begin()) return false;
    --it;
    return (char *)p + b <= it->first + it->second;
}

int main() {
    using bfc::Allocs;
    const size_t sizes[] = {0, 1, 255, 256, 257, 4096, 100000, 131071, 131072, 131073, 200000, 524287, 524288, 524289, 3000000};
    for (size_t first : {size_t(64) << 10, Allocs::kSlab}) {
        // carved and whole pieces: aligned, apart, and all of them given back
        Allocs a;
        a.slab_next = first;
        std::map<char *, size_t> got;
        for (size_t s : sizes) {
            char *p = nullptr;
            CHECK(a.get(&p, s) == cudaSuccess);
            CHECK((size_t)p % 256 == 0 && inside(p, s));
            got[p] = s;
        }
        char *end = nullptr;
        for (auto &e : got) { CHECK(e.first >= end); end = e.first + e.second; }
        CHECK(a.total == in_use && (size_t)a.n == live.size());
        a.release();
        CHECK(in_use == 0 && live.empty() && a.n == 0 && a.total == 0);

        // pieces of their own go back one by one, of every size, also where a
        // slab has the same size or starts the list
        char *kept = nullptr;
        CHECK(a.get(&kept, 1000) == cudaSuccess);
        for (size_t s : sizes) {
            const size_t before = in_use;
            const int n = a.n;
            for (int k = 0; k < 300; ++k) {
                char *p = nullptr, *q = nullptr;
                CHECK(a.get_own(&p, s) == cudaSuccess && a.get_own(&q, s) == cudaSuccess);
                CHECK(p != q && inside(p, s) && inside(q, s));
                a.drop(p);
                a.drop(q);
            }
            CHECK(in_use == before && a.n == n && a.total == in_use);
        }
        a.drop(nullptr);
        CHECK(inside(kept, 1000));

        // a piece of the current slab only where it fits
        const size_t held = in_use, rest = a.slab_left;
        char *c = nullptr;
        CHECK(!a.carve(&c, rest + 1) && c == nullptr && in_use == held);
        CHECK(a.carve(&c, rest < Allocs::kCarve ? rest : Allocs::kCarve) && inside(c, 256) && in_use == held);
        a.release();
        CHECK(in_use == 0);

        // a small list holds little more than it asked for
        size_t asked = 0;
        for (int k = 0; k < 40; ++k) {
            char *p = nullptr;
            CHECK(a.get(&p, 700 * k) == cudaSuccess);
            asked += 700 * k;
        }
        CHECK(a.total <= 2 * asked + first);
        a.release();

        // the pool's refusal is reported, and nothing is lost
        limit = 3000000;
        int ok = 0;
        char *p = nullptr;
        while (a.get(&p, 50000) == cudaSuccess) ++ok;
        CHECK(ok >= 40 && a.total == in_use);
        CHECK(a.get_own(&p, 3000000) != cudaSuccess && a.total == in_use);
        a.release();
        limit = ~size_t(0);
        CHECK(in_use == 0);
    }
    return failures != 0;
}
"""


def test_alloc_list(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "alloc_list.cu", tmp_path / "alloc_list"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1812_00283_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_chunk_table_of_a_batch_is_set_whole():
    # a count takes a batch's chunk table as two arrays: with only the first one set
    # (the pool refused the second) it would index the first as a single graph's
    src = open(os.path.join(ROOT, "paper_1812_00283_gb300", "csrc", "prepare.cu")).read()
    batch = src[src.index("if (ventries <= kChunkTableMaxEntries)"):]
    batch = batch[:batch.index("\n            }\n")]
    last_request = batch.rindex("GET(")
    assert 0 < last_request < batch.index("g->coff = ") and "&g->coff" not in batch and "g->mem, g->" not in batch


@pytest.mark.gpu
@pytest.mark.parametrize("orientation", [0, 1])
@pytest.mark.parametrize("size", [(2000, 3000, 20_000), (48_611, 31_013, 2_000_000)])
def test_tuned_again_and_again(size, orientation):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00283_gb300 import bfc
    g = G.chung_lu_bipartite(*size, 2.1, 2.2, 5)
    want = oracle.vp(g)["total"]
    off, adj = torch.from_numpy(np.ascontiguousarray(g.off_u)).cuda(), torch.from_numpy(np.ascontiguousarray(g.adj_u)).cuda()
    s = torch.cuda.current_stream().cuda_stream
    tot = torch.zeros(1, dtype=torch.int64, device="cuda")
    h = bfc.bfc_prepare(g.num_u, g.num_l, g.num_edges, off.data_ptr(), adj.data_ptr(), bfc.bfc_options_init(orientation=orientation), s)
    held = []
    try:
        for k in range(30):
            bfc.bfc_autotune(h, s, 1)
            held.append(bfc.bfc_graph_info(h)["device_bytes"])
            if k % 10 == 9:
                tot.fill_(-1)
                bfc.bfc_count(h, s, tot.data_ptr())
                bfc.bfc_sync(h, s)
                assert int(tot.item()) == want
    finally:
        bfc.bfc_release(h)
    assert len(set(held)) == 1, held   # every bound has been tried after the first tuning
