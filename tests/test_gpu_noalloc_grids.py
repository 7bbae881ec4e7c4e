"""The allocation-free count on devices with fewer resident CTAs than there are tiles of
1,024 vertices: its source is compiled into a program that launches smaller grids."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from bfc_inputs import generators as G

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "noalloc.cu"
namespace bfc {
void set_last_error(const std::string &) {}
void note_launch() {}
int cuda_fail(cudaError_t e, const char *what) { printf("%s: %s\n", what, cudaGetErrorString(e)); return BFC_ERR_CUDA; }
}  // namespace bfc
int main(int argc, char **argv) {
    FILE *f = fopen(argv[1], "rb");
    int32_t head[3];
    if (!f || fread(head, 4, 3, f) != 3) return 1;
    std::vector<int32_t> a(head[0] + 1 + head[2]);
    if (fread(a.data(), 4, a.size(), f) != a.size()) return 1;
    int32_t *dev;
    unsigned long long *out, total;
    if (cudaMalloc(&dev, 4 * a.size()) || cudaMalloc(&out, 16)) return 1;
    if (cudaMemcpy(dev, a.data(), 4 * a.size(), cudaMemcpyHostToDevice)) return 1;
    int32_t *scratch, status;
    int whole;
    if (bfc::noalloc_setup(0, &scratch, &whole)) return 1;
    for (int i = 2; i < argc; ++i) {
        const int grid = atoi(argv[i]);
        if (grid < 1 || grid > whole) return 1;
        bfc::g_na_grid[0] = grid;
        if (bfc_count_small_noalloc(head[0], head[1], head[2], dev, dev + head[0] + 1, nullptr, (uint64_t *)out,
                                    (int32_t *)(out + 1))) return 1;
        if (cudaMemcpy(&total, out, 8, cudaMemcpyDeviceToHost) || cudaMemcpy(&status, out + 1, 4, cudaMemcpyDeviceToHost)) return 1;
        printf("%d %llu\n", status, total);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("noalloc")
    (d / "grids.cu").write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1812_00283_gb300", "csrc"),
                    str(d / "grids.cu"), "-o", str(d / "grids")], check=True)
    return str(d / "grids")


@pytest.mark.parametrize("size", [(300, 200, 2000), (1024, 1024, 9000), (12_007, 8_001, 150_001), (49_152, 16_384, 300_000)])
def test_smaller_grids(program, tmp_path, size):
    g = G.chung_lu_bipartite(*size, 2.1, 2.2, 7)
    path = tmp_path / "graph.bin"
    with open(path, "wb") as f:
        for a in ([g.num_u, g.num_l, g.num_edges], g.off_u, g.adj_u):
            np.asarray(a, dtype=np.int32).tofile(f)
    grids = [1, 2, 7, 63, 64, 65]
    r = subprocess.run([program, str(path), *map(str, grids)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.split("\n")[:-1] == [f"0 {oracle.vp(g)['total']}"] * len(grids)
