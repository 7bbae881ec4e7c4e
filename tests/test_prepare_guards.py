"""The prepare kernels leave early when the input check's error word is set, and
the row kernels set that word themselves (an edge to another graph of a batch).
A kernel whose threads work together must therefore decide once per CTA, or per
warp: a CTA of which some warps left would go on with shared memory that
nobody wrote.  Read from the source, because the fault depends on timing; then one
malformed batch of several waves of CTAs on the GPU.
"""
import os
import re

import numpy as np
import pytest

from bfc_inputs import generators as G

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_00283_gb300", "csrc")


def _functions(text):
    """(name, is a kernel, header, body) of every function that starts in column 0."""
    text = re.sub(r"//[^\n]*", "", text)
    out = []
    for m in re.finditer(r"^(?:template <[^{;]*?>\s*)?((?:static |__global__ |__device__ )[^{;]*?\b(\w+)\(([^{;]*)\))\s*\{",
                         text, re.M):
        out.append((m.group(2), "__global__" in m.group(1), m.group(1), text[m.end():text.index("\n}\n", m.end())]))
    return out


def _scope(body, functions):
    """How closely the threads of a body work together: cta, warp or none."""
    if "__syncthreads" in body:
        return "cta"
    if re.search(r"__\w+_sync\(|__syncwarp", body):
        return "warp"
    for name, _, _, b in functions:
        if not name.startswith("aborted") and re.search(r"\b%s(<\w+>)?\(" % name, body) and re.search(r"_sync\(|__syncwarp", b):
            return "warp"
    return "none"


def test_kernels_leave_together():
    functions = _functions(open(os.path.join(CSRC, "prepare.cu")).read())
    guarded = [(n, h, b) for n, kernel, h, b in functions if kernel and "*guard" in h]
    assert len(guarded) >= 15
    for name, _, body in guarded:
        want = {"cta": "aborted_cta", "warp": "aborted_warp", "none": "aborted"}[_scope(body, functions)]
        assert f"if ({want}(guard)) return;" in body, name


@pytest.mark.gpu
@pytest.mark.parametrize("deg,num_l", [(300, 400_000), (5000, 400_000), (300, 524_288), (100, 30_000)])
def test_malformed_batch_of_several_waves(deg, num_l):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00283_gb300 import bfc
    rows = 4000 if deg < 1000 else 800
    b = G.union_batch([G.rows_of_degrees([deg] * rows, num_l, 3), G.rows_of_degrees([2, 5], 500, 4)])
    bad = b.union.adj_u.copy()
    bad[::deg * 7 + 11] = num_l + 7     # an L vertex of the second graph, in every seventh row or so
    bad[b.union.num_edges - 7:] = b.union.adj_u[b.union.num_edges - 7:]
    s = torch.cuda.current_stream().cuda_stream
    dev = [torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (b.union.off_u, b.u_start, b.l_start)]
    totals = []
    for adj in (b.union.adj_u, bad, b.union.adj_u):
        a = torch.from_numpy(adj).cuda()
        args = (b.union.num_u, b.union.num_l, b.union.num_edges, dev[0].data_ptr(), a.data_ptr(), 2, dev[1].data_ptr(),
                dev[2].data_ptr(), None, s)
        if adj is bad:
            with pytest.raises(bfc.BfcError) as e:
                bfc.bfc_prepare_batch(*args)
            assert e.value.status == 2
            continue
        h = bfc.bfc_prepare_batch(*args)
        tot = torch.full((2,), -1, dtype=torch.int64, device="cuda")
        bfc.bfc_count_batch(h, s, tot.data_ptr())
        bfc.bfc_sync(h, s)
        bfc.bfc_release(h)
        totals.append(tot.tolist())
    assert totals[0] == totals[1] and totals[0][0] > 0
