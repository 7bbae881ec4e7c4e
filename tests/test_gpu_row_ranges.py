"""Rows of 33 to 256 neighbours where the L ranks just fit the 24 bits of the register
sort's keys, and where they just do not (sorted in shared memory then)."""
import numpy as np
import pytest

import oracle
from bfc_inputs import generators as G

from gpu_path import run_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("validate", [1, 0])
@pytest.mark.parametrize("num_l", [1 << 24, (1 << 24) + 1])
def test_24_bit_ranks(num_l, validate):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00283_gb300 import bfc
    # the last L vertex is in every row, so it has the highest rank, and index d - 1
    rng = np.random.default_rng(24)
    pool = rng.choice(num_l - 1, 400, replace=False)
    degs = [33, 63, 64, 65, 127, 128, 129, 254, 255, 256, 256, 256]
    rows = [np.sort(np.append(rng.choice(pool, d - 1, replace=False), num_l - 1)) for d in degs]
    g = G.BipartiteCSR(len(degs), num_l, np.concatenate([[0], np.cumsum(degs)]).astype(np.int32),
                       np.concatenate(rows).astype(np.int32), "wide_ranks")
    ref = oracle.vp(g, vertices=True, edges=True)
    got = run_gpu(g, vertices=True, edges=True, export=True, options=bfc.bfc_options_init(validate=validate))
    assert got["rank_l"][num_l - 1] == num_l - 1
    assert got["total"] == got["total_all"] == ref["total"]
    for key in ("pv_u", "pv_l", "pe"):
        assert np.array_equal(got[key], ref[key])
    if validate:   # the sort still sees an edge that occurs twice
        twice = G.BipartiteCSR(g.num_u, num_l, g.off_u, g.adj_u.copy(), "twice")
        twice.adj_u[g.off_u[-2]] = num_l - 1
        with pytest.raises(bfc.BfcError) as e:
            run_gpu(twice)
        assert e.value.status == 2
