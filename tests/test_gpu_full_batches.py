"""A start whose middles fill the walk's batches exactly, one short and one over: the
last group of segments then reaches past the last run of the batch.  A batch takes
2,048 middles of a CTA's start and 512 of a team's (half of that with 64-bit
positions)."""
import numpy as np
import pytest

import oracle
from bfc_inputs import generators as G

from gpu_path import run_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _hub(middles, run, seed):
    """One U vertex with all `middles` L vertices as neighbours, each of which has `run`
    neighbours of lower degree: as many runs of that length as middles."""
    rng = np.random.default_rng(seed)
    others = max(2 * run, 40, middles * run // 60)
    us = [np.zeros(middles, dtype=np.int64)] + [1 + rng.choice(others, run, replace=False) for _ in range(middles)]
    vs = [np.arange(middles), np.repeat(np.arange(middles), run)]
    return G.from_edges(1 + others, middles, np.concatenate(us), np.concatenate(vs))


@pytest.mark.parametrize("run", [1, 5, 30])
@pytest.mark.parametrize("batch", [256, 512, 1024, 2048])
def test_full_batches(batch, run):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00283_gb300 import bfc
    for middles in (batch - 1, batch, batch + 1):
        g = _hub(middles, run, middles + run)
        ref = oracle.vp(g, vertices=True, edges=True)
        for opts in (dict(), dict(wide_positions=1), dict(warp_max_work=0, team_max_work=0)):
            got = run_gpu(g, vertices=True, edges=True, options=bfc.bfc_options_init(**opts))
            assert got["total"] == got["total_v"] == got["total_e"] == got["total_all"] == ref["total"]
            for key in ("pv_u", "pv_l", "pe"):
                assert np.array_equal(got[key], ref[key]) and np.array_equal(got["all_" + key], ref[key])
