"""Sizes at which the library changes its way of working: row tiers of the
projection, work queues, light starts (one window, packed and split tables,
team counters), segment lengths of the walk, the allocation-free count's classes,
groups of sparsified samples, and the batch check inside the row kernels.  Whole
numbers throughout, so every comparison is for equality.
"""
import numpy as np
import pytest

import oracle
from bfc_inputs import generators as G

from gpu_path import as_u64, run_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _opts(**kw):
    from paper_1812_00283_gb300 import bfc
    return bfc.bfc_options_init(**kw)


def _same_as_oracle(g, opts=None):
    ref = oracle.vp(g, vertices=True, edges=True)
    got = run_gpu(g, vertices=True, edges=True, options=opts)
    assert got["total"] == got["total_v"] == got["total_e"] == got["total_all"] == ref["total"]
    assert got["info"]["wedges"] == ref["wedges"]
    for key in ("pv_u", "all_pv_u"):
        assert np.array_equal(got[key], ref["pv_u"])
    for key in ("pv_l", "all_pv_l"):
        assert np.array_equal(got[key], ref["pv_l"])
    for key in ("pe", "all_pe"):
        assert np.array_equal(got[key], ref["pe"])
    return got


def _wider(g, num_u, num_l):
    """g with vertices that have no edges added to both layers."""
    off = np.concatenate([g.off_u, np.full(num_u - g.num_u, g.off_u[-1], dtype=np.int32)])
    return G.BipartiteCSR(num_u, num_l, off, g.adj_u, g.name + "_wider")


# degrees at both sides of every row tier and of the work queues' limits
EDGE_DEGREES = [1, 2, 7, 8, 9, 24, 25, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 300]


@pytest.mark.parametrize("num_l,long_rows,validate", [
    (300, [], 1), (5000, [4095, 4096, 4097, 4999], 1), (5000, [4095, 4096, 4097, 4999], 0),
    (524_288, [4096, 4097, 9000], 1), (524_289, [4096, 4097, 9000], 1)])
def test_row_tiers(num_l, long_rows, validate):
    g = G.shuffle_lists(G.rows_of_degrees(EDGE_DEGREES * 3 + long_rows * 2, num_l, 17), 5)
    _same_as_oracle(g, _opts(validate=validate))
    got = run_gpu(g, export=True, options=_opts(validate=validate))
    # every list ascending, and both sides' slots name the edge they stand for
    off, adj, eid, m = got["off"], got["adj"], got["eid"], g.num_edges
    rows = np.repeat(np.arange(off.size - 1), np.diff(off))
    same = rows[1:] == rows[:-1]
    assert np.all(adj[1:][same] > adj[:-1][same])
    u_of_edge = np.repeat(np.arange(g.num_u), np.diff(g.off_u))
    assert np.array_equal(np.sort(eid[:m]), np.arange(m)) and np.array_equal(np.sort(eid[m:]), np.arange(m))
    assert np.array_equal(adj[m:], got["rank_l"][g.adj_u[eid[m:]]])
    assert np.array_equal(adj[:m], num_l + got["rank_u"][u_of_edge[eid[:m]]])
    assert np.array_equal(rows[m:], num_l + got["rank_u"][u_of_edge[eid[m:]]])


@pytest.mark.parametrize("opts", [{}, dict(warp_max_work=0, hash_max_work=0), dict(wide_positions=1)])
def test_segment_lengths(opts):
    # middles whose lists have every length around the segments' and windows' limits
    lens = [1, 3, 8, 15, 16, 31, 32, 33, 47, 63, 64, 65, 95, 96, 97, 127, 128, 129, 255, 256, 257, 288, 511, 512, 513]
    _same_as_oracle(G.rows_of_degrees(lens * 30, 640, 23), _opts(**opts))


def _blocks():
    """Many little components: complete blocks (starts of 1 to about 60 wedges,
    on both sides of the one-window limit) and paths between them."""
    g = G.path(3)
    rng = np.random.default_rng(3)
    us, vs, nu, nl = [], [], 0, 0
    for a, b in rng.integers(1, 11, size=(900, 2)):
        us.append(np.repeat(np.arange(a), b) + nu)
        vs.append(np.tile(np.arange(b), a) + nl)
        nu, nl = nu + int(a), nl + int(b)
    g = G.from_edges(nu, nl, np.concatenate(us), np.concatenate(vs), "blocks")
    h = G.rows_of_degrees([1] * 40 + [2] * 40 + [40, 33, 32, 31] * 3, 60, 9)   # more than 32 middles, few wedges
    return G.disjoint_union(g, h)


@pytest.mark.parametrize("wider", [0, 70_000, 450_000])
def test_light_starts(wider):
    # without extra vertices the light starts' ends fit the team's counters;
    # with them they take tables
    for g in (_blocks(), G.chung_lu_bipartite(6000, 4000, 60_000, 2.1, 2.2, 31)):
        if wider:
            g = _wider(g, g.num_u + wider, g.num_l + wider)
        got = _same_as_oracle(g)
        assert got["info"]["warp_starts"] > 32
        _same_as_oracle(g, _opts(warp_max_work=20))


def test_keys_and_counts_beyond_one_word():
    # 2^24 ends and counts of 9 bits: keys and counts apart
    g = G.chung_lu_bipartite(5000, 400, 60_000, 2.3, 2.0, 12)
    g = _wider(g, (1 << 24) + 5, 500)
    ref = oracle.vp(g, vertices=True)
    got = run_gpu(g, vertices=True, options=_opts(team_max_work=0))
    assert got["total"] == got["total_v"] == ref["total"] and got["info"]["hash_starts"] > 0
    assert np.array_equal(got["pv_u"], ref["pv_u"]) and np.array_equal(got["pv_l"], ref["pv_l"])


def test_light_starts_in_a_batch():
    from paper_1812_00283_gb300 import bfc
    graphs = [G.complete_bipartite(a, b) for a in (1, 2, 5, 9) for b in (1, 3, 6, 8)] * 8
    graphs += [G.chung_lu_bipartite(3000, 2000, 20_000, 2.1, 2.2, s) for s in range(4)]
    b = G.union_batch(graphs)
    dev = [torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (b.union.off_u, b.union.adj_u, b.u_start, b.l_start)]
    s = torch.cuda.current_stream().cuda_stream
    want = [oracle.vp(g)["total"] for g in graphs]
    tot = torch.zeros(b.num_graphs, dtype=torch.int64, device="cuda")
    h = bfc.bfc_prepare_batch(b.union.num_u, b.union.num_l, b.union.num_edges, dev[0].data_ptr(), dev[1].data_ptr(),
                              b.num_graphs, dev[2].data_ptr(), dev[3].data_ptr(), None, s)
    bfc.bfc_count_batch(h, s, tot.data_ptr())
    bfc.bfc_sync(h, s)
    bfc.bfc_release(h)
    assert as_u64(tot).tolist() == want
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    plan = bfc.bfc_batch_plan_create(b.union.num_u, b.union.num_l, b.union.num_edges, b.num_graphs, 3000, None, s)
    tot.fill_(-1)
    bfc.bfc_batch_plan_run(plan, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), dev[3].data_ptr(), s,
                           tot.data_ptr(), status.data_ptr())
    torch.cuda.synchronize()
    bfc.bfc_batch_plan_destroy(plan)
    assert int(status.item()) == 0 and as_u64(tot).tolist() == want


@pytest.mark.parametrize("deg", [3, 20, 100, 400])
def test_edge_to_another_graph_in_every_row_tier(deg):
    from paper_1812_00283_gb300 import bfc
    graphs = [G.rows_of_degrees([deg] * 5, 500, 3), G.rows_of_degrees([2, 5], 500, 4)]
    b = G.union_batch(graphs)
    bad = b.union.adj_u.copy()
    bad[deg + 1] = 500 + 7        # row 1 of the first graph, an L vertex of the second
    s = torch.cuda.current_stream().cuda_stream
    off, us, ls = (torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (b.union.off_u, b.u_start, b.l_start))
    for validate in (1, 0):
        for adj, ok in ((bad, False), (b.union.adj_u, True)):
            adj = torch.from_numpy(adj).cuda()
            args = (b.union.num_u, b.union.num_l, b.union.num_edges, off.data_ptr(), adj.data_ptr(), 2, us.data_ptr(),
                    ls.data_ptr(), _opts(validate=validate), s)
            if ok:
                bfc.bfc_release(bfc.bfc_prepare_batch(*args))
            else:
                with pytest.raises(bfc.BfcError) as e:
                    bfc.bfc_prepare_batch(*args)
                assert e.value.status == 2


@pytest.mark.parametrize("case", ["largest", "hub", "ties", "high_class", "one_edge"])
def test_no_alloc_classes(case):
    from paper_1812_00283_gb300 import bfc
    g = {"largest": lambda: G.chung_lu_bipartite(49_152, 16_384, 300_000, 2.2, 2.0, 3),
         # lists above 512 and 1,024 entries, most of their middles of degree 1
         "hub": lambda: G.disjoint_union(G.rows_of_degrees([3000, 2999, 1500, 1025, 1024, 513, 512], 3000, 2), G.star(2000)),
         "ties": lambda: G.complete_bipartite(64, 64),
         # degrees of 254, 255, 256 and above
         "high_class": lambda: G.rows_of_degrees([254, 255, 256, 257, 700, 700, 254] * 20, 1024, 8),
         "one_edge": lambda: G.from_edges(1, 1, [0], [0])}[case]()
    off, adj = torch.from_numpy(g.off_u).cuda(), torch.from_numpy(g.adj_u).cuda()
    total = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    bfc.bfc_count_small_noalloc(g.num_u, g.num_l, g.num_edges, off.data_ptr(), adj.data_ptr(), s, total.data_ptr(),
                                status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(total.item()) == oracle.vp(g)["total"]


def test_sparsified_samples_in_two_groups():
    # the keep masks of 230 samples of 40M edges pass 2 GB: two groups
    from paper_1812_00283_gb300 import bfc
    gen = torch.Generator(device="cuda").manual_seed(4)
    keep = torch.rand((8000, 8000), device="cuda", generator=gen) < 0.625
    adj = keep.nonzero()[:, 1].int().contiguous()
    off = torch.zeros(8001, dtype=torch.int64, device="cuda")
    off[1:] = keep.sum(1).cumsum(0)
    off = off.int()
    m, samples, p = adj.numel(), 230, 0.002
    assert samples * (m // 32 + 1) * 8 > 1 << 31
    s = torch.cuda.current_stream().cuda_stream
    kept = torch.zeros(samples, dtype=torch.int64, device="cuda")
    tot = torch.zeros(samples, dtype=torch.int64, device="cuda")
    h = bfc.bfc_prepare_sparsified(8000, 8000, m, off.data_ptr(), adj.data_ptr(), p, 99, samples, None, s, kept.data_ptr())
    bfc.bfc_count_batch(h, s, tot.data_ptr())
    bfc.bfc_sync(h, s)
    bfc.bfc_release(h)
    g = G.BipartiteCSR(8000, 8000, off.cpu().numpy(), adj.cpu().numpy(), "dense_half")
    for j in (0, 1, 213, 214, 229):
        ref = oracle.sparsify(g, p, 99, j)
        assert int(kept[j]) == ref.num_edges and int(tot[j]) == oracle.vp(ref)["total"]


def test_unchecked_duplicate_edges_count_as_parallel_edges():
    # validate = 0 leaves duplicates to the caller: they are walked as parallel
    # edges in Definition 3's order, in rows of every tier
    from paper_1812_00283_gb300 import bfc
    rng = np.random.default_rng(5)
    rows = [np.sort(np.concatenate([rng.choice(340, d, replace=False), rng.integers(0, 340, k)]))
            for d, k in ((5, 2), (6, 1), (20, 3), (30, 2), (60, 4), (120, 5), (240, 9), (300, 20), (12, 0), (3, 1))]
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    adj = np.concatenate(rows).astype(np.int32)
    r, l, m = len(rows), 340, adj.size
    mult = np.zeros((r, l), dtype=np.int64)
    np.add.at(mult, (np.repeat(np.arange(r), np.diff(off)), adj), 1)
    deg = np.concatenate([mult.sum(0), mult.sum(1)])
    pri = np.lexsort((np.arange(r + l), deg)).argsort()
    full = np.zeros((r + l, r + l), dtype=np.int64)
    full[l:, :l], full[:l, l:] = mult, mult.T
    want = 0
    for x in range(r + l):
        lower = pri < pri[x]
        c = ((full[x] * lower) @ full) * lower
        want += int((c * (c - 1) // 2).sum())
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    s = torch.cuda.current_stream().cuda_stream
    h = bfc.bfc_prepare(r, l, m, o.data_ptr(), a.data_ptr(), _opts(validate=0), s)
    tot = torch.zeros(1, dtype=torch.int64, device="cuda")
    bfc.bfc_count(h, s, tot.data_ptr())
    bfc.bfc_sync(h, s)
    bfc.bfc_release(h)
    assert int(tot.item()) == want
    start = [torch.tensor(v, dtype=torch.int32, device="cuda") for v in ([0, r], [0, l])]
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    plan = bfc.bfc_batch_plan_create(r, l, m, 1, 400, _opts(validate=0), s)
    bfc.bfc_batch_plan_run(plan, o.data_ptr(), a.data_ptr(), start[0].data_ptr(), start[1].data_ptr(), s, tot.data_ptr(),
                           status.data_ptr())
    torch.cuda.synchronize()
    bfc.bfc_batch_plan_destroy(plan)
    assert int(status.item()) == 0 and int(tot.item()) == want
