"""validate = 0 with edges that occur more than once: they count as parallel edges.
A count of wedges is then a sum of products of multiplicities, which neither the
number of middles nor an end's degree bounds, and a degree can pass the size of
the other layer.  Against plain integer matrices of multiplicities.
"""
import numpy as np
import pytest

from gpu_path import as_u64

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _reference(mult):
    """Totals of the wedges' pairs from mult[u, v]: total, per vertex (L, then U) and
    per copy of each edge (u, v), by Definition 3's order."""
    r, l = mult.shape
    n = r + l
    full = np.zeros((n, n), dtype=np.int64)
    full[l:, :l], full[:l, l:] = mult, mult.T
    pri = np.lexsort((np.arange(n), full.sum(1))).argsort()
    total, pv, pe = 0, np.zeros(n, dtype=np.int64), np.zeros((n, n), dtype=np.int64)
    for x in range(n):
        mids = np.nonzero((full[x] > 0) & (pri < pri[x]))[0]
        ends = np.nonzero(pri < pri[x])[0]
        if not mids.size or not ends.size:
            continue
        sub = full[np.ix_(mids, ends)]
        c = full[x, mids] @ sub
        ends, sub, c = ends[c > 1], sub[:, c > 1], c[c > 1]
        pairs = c * (c - 1) // 2
        total += int(pairs.sum())
        pv[x] += pairs.sum()
        pv[ends] += pairs
        through = sub @ (c - 1)              # per copy of (x, middle)
        pv[mids] += full[x, mids] * through
        pe[x, mids] += through
        pe[np.ix_(mids, ends)] += full[x, mids][:, None] * (c - 1)[None, :] * (sub > 0)
    return total, pv[l:], pv[:l], (pe + pe.T)[l:, :l]


def _csr(mult, rng):
    rows = [rng.permutation(np.repeat(np.arange(mult.shape[1]), m)) for m in mult]
    off = np.concatenate([[0], np.cumsum([len(x) for x in rows])]).astype(np.int32)
    return off, np.concatenate(rows).astype(np.int32)


def _mult(case, rng):
    if case == "bundles":            # 8 copies each: one pair with 64 wedges
        m = np.zeros((2, 9), dtype=np.int64)
        m[:, 0] = 8
        m[1, 1:] = 1
    elif case == "triples":
        m = np.array([[3, 0, 0], [3, 2, 2]], dtype=np.int64)
    elif case == "past_the_layer":   # degrees far above both layers' sizes
        m = rng.integers(0, 60, (7, 5))
    elif case == "wide_counts":      # one pair with more wedges than 16 bits hold
        m = np.zeros((40, 60), dtype=np.int64)
        m[2:, :] = rng.random((38, 60)) < 0.2
        m[:, 0] = 0
        m[:2, 0] = 300
        m[1, 1:] = 6
    elif case == "light":            # many light starts of small multiplicity
        m = (rng.random((300, 250)) < 0.02) * rng.integers(1, 9, (300, 250))
    else:                            # starts of every size, rows of every tier below 4,096
        m = (rng.random((90, 300)) < rng.random((90, 1)) ** 2) * (1 + 11 * (rng.random((90, 300)) < 0.1))
        m[3] *= 7
    return m.astype(np.int64)


CASES = ["bundles", "triples", "past_the_layer", "wide_counts", "light", "mixed"]
OPTS = [{}, dict(warp_max_work=0), dict(warp_max_work=0, team_max_work=0), dict(warp_max_work=0, team_max_work=0, hash_max_work=0),
        dict(orientation=1), dict(orientation=1, warp_max_work=0, hash_max_work=0), dict(core_vertices=64), dict(wide_positions=1)]


@pytest.mark.parametrize("extra", [0, 70_000])
@pytest.mark.parametrize("case", CASES)
def test_parallel_edges(case, extra):
    # extra vertices without edges take the lowest ranks: ends' ranges then need tables and chunks
    from paper_1812_00283_gb300 import bfc
    rng = np.random.default_rng(CASES.index(case))
    mult = _mult(case, rng)
    total, pu, pl, pe = _reference(mult)
    off, adj = _csr(mult, rng)
    r, l, m = mult.shape[0] + extra, mult.shape[1] + extra, adj.size
    off = np.concatenate([off, np.full(extra, m, dtype=np.int32)])
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    want_pe = pe[np.repeat(np.arange(mult.shape[0]), mult.sum(1)), adj]
    s = torch.cuda.current_stream().cuda_stream

    def out(n):
        return torch.full((max(n, 1),), -1, dtype=torch.int64, device="cuda")

    for kw in OPTS:
        h = bfc.bfc_prepare(r, l, m, o.data_ptr(), a.data_ptr(), bfc.bfc_options_init(validate=0, **kw), s)
        t, vu, vl, e, t4 = out(1), out(r), out(l), out(m), out(4)
        bfc.bfc_count(h, s, t4[0:].data_ptr())
        bfc.bfc_count_vertices(h, s, vu.data_ptr(), vl.data_ptr(), t4[1:].data_ptr())
        assert np.array_equal(as_u64(vu)[:mult.shape[0]], pu) and np.array_equal(as_u64(vl)[:mult.shape[1]], pl), kw
        bfc.bfc_count_edges(h, s, e.data_ptr(), t4[2:].data_ptr())
        assert np.array_equal(as_u64(e), want_pe), kw
        vu.fill_(-1), vl.fill_(-1), e.fill_(-1)
        bfc.bfc_count_all(h, s, vu.data_ptr(), vl.data_ptr(), e.data_ptr(), t4[3:].data_ptr())
        bfc.bfc_sync(h, s)
        assert t4.tolist() == [total] * 4, kw
        assert not as_u64(vu)[mult.shape[0]:].any() and not as_u64(vl)[mult.shape[1]:].any()
        assert np.array_equal(as_u64(vu)[:mult.shape[0]], pu) and np.array_equal(as_u64(vl)[:mult.shape[1]], pl), kw
        assert np.array_equal(as_u64(e), want_pe), kw
        bfc.bfc_release(h)
        with pytest.raises(bfc.BfcError) as err:
            bfc.bfc_prepare(r, l, m, o.data_ptr(), a.data_ptr(), bfc.bfc_options_init(**kw), s)
        assert err.value.status == 2


@pytest.mark.parametrize("extra", [0, 45_000])
def test_parallel_edges_in_batches_and_plans(extra):
    # several multigraphs and a simple graph side by side; "wide_counts" stays out of
    # the plan, whose counters hold 16 bits
    from paper_1812_00283_gb300 import bfc
    rng = np.random.default_rng(77)
    s = torch.cuda.current_stream().cuda_stream
    for plan in (False, True):
        mults = [_mult(c, rng) for c in CASES if not (plan and c == "wide_counts")]
        mults.append((rng.random((50, 60)) < 0.3).astype(np.int64))
        want = [_reference(x)[0] for x in mults]
        off, adj, us, ls = [np.zeros(1, dtype=np.int32)], [], [0], [0]
        for x in mults:
            o, a = _csr(x, rng)
            adj.append(a + ls[-1])
            off.append(o[1:] + off[-1][-1])
            off.append(np.full(extra, off[-1][-1], dtype=np.int32))
            if not extra:
                off.pop()
            us.append(us[-1] + x.shape[0] + extra)
            ls.append(ls[-1] + x.shape[1] + extra)
        dev = [torch.from_numpy(np.concatenate(t).astype(np.int32)).cuda() for t in (off, adj)]
        dev += [torch.tensor(t, dtype=torch.int32, device="cuda") for t in (us, ls)]
        m, opts = dev[1].numel(), bfc.bfc_options_init(validate=0)
        tot = torch.full((len(mults),), -1, dtype=torch.int64, device="cuda")
        if plan:
            status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
            h = bfc.bfc_batch_plan_create(us[-1], ls[-1], m, len(mults), 50_000, opts, s)
            bfc.bfc_batch_plan_run(h, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), dev[3].data_ptr(), s,
                                   tot.data_ptr(), status.data_ptr())
            torch.cuda.synchronize()
            bfc.bfc_batch_plan_destroy(h)
            assert int(status.item()) == 0
        else:
            h = bfc.bfc_prepare_batch(us[-1], ls[-1], m, dev[0].data_ptr(), dev[1].data_ptr(), len(mults),
                                      dev[2].data_ptr(), dev[3].data_ptr(), opts, s)
            bfc.bfc_count_batch(h, s, tot.data_ptr())
            bfc.bfc_sync(h, s)
            bfc.bfc_release(h)
        assert tot.tolist() == want


def test_one_edge_many_times():
    # the first of a long group of equal edges is found by halving, not by walking back
    from paper_1812_00283_gb300 import bfc
    k = 400_000
    off = torch.tensor([0, k, 2 * k + 13], dtype=torch.int32, device="cuda")
    adj = torch.ones(2 * k + 13, dtype=torch.int32, device="cuda")
    adj[:k + 3] = 0                    # k and 3 copies to L vertex 0, k + 10 to L vertex 1
    assert int(off[-1]) == adj.numel()
    s = torch.cuda.current_stream().cuda_stream
    t = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    h = bfc.bfc_prepare(2, 2, adj.numel(), off.data_ptr(), adj.data_ptr(), bfc.bfc_options_init(validate=0), s)
    bfc.bfc_count(h, s, t.data_ptr())
    bfc.bfc_sync(h, s)
    bfc.bfc_release(h)
    c = 3 * k
    assert int(t.item()) == c * (c - 1) // 2


@pytest.mark.parametrize("extra", [0, 16_000, 32_000])
@pytest.mark.parametrize("case", CASES + ["two_pairs"])
def test_parallel_edges_without_allocation(case, extra):
    # "two_pairs": counts above 16 bits at neighbouring ranks and at 65,535 exactly;
    # extra vertices move the ends' ranks into the upper half of the 32-bit pass
    from paper_1812_00283_gb300 import bfc
    rng = np.random.default_rng(len(case))
    if case == "two_pairs":
        mult = np.zeros((4, 5), dtype=np.int64)
        mult[:, 0] = 255, 257, 258, 257
        mult[3, 1:] = 300
    else:
        mult = _mult(case, rng)
    total = _reference(mult)[0]
    off, adj = _csr(mult, rng)
    off = np.concatenate([off, np.full(extra, adj.size, dtype=np.int32)])
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    out = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for _ in range(2):
        bfc.bfc_count_small_noalloc(mult.shape[0] + extra, mult.shape[1] + extra, adj.size, o.data_ptr(), a.data_ptr(), s,
                                    out.data_ptr(), status.data_ptr())
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and int(out.item()) == total


def test_many_long_middles_without_allocation():
    # one start with 5,000 copies of edges to middles of more than 512 neighbours each:
    # more long lists in one start than a simple graph of this size can have
    from paper_1812_00283_gb300 import bfc
    mult = np.zeros((602, 4), dtype=np.int64)
    mult[:600, :3] = 1
    mult[600, :3] = 1700
    mult[601, 3] = 6000
    rng = np.random.default_rng(3)
    total = _reference(mult)[0]
    off, adj = _csr(mult, rng)
    o, a = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
    out = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    bfc.bfc_count_small_noalloc(602, 4, adj.size, o.data_ptr(), a.data_ptr(), torch.cuda.current_stream().cuda_stream,
                                out.data_ptr(), status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(out.item()) == total > 0
