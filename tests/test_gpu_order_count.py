"""The count of product orders from their coordinates against the oracle's
count of the causal matrix, every N_k.  All values are integers: exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    from paper_1805_04463_gb300 import build
    build.build()
    import paper_1805_04463_gb300 as m
    return m


def _count(cs, kind, coords):
    import torch
    n = coords.shape[1]
    c = torch.from_numpy(np.ascontiguousarray(coords, dtype=np.int32)).cuda()
    hist = torch.full((cs.hist_len(n),), -5, dtype=torch.int64, device="cuda")
    ws = torch.full((cs.coords_abundance_workspace(kind, n),), 255, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        cs.coords_abundance(kind, n, c, hist, ws)
    assert cs.workspace_status(ws) == 0
    return hist.cpu().numpy()


def _order(v):
    return np.stack([np.arange(len(v)), np.asarray(v)])


# one band, its edges, one tile of the ranks and its edges, several words of the table's step
@pytest.mark.parametrize("kind", [0, 1, 5])
@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 64, 65, 255, 257, 1023, 1024, 1025, 2049, 3071, 3072, 3073, 4133, 8193, 9001])
def test_sprinkled(cs, oracle, kind, n):
    c = oracle.sprinkle(kind, n, 0x0D0 + n)
    want = oracle.interval_abundance(oracle.causal_matrix(kind, c))
    assert (_count(cs, kind, c) == want).all()


@pytest.mark.parametrize("n", [33, 1024, 2100])
@pytest.mark.parametrize("shape", ["chain", "antichain", "blocks", "clustered"])
def test_degenerate_orders(cs, oracle, shape, n):
    v = {"chain": np.arange(n), "antichain": np.arange(n)[::-1], "blocks": np.arange(n) ^ 31,
         "clustered": np.random.default_rng(n).permutation(n) + (2 ** 31 - 1 - n)}[shape]
    if shape == "blocks":
        v = np.argsort(np.argsort(v, kind="stable"))
    c = _order(v)
    want = oracle.interval_abundance(oracle.causal_matrix(0, c))
    assert (_count(cs, 0, c) == want).all()


@pytest.mark.parametrize("kind", [1, 5])
@pytest.mark.parametrize("grid", [1, 7, 60, 1000])
def test_equal_coordinates(cs, oracle, kind, grid):
    """Many elements equal in u, in v or in both (unrelated by the strict test), in time order."""
    rng = np.random.default_rng(grid)
    c = rng.integers(0, grid, (2, 2500))
    c[:, :5] = 2 ** 31 - 1
    c = c[:, np.argsort(c.sum(0), kind="stable")]
    want = oracle.interval_abundance(oracle.causal_matrix(kind, c.astype(np.int32)))
    assert (_count(cs, kind, c) == want).all()


def test_more_counts_than_shared_bins(cs):
    """n past the shared bins: a chain (every size once per start) and a random order against
    the tensor path."""
    import torch
    n = 60001
    got = _count(cs, 0, _order(np.arange(n)))
    assert (got == n - 1 - np.arange(n - 1)).all()
    buf = cs.allocate(0, n, path=cs.PATH_MMA4)
    cs.run(buf, 99, eps=(0.0,))
    auto = cs.allocate(0, n)
    assert auto.by_coords
    cs.run(auto, 99, eps=(0.0,))
    torch.cuda.synchronize()
    assert torch.equal(buf.hist, auto.hist) and torch.equal(buf.actions[:1], auto.actions[:1])
    assert torch.equal(buf.bits, auto.bits) and torch.equal(buf.coords, auto.coords)


@pytest.mark.parametrize("kind", [0, 1, 5])
@pytest.mark.parametrize("n", [1, 2, 700, 3001])
def test_evaluate_from_labels_in_any_time_order_position(cs, oracle, kind, n):
    c = oracle.sprinkle(kind, n, 5 + n)
    want = oracle.interval_abundance(oracle.causal_matrix(kind, c))
    for coords in (None, np.ascontiguousarray(c, dtype=np.int32)):
        h, a, br = cs.evaluate(kind, n, seed=5 + n, coords_host=coords, eps=(0.0, 0.1))
        assert (h == want).all() and br == oracle.action(2, n, want, 0.0)[1]
        assert abs(a[1] - oracle.action(2, n, want, 0.1)[0]) <= 1e-12 * max(1.0, abs(a[1]))


def test_other_kinds_are_refused(cs):
    import torch
    assert all(cs.coords_abundance_workspace(k, 500) == 0 for k in (2, 3, 4, 6))
    t = torch.zeros(1 << 16, dtype=torch.int64, device="cuda")
    with pytest.raises(cs.CsError) as e:
        cs.coords_abundance(2, 500, t, t, t)
    assert e.value.status == -5


@pytest.mark.parametrize("others", [True, False])
def test_batch_counts_product_orders_from_coordinates(cs, oracle, others):
    """AUTO batches at the edges of bands, chunks and table steps, with and without sets that need
    their causal matrix; replayed as a graph too."""
    import torch
    sets = [(k, n, 900 + 7 * n + k) for k in (0, 1, 5) for n in (2, 3, 63, 64, 65, 128, 129, 1000, 2049, 3073)]
    sets += [(1, 8192, 31), (0, 8191, 32), (5, 4097, 33)]
    if others:
        sets = [(2, 700, 1), (4, 333, 2)] + sets + [(3, 1025, 3), (0, 1, 4), (6, 100, 5)]
    b = cs.Batch(sets, n_eps=2)
    for _ in range(2):
        b.hist.fill_(-1)
        b.launch((0.0, 0.1))
    torch.cuda.synchronize()
    assert b.status() == 0
    for s, (kind, n, seed) in enumerate(sets):
        want = oracle.interval_abundance(oracle.causal_matrix(kind, oracle.sprinkle(kind, n, seed)))
        assert (b.set_hist(s).cpu().numpy() == want).all(), (kind, n)
        so, br = oracle.action(oracle.dim(kind), n, want, 0.1)
        assert int(b.brackets[s]) == br
        assert abs(float(b.actions[s, 1]) - so) <= 1e-12 * max(1.0, abs(so))
    ref = b.hist.clone()
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        with torch.cuda.graph(g, stream=st):
            b.launch((0.0, 0.1), stream=st)
    b.hist.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(b.hist, ref)


def test_server_counts_orders_whole_among_sliced_requests(cs):
    """AUTO server: product orders and other kinds together; each as alone."""
    import torch
    from paper_1805_04463_gb300 import serve
    reqs = [(0.0, (0, 2, 1, 3, 5, 4)[r % 6], 1030 + 517 * r, 60 + r) for r in range(14)]
    srv = serve.Server(tick_macs=2e9)
    for _ in range(2):
        stats, res = srv.run(reqs, realtime=False)
        assert stats["requests"] == len(reqs)
        for rid, (_, kind, n, seed) in enumerate(reqs):
            buf = cs.allocate(kind, n, path=3)
            cs.run(buf, seed, eps=serve.EPS)
            torch.cuda.synchronize()
            assert (res[rid][0] == buf.hist.cpu().numpy()).all(), rid
            assert np.allclose(res[rid][1], buf.actions.cpu().numpy()[:4], rtol=1e-12, atol=1e-12)
