"""The search that ranks a prefix of each query's centroid order first and
extends it where the stop line passes it, against the same search on a given
full order: probes, counts and ids must be the same, scores within 1e-5.

Low thresholds make most probes hit, so stop lines run far past the prefix
(16 or 32 entries less the margin); identical centroids leave no verified
prefix at all.  A search takes a prefix only at a tight threshold, so a low one
is reached by longer vectors: rows and queries times a turn a threshold of tau
into tau a^2 (``_stretch``), with the same hits."""
import numpy as np
import pytest
import torch

from parity import assert_parity, compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda:0")


def _stretch(tau, at=0.9):
    """The factor with which rows and queries meet the threshold `at` where the
    unit ones meet tau."""
    return (at / tau) ** 0.5


def _index(sieve, dev, n, d, nlist, seed, grouped=False, equal=0, tau=0.9):
    g = torch.Generator().manual_seed(seed)
    unit = lambda x: x / x.norm(dim=1, keepdim=True)
    C = unit(torch.randn(nlist, d, generator=g))
    if grouped:   # neighbours with adjacent ids
        base = unit(torch.randn(-(-nlist // 32), d, generator=g)).repeat_interleave(32, 0)[:nlist]
        C = unit(base + 0.3 * C)
    if equal:     # blocks of identical centroids: exact ties
        C = C[torch.arange(nlist) // equal * equal].contiguous()
    a = torch.randint(0, nlist, (n,), generator=g)
    X = unit(C[a] + 0.9 * torch.randn(n, d, generator=g) / d ** 0.5) * _stretch(tau)
    ix = sieve.build_layout(X.to(dev), a.int().to(dev), nlist, C.to(dev))
    ix.assign = a.int()
    return ix, X


# Edges of the dispatch (512 centroids and 4,096 queries, 1,024 for the longer
# lists, 2,049 for a few queries), of the tiles (128 and 256 queries), of the
# groups and chunks of centroids (32, 128, 192), of d (16, 64, 128, 256, 512).
# Lists are of 16 groups up to W = 10, below 256 and from 8,192 queries, else 32.
CASES = [  # n, d, nlist, nq, nprobe, W, tau, lookahead, grouped, equal
    (6_000, 64, 512, 4_100, 45, 4, 0.30, True, False, 0),
    (6_000, 64, 513, 9_000, 64, 8, 0.55, False, False, 0),
    (9_000, 96, 700, 5_000, 90, 8, 0.35, True, True, 0),
    (9_000, 128, 1_025, 4_613, 63, 10, 0.30, True, False, 0),
    (9_000, 256, 1_100, 4_100, 100, 24, 0.50, True, False, 0),
    (12_000, 36, 2_500, 300, 77, 2, 0.60, True, False, 0),
    (12_000, 200, 2_049, 130, 128, 8, 0.45, True, True, 0),
    (5_000, 32, 600, 8_200, 40, 8, 0.50, True, False, 8),
    (5_000, 96, 1_152, 4_100, 50, 16, 0.50, True, False, 128),
    (40_000, 96, 5_000, 600, 64, 8, 0.45, True, True, 0),
    (40_000, 96, 1_024, 40_000, 64, 8, 0.60, True, True, 0),   # several tiles per block
    (20_000, 256, 1_024, 20_000, 40, 8, 0.70, True, False, 0),
    (20_000, 512, 3_000, 1_000, 90, 8, 0.45, True, False, 0),   # past the layout's width
    (12_000, 260, 2_100, 300, 64, 16, 0.45, True, True, 0),
    (12_000, 448, 2_100, 129, 64, 8, 0.50, False, False, 0),
    (12_000, 512, 2_049, 1, 64, 8, 0.05, True, False, 0),
    (9_000, 96, 2_049, 1, 64, 8, 0.20, True, False, 0),
    (9_000, 4, 2_081, 127, 40, 4, 0.97, True, False, 0),
    (9_000, 100, 2_176, 129, 64, 8, 0.45, True, False, 0),
    (9_000, 132, 2_305, 257, 64, 8, 0.45, True, False, 0),
    (12_000, 64, 2_500, 9_001, 64, 8, 0.20, True, False, 0),   # nearly every query extended: two parts
    (12_000, 32, 2_100, 262_145, 40, 8, 0.20, True, False, 0),  # and all three
    (8_000, 96, 2_309, 5_000, 64, 16, 0.45, True, True, 0),    # a last group of five centroids
]


@pytest.mark.parametrize("n,d,nlist,nq,nprobe,W,tau,lookahead,grouped,equal", CASES)
def test_prefix_equals_full_order(dev, n, d, nlist, nq, nprobe, W, tau, lookahead, grouped, equal):
    """A query may differ only where the oracle's tags put one of its decisions
    (two centroid scores, two results, a result and tau) within 1e-5 of a flip."""
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, n, d, nlist, seed=n + d + nlist, grouped=grouped, equal=equal, tau=tau)
    g = torch.Generator().manual_seed(3)
    rows = torch.randint(0, n, (nq,), generator=g) if nq > n else torch.randperm(n, generator=g)[:nq]
    Q, qids = X[rows].to(dev), rows.to(dev)
    order = sieve.rank_partitions(ix, Q, nprobe)
    kw = dict(lookahead=lookahead, query_ids=qids, stats=True)
    as_dict = lambda out: dict(zip(("ids", "scores", "count", "probes"), (x.cpu().numpy() for x in out[:4])))
    want = sieve.search(ix, Q, 0.9, 10, nprobe, W, order=order, **kw)
    host = dict(X=X.numpy(), ids=np.arange(n), assign=ix.assign.numpy(), centroids=ix.centroids.cpu().numpy())
    for loop in (0, 1):
        got = sieve.search(ix, Q, 0.9, 10, nprobe, W, loop=loop, **kw)
        # the prefix ran, and whoever goes past it (it has 32 ranks at most) was extended
        assert want[4]["extended"] == -1
        assert got[4]["extended"] >= max(int((want[3] > 32).sum()), 1 if tau < 0.35 else 0)
        rep = compare(as_dict(got), as_dict(want), host, X[rows].numpy(), rows.numpy(), 0.9, 10, nprobe,
                      order.cpu().numpy())
        assert_parity(rep)
        # no partition visited twice: no result id repeats
        for r in got[0].cpu().numpy()[got[2].cpu().numpy() > 1][:2000]:
            r = r[r >= 0]
            assert len(set(r.tolist())) == len(r)


@pytest.mark.parametrize("nlist,nq,W,d,prefix", [
    (511, 4_096, 8, 32, False), (512, 4_096, 8, 32, True), (1_023, 4_096, 16, 32, False), (1_024, 4_096, 16, 32, True),
    (2_048, 4_095, 8, 32, False), (2_049, 1, 8, 32, True), (2_049, 1, 25, 32, False), (2_049, 1, 8, 512, True),
    (2_049, 1, 8, 516, False)])
def test_which_ranking_runs(dev, nlist, nq, W, d, prefix):
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 5_000, d, nlist, seed=1)
    Q = X[:nq].to(dev)
    got = sieve.search(ix, Q, 0.9, 10, 32, W, stats=True)
    assert (got[4]["extended"] >= 0) == prefix
    want = sieve.search(ix, Q, 0.9, 10, 32, W, order=sieve.rank_partitions(ix, Q, 32), stats=True)
    assert got[4]["status"] == want[4]["status"] == 0
    assert torch.equal(got[3], want[3]) and torch.equal(got[2], want[2])


@pytest.mark.parametrize("d", [96, 320])
def test_prefix_host_path(dev, d):
    """Each upload chunk's prefix, with the largest norm and the wide rows'
    layout made once for all of them."""
    import ctypes
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 30_000, d, 600, seed=9, tau=0.2)
    nq = 25_000                          # two upload chunks
    Q = X[:nq].contiguous().pin_memory()
    ids = torch.arange(nq).pin_memory()
    a = sieve.search(ix, Q.to(dev), 0.9, 10, 100, 8, query_ids=ids.to(dev), stats=True)
    b = sieve.search_host(ix, Q, 0.9, 10, 100, 8, query_ids_host=ids)
    for x, y in zip(a, b):
        assert torch.equal(x.cpu(), y)
    v, p, st = ix.view(), sieve._params(0.9, 10, 100, 8, True, 0, 0), sieve.StatsC()
    ws = torch.empty(sieve.workspace_size(ix, nq, 0.9, 10, 100, 8, host_io=True), dtype=torch.uint8, device=dev)
    out = [torch.empty_like(y) for y in b]
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = sieve.lib().sieve_search_host(ctypes.byref(v), ptr(Q), nq, ptr(ids), ctypes.byref(p), *map(ptr, out),
                                       ctypes.byref(st), ptr(ws), ws.numel(), None)
    assert rc == 0
    for x, y in zip(out, b):
        assert torch.equal(x, y)
    host = dict(zip(sieve.KERNELS, st.kernel_launches))
    device = a[4]["kernel_launches"]
    # a second scan and a second final, and nothing else, for the second chunk
    assert host["rank"] == device["rank"] + 2 and host["rank_mma"] == device["rank_mma"] + 1
    assert st.extended == a[4]["extended"] > 0


@pytest.mark.parametrize("d", [96, 320])
@pytest.mark.parametrize("odd", ["nan centroid", "long centroid", "infinite centroid", "long centroids",
                                 "nan query", "infinite query", "long query", "zero query"])
def test_rows_that_cannot_be_screened_are_ranked_as_by_the_full_order(dev, d, odd):
    """NaN, infinities and norms from 200 up leave the prefix empty: of every
    query where a centroid has them, of the query alone where a query does."""
    import paper_2608_03199_gb300 as sieve
    nlist, nq = 2_100, 700
    ix, X = _index(sieve, dev, 10_000, d, nlist, seed=4, tau=0.5)
    ix = sieve.build_layout(ix.vectors, torch.repeat_interleave(
        torch.arange(nlist, device=dev), ix.list_offsets.diff()).int(), nlist, ix.centroids.clone())
    C, Q = ix.centroids, X[:nq].to(dev)
    if odd == "nan centroid":
        C[17, 3] = float("nan")
    elif odd == "long centroid":
        C[17] *= 210.
    elif odd == "infinite centroid":
        C[2_099, 0] = float("inf")
    elif odd == "long centroids":
        C *= 300.
    elif odd == "nan query":
        Q[5, 7] = float("nan")
    elif odd == "infinite query":
        Q[699, 0] = -float("inf")
    elif odd == "long query":
        Q[5] *= 250.
    else:
        Q[5] = 0.
    if ix.tc_centroids is not None:
        ix = sieve.add_tc_layout(ix)
    qids = torch.full((nq,), -1, dtype=torch.int64, device=dev)
    order = sieve.rank_partitions(ix, Q, 64)
    want = sieve.search(ix, Q, 0.9, 10, 64, 8, query_ids=qids, order=order, check=True)
    got = sieve.search(ix, Q, 0.9, 10, 64, 8, query_ids=qids, stats=True)
    if "centroid" in odd:
        assert got[4]["extended"] == nq
    else:
        assert 1 <= got[4]["extended"] <= nq
    for x, y in zip(got[:4], want):
        assert torch.equal(x, y)


class _Fixed:
    """A workspace of a given size, whatever a call asks for."""

    def __init__(self, nbytes, device):
        self.buf = torch.empty(nbytes, dtype=torch.uint8, device=device)

    def get(self, nbytes, device):
        return self.buf


@pytest.mark.parametrize("call", ["search", "host", "sharded", "calibrated"])
def test_workspace_without_room_for_the_lists(dev, call):
    """A workspace of the full ranking's size (what the same index without the
    centroids' layout asks for) is taken, and the orders are ranked whole; half
    of it is refused, as ever."""
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 12_000, 96, 2_309, seed=6)
    nq, k, nprobe, W = 2_000, 10, 64, 8
    Q, qids = X[:nq].contiguous(), torch.arange(nq)
    Qd, qd = Q.to(dev), qids.to(dev)
    sample = torch.arange(0, nq, 10, device=dev)
    asked = []

    class Asks(sieve.Workspace):
        def get(self, nbytes, device):
            asked.append(nbytes)
            return super().get(nbytes, device)

    def run(index, ws):
        if call == "search":
            return sieve.search(index, Qd, 0.9, k, nprobe, W, query_ids=qd, workspace=ws, check=True)
        if call == "host":
            return sieve.search_host(index, Q.pin_memory(), 0.9, k, nprobe, W,
                                     query_ids_host=qids.pin_memory(), workspace=ws)
        if call == "sharded":
            return sieve.sharded_search([index], Qd, 0.9, k, nprobe, W, query_ids=qd, workspace=ws)
        return sieve.calibrated_search(index, Qd, 0.9, k, nprobe, sample, 0.1, min_queries=1,
                                       query_ids=qd, workspace=ws)[:4]

    want = [x.cpu() for x in run(ix, Asks())]
    bare = sieve.Index(ix.vectors, ix.ids, ix.list_offsets, ix.centroids, ix.tc_rows, ix.tc_row_blocks, None)
    bare.view = lambda v=bare.without_tc_layout().view(): v
    run(bare, Asks())
    full, least = asked
    assert least < full
    got = [x.cpu() for x in run(ix, _Fixed(least, dev))]
    for x, y in zip(got, want):
        # near-ties of centroids and of the two scan paths' sums apart
        same = (x == y) if x.dtype != torch.float32 else ((x - y).abs() <= 1e-5) | (x == y)
        assert (~same).reshape(nq, -1).any(1).sum() <= 2
    with pytest.raises(sieve.SieveError) as e:
        run(ix, _Fixed(least // 2, dev))
    assert e.value.status == -3


@pytest.mark.parametrize("nq", [200, 9_001])
def test_stats_tell_which_ranking_ran(dev, nq):
    """extended: -1 where every order is ranked whole or given, else the queries
    ranked whole after their prefix, whose launches count as the ranking's."""
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 12_000, 64, 2_500, seed=2, tau=0.2)
    Q, qids = X[:nq].to(dev), torch.arange(nq, device=dev)
    run = lambda tau, W, **kw: sieve.search(ix, Q, tau, 10, 64, W, query_ids=qids, stats=True, **kw)[4]
    assert run(0.9, 8, order=sieve.rank_partitions(ix, Q, 64))["extended"] == -1
    assert run(0.9, 64)["extended"] == -1
    assert run(0.9, 8, scan_path="simt")["extended"] == -1
    none = run(0.999 * _stretch(0.2) ** 2, 8)
    assert none["extended"] == 0
    assert none["kernel_launches"]["rank"] == 3 and none["kernel_launches"]["rank_mma"] == 1
    for loop in (0, 1):
        some = run(0.9, 8, loop=loop)
        assert nq // 2 < some["extended"] <= nq
        # a part of an extension is a gather, a full ranking and a merge
        assert some["kernel_launches"]["rank"] >= 3 + 8 and some["kernel_launches"]["rank_mma"] >= 1 + 2
    prof = sieve.search(ix, Q, 0.9, 10, 64, 8, query_ids=qids, profile=True)[4]
    assert prof["kernel_launches"]["rank_mma"] == some["kernel_launches"]["rank_mma"]
    assert prof["kernel_ms"]["rank"] > prof["kernel_ms"]["rank_mma"] > 0


@pytest.mark.parametrize("lookahead", [True, False])
@pytest.mark.parametrize("nq,d,nlist,W", [(300, 64, 2_500, 8), (9_001, 96, 2_309, 8), (1_000, 128, 2_100, 16)])
def test_an_extension_takes_no_round_of_its_own(dev, lookahead, nq, d, nlist, W):
    """A query is listed in the round that raises its stop line, so the rounds
    are those of the same search on the whole order."""
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 12_000, d, nlist, seed=8, tau=0.3)
    Q, qids = X[:nq].to(dev), torch.arange(nq, device=dev)
    kw = dict(lookahead=lookahead, query_ids=qids, stats=True)
    want = sieve.search(ix, Q, 0.9, 10, 64, W, order=sieve.rank_partitions(ix, Q, 64), **kw)
    for loop in (0, 1):
        got = sieve.search(ix, Q, 0.9, 10, 64, W, loop=loop, **kw)
        assert got[4]["extended"] > 0
        assert got[4]["rounds"] == want[4]["rounds"]
        assert got[4]["items"] == want[4]["items"]
        # rounds cut short by a cap defer queries, listed ones among them
        cut = sieve.search(ix, Q, 0.9, 10, 64, W, loop=loop, max_items_per_round=nq + 7, **kw)
        for x, y in zip(cut[:4], got[:4]):
            assert torch.equal(x, y)


@pytest.mark.parametrize("nq,tau,prefix", [(1_000, 0.85, True), (1_000, 0.84, False), (16_383, 0.84, False),
                                           (16_384, 0.70, True), (16_384, 0.69, False)])
def test_a_loose_threshold_ranks_whole(dev, nq, tau, prefix):
    """Below the threshold lines every order is ranked whole at once."""
    import paper_2608_03199_gb300 as sieve
    ix, X = _index(sieve, dev, 20_000, 32, 2_100, seed=12)
    Q = X[:nq].to(dev)
    order = sieve.rank_partitions(ix, Q, 32)
    want = sieve.search(ix, Q, tau, 10, 32, 8, order=order)
    got = sieve.search(ix, Q, tau, 10, 32, 8, stats=True)
    assert (got[4]["extended"] >= 0) == prefix
    if not prefix:
        for x, y in zip(got[:4], want):
            assert torch.equal(x, y)


def test_several_passes_of_one_batch(dev):
    """400,000 queries at W = 16 need more than the 1 GiB of lists: two passes,
    the second from a whole number of waves of tiles on."""
    import paper_2608_03199_gb300 as sieve
    nq, nprobe, W = 400_000, 32, 16
    ix, X = _index(sieve, dev, 20_000, 32, 2_100, seed=14)
    rows = torch.randint(0, 20_000, (nq,), generator=torch.Generator().manual_seed(15))
    Q, qids = X[rows].to(dev), rows.to(dev)
    order = sieve.rank_partitions(ix, Q, nprobe)
    kw = dict(query_ids=qids, stats=True)
    want = sieve.search(ix, Q, 0.9, 10, nprobe, W, order=order, **kw)
    got = sieve.search(ix, Q, 0.9, 10, nprobe, W, **kw)
    st = got[4]
    assert st["extended"] >= 0 and st["kernel_launches"]["rank_mma"] - 2 * (st["extended"] > 0) >= 2
    bad = (got[3] != want[3]) | (got[2] != want[2]) | (got[0] != want[0]).any(1)
    as_dict = lambda out: {k: x[bad].cpu().numpy() for k, x in zip(("ids", "scores", "count", "probes"), out)}
    host = dict(X=X.numpy(), ids=np.arange(20_000), assign=ix.assign.numpy(), centroids=ix.centroids.cpu().numpy())
    at = bad.nonzero()[:, 0].cpu().numpy()
    print(f"{len(at)} of {nq} queries differ")
    assert len(at) <= nq // 1000
    if len(at):
        rep = compare(as_dict(got), as_dict(want), host, Q[bad].cpu().numpy(), rows.numpy()[at], 0.9, 10, nprobe,
                      order[bad].cpu().numpy())
        assert len(rep["unexplained"]) == 0
