"""The 4-cycle kernels that count pivots in shared memory, at the sizes where
their geometry changes, against the oracle (exact, as every count is)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import gen

pytestmark = pytest.mark.gpu

ALL_DENSE = dict(c4_reg_max=1, c4_warp_max=1, c4_block_max=1, c4_cta_max=1)
TABLES = dict(c4_reg_max=1, c4_warp_max=1, c4_block_max=8192, c4_cta_max=32768)


@pytest.fixture(scope="module")
def gcb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2308_14493_gb300 import gc

    return gc


def hub_graph(n, m, hub_degree, seed):
    """Sparse background plus three hubs that share most neighbours, at the
    lowest, middle and highest ids."""
    rng = np.random.default_rng(seed)
    keys = set(int(k) for k in gen.er_graph(n, m, seed))
    for h in (0, n // 2, n - 1):
        for v in rng.choice(n, hub_degree, replace=False):
            if int(v) != h:
                keys.add((min(h, int(v)) << 32) | max(h, int(v)))
    return np.array(sorted(keys), dtype=np.uint64)


# small and large block geometry (16,384 / 16,385 ids), 16-bit counters by the
# number of ids alone or by the degrees (65,536 / 65,537), several chunks of
# 4-, 8- and 16-bit counters (300,001)
@pytest.mark.parametrize("n,hub", [(5, 2), (16384, 3000), (16385, 3000), (65536, 9000), (65537, 300), (300001, 12000)])
@pytest.mark.parametrize("tuning", [ALL_DENSE, TABLES], ids=["chunks", "tables"])
def test_pivots_at_the_edges_of_the_geometry(gcb, n, hub, tuning):
    keys = hub_graph(n, min(3 * n, n * (n - 1) // 4), hub, n)
    rp, col = gen.csr_from_keys(n, keys)
    F0 = oracle.static_counts(rp, col)
    ins, dels = gen.random_batch(n, keys, min(200, n // 3), min(200, n // 3), 3)
    r = oracle.fdgc_step(rp, col, ins, dels, F0)
    with gcb.Graph(n, rp, col) as g:
        assert g.counts() == F0
        g.set_tuning(**tuning)
        assert g.count_static() == F0
        assert g.count_batch(ins, dels) == r["F"]
        assert g.apply(ins, dels) == r["F"]
        assert g.count_static() == r["F"]


def test_more_one_graph_wedges_than_a_block_lists(gcb):
    """A batch that changes most of a dense graph: single pivots have tens of
    thousands of wedges in one graph only, more than the 16,384 a block
    lists, and walk them again."""
    n = 500
    keys = gen.er_graph(n, 50000, 7)
    rp, col = gen.csr_from_keys(n, keys)
    F0 = oracle.static_counts(rp, col)
    ins, dels = gen.random_batch(n, keys, 20000, 20000, 8, ins_weighting="uniform")
    r = oracle.fdgc_step(rp, col, ins, dels, F0)
    with gcb.Graph(n, rp, col) as g:
        g.set_tuning(**ALL_DENSE)
        assert g.count_batch(ins, dels) == r["F"]
        assert g.apply(ins, dels) == r["F"]
        assert [x % 2**64 for x in g.stats()["Ca"]] == [x % 2**64 for x in r["Ca"]]
        assert [x % 2**64 for x in g.stats()["Cb"]] == [x % 2**64 for x in r["Cb"]]


@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_full_tables(gcb, extra):
    """A pivot whose wedges end at distinct ids, as many as the large table
    takes (w~ = 19,456) and one more or less: K_{2,..}-free stars chained to
    one pivot.  The pivot's only 4-cycles come from one shared endpoint."""
    arms, per = 128, 152  # w~ = 128 x 152 = 19,456
    edges, nxt = [], arms + 1
    for a in range(1, arms + 1):
        edges.append((0, a))
        k = per - 1 + (extra if a == 1 else 0)  # the arm's degree counts its edge to the pivot
        for _ in range(k):
            edges.append((a, nxt))
            nxt += 1
    edges.append((2, nxt - 1))  # a second path from the pivot to the last arm's last leaf
    n = nxt
    keys = np.array(sorted((min(a, b) << 32) | max(a, b) for a, b in edges), dtype=np.uint64)
    rp, col = gen.csr_from_keys(n, keys)
    with gcb.Graph(n, rp, col) as g:
        g.set_tuning(**TABLES)
        assert g.count_static() == oracle.static_counts(rp, col)


def test_repeated_static_counts(gcb):
    """Static counts of a small graph replay a captured sequence from the
    third on: between batches that move buffers, tuning changes and new
    vertices every count is that of the graph as it is then."""
    n = 3000
    keys = hub_graph(n, 6000, 500, 12)
    rp, col = gen.csr_from_keys(n, keys)
    og = oracle.OracleGraph(rp, col)
    with gcb.Graph(n, rp, col) as g:
        for i, size in enumerate((0, 50, 4000, 10, 0, 0)):
            if size:
                grp, gcol = g.export_csr()
                ins, dels = gen.random_batch(g.n, gen.keys_from_csr(grp, gcol), size, size // 2, 100 + i)
                assert g.apply(ins, dels) == og.apply(ins, dels)["F"]
            if i == 4:
                g.set_tuning(**ALL_DENSE)
            if i == 5:
                g.add_vertices(20000)
            for _ in range(5):
                assert g.count_static() == og.F
            assert g.counts() == og.F


@pytest.mark.parametrize("mid_degree,hub_degree", [(63, 5000), (64, 2048), (70, 3000), (150, 5000)])
def test_local_pairs_between_mid_vertices_under_hubs(gcb, mid_degree, hub_degree):
    """Edge-local 4-cycles where the staged rows have about 64 entries (the
    shortest staged) and the walked rows are hubs on both sides of 32 times
    their length (walked, or searched)."""
    n, mids = 8000, 60
    rng = np.random.default_rng(mid_degree + hub_degree)
    keys = set(int(k) for k in gen.er_graph(n, 4000, 5))
    for h in (0, 1):
        for v in rng.choice(np.arange(2, n), hub_degree, replace=False):
            keys.add((h << 32) | int(v))
    for u in range(2, 2 + mids):
        keys.add(u)  # (0, u): every mid vertex hangs on the first hub
        for v in rng.choice(np.arange(100, n), mid_degree, replace=False):
            keys.add((u << 32) | int(v))
    keys = np.array(sorted(keys), dtype=np.uint64)
    rp, col = gen.csr_from_keys(n, keys)
    F0 = oracle.static_counts(rp, col)
    have = set(int(k) for k in keys)
    pairs = [(a, b) for a in range(2, 2 + mids) for b in range(a + 1, 2 + mids)]
    rng.shuffle(pairs)
    ins = np.array([p for p in pairs if ((p[0] << 32) | p[1]) not in have][:200], np.int32)
    dels = gen.random_batch(n, keys, 0, 150, 9)[1]
    r = oracle.fdgc_step(rp, col, ins, dels, F0)
    with gcb.Graph(n, rp, col, local_max_pairs=100000) as g:
        assert g.apply(ins, dels) == r["F"]
        assert g.stats()["path"] == 1
        assert g.apply(dels, ins) == F0


# a plan with one thread per granule of ids: around the number of ids that
# fills its threads (512 granules of 64)
@pytest.mark.parametrize("n", [32767, 32768, 32769, 33279, 33280])
def test_pivot_plans_cover_every_id(gcb, n):
    keys = hub_graph(n, 2 * n, 4000, n)
    rp, col = gen.csr_from_keys(n, keys)
    with gcb.Graph(n, rp, col) as g:
        g.set_tuning(**ALL_DENSE)
        assert g.count_static() == oracle.static_counts(rp, col)
