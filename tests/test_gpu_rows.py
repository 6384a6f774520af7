"""The passes over whole rows of the union graph, around the lengths where a
row goes to the block or to the whole warp, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from synth import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gcb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2308_14493_gb300 import gc

    return gc


def mod64(xs):
    return [int(x) % (1 << 64) for x in xs]


# hubs of 255 to 258 and 511 to 514 entries (rows by a warp, by a block), and
# of 3,000; the last graph has hubs next to each other at both ends of the ids
@pytest.mark.parametrize("n,hubs,degrees", [
    (1500, (3, 700, 1499), (255, 256, 257)),
    (1500, (3, 700, 1499), (258, 511, 512)),
    (1501, (0, 750, 1500), (513, 514, 1200)),
    (4099, (0, 1, 2, 3, 4, 4095, 4096, 4097, 4098), (3000,) * 9),
])
@pytest.mark.parametrize("independent", [False, True], ids=["sequential", "independent"])
def test_long_rows(gcb, n, hubs, degrees, independent):
    rng = np.random.default_rng(n + sum(degrees))
    keys = set(int(k) for k in gen.er_graph(n, 2 * n, 5))
    for h, d in zip(hubs, degrees):
        for v in rng.choice(n, d, replace=False):
            if int(v) != h:
                keys.add((min(h, int(v)) << 32) | max(h, int(v)))
    keys = np.array(sorted(keys), dtype=np.uint64)
    rp, col = gen.csr_from_keys(n, keys)
    batches = gen.batch_stream(n, keys, [n, n // 2, 400, 7], 0.5, 9, sequential=not independent)
    og = oracle.OracleGraph(rp, col)
    F0 = og.F
    if independent:
        want = [oracle.fdgc_step(rp, col, ins, dels, F0, 3)["F"] for ins, dels in batches]
    else:
        want = [og.apply(ins, dels)["F"] for ins, dels in batches]
    with gcb.Graph(n, rp, col) as g:
        assert g.counts() == mod64(F0)
        got = g.apply_many(batches, independent=independent)
        assert [list(map(int, x)) for x in got] == [mod64(x) for x in want]
        assert g.count_static() == mod64(F0 if independent else want[-1])
