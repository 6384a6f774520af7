"""Local counts of several handles at once: their scratch comes from one pool."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from synth import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rounds", [1, 3])
def test_handles_share_the_scratch_pool(rounds):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2308_14493_gb300 import gc

    graphs = []
    for n, m in ((3000, 20000), (500, 9000), (3000, 60000)):
        graphs.append((n, *gen.csr_from_keys(n, gen.er_graph(n, m, n + m))))
    want = []
    for n, rp, col in graphs:
        with gc.Graph(n, rp, col) as g:
            want.append((g.vertex_orbits(), *g.edge_orbits()))
    bad = []

    def work(k):
        for _ in range(rounds):
            n, rp, col = graphs[k % 3]
            with gc.Graph(n, rp, col) as g:
                for _ in range(3):
                    got = (g.vertex_orbits(), *g.edge_orbits())
                    if not all(np.array_equal(a, b) for a, b in zip(got, want[k % 3])):
                        bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
