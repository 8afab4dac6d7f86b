"""The first attempt on an edge, which takes both its vertices at once, where
attempts meet: vertices that share state words, rows that all name their
neighbours or one vertex, the smallest graphs, every layout, in the sweep (its
grain set, so that no graph is left to one SM; graphs of few entries a row take
the instance that visits a chunk twice) and on the chip.  The oracle's
checker decides; no reservation, stray or held, is left behind."""
import numpy as np
import pytest
import torch  # noqa: F401

import graphgen as gg
import oracle
from tests.conftest import cuda_ok
from tests.test_serial_walk_gpu import _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

GRAPHS = {
    "path2": lambda: gg.path(2), "path3": lambda: gg.path(3), "path17": lambda: gg.path(17), "path33": lambda: gg.path(33),
    "path100k": lambda: gg.path(100001), "star": lambda: gg.star(5000), "complete": lambda: gg.complete(130),
    "bipartite": lambda: gg.complete_bipartite(5, 3000), "grid": lambda: gg.grid(301, 333),
    "edges": lambda: gg.disjoint_edges(35), "rmat": lambda: gg.rmat(13, 8, seed=6),
    # rows of ids near the row and anywhere, unsorted, with loops and repeats, one-sided
    "near": lambda: _ragged(70001, [0, 1, 3, 9], 5), "near33": lambda: _ragged(33, [1, 4], 6),
    "near-long": lambda: _ragged(9001, [0, 1, 2, 150], 7),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("bits", [2, 8, 32])
def test_attempts_that_meet(name, bits):
    import paper_2507_04420_gb300 as skp
    g = GRAPHS[name]()
    d = g.to("cuda")
    with skp.Graph(d.offsets, d.nbrs) as h:
        for kw in ({}, {"grain": 128}, {"grain": 128, "symmetric": 1}, {"grain": 128, "unit_order": 2}):
            if "symmetric" in kw and name.startswith("near"):
                continue
            mate, _, count = h.skipper(pairs=True, status_bits=bits, **kw)
            k = int(count)
            v = oracle.check(g.offsets.numpy(), g.nbrs.numpy(), mate.cpu().numpy().view(np.uint32))
            assert v.flags == 0, (kw, v.as_dict())
            assert h.state_census() == {"acc": g.n - 2 * k, "rsvd": 0, "mchd": 2 * k, "other": 0}
