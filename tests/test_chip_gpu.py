"""The pass with its states in one SM's shared memory (small single graphs) at
the sizes where it can go wrong: groups of 32 rows that end early, windows of
more than 8192 entries, the largest graph it takes and the smallest it leaves
to the sweep, one-sided rows with loops and repeats, every layout.  The
oracle's checker decides; the states left behind are counted."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
from tests.conftest import cuda_ok
from tests.test_serial_walk_gpu import _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

LIMIT = 32768   # rows + entries


def _graphs():
    for n, ln in ((1, [0, 1]), (2, [1]), (31, [1, 3]), (32, [5, 0]), (33, [128, 1]), (97, [0, 127, 129]),
                  (40, [700, 300, 0]), (1000, [0, 1, 2, 30]), (20, [1600])):
        yield False, _ragged(n, ln, n)
    for g in (gg.path(2), gg.path(10922), gg.path(10923), gg.path(10924), gg.star(10000), gg.complete_bipartite(3, 4000),
              gg.complete(150), gg.grid(80, 82), gg.rmat(9, 16, seed=4), gg.disjoint_edges(33),
              gg.CSR(torch.zeros(41, dtype=torch.int64), torch.zeros(0, dtype=torch.int32))):
        yield True, g


@pytest.mark.parametrize("bits", [2, 8, 32])
def test_small_graphs(bits):
    import paper_2507_04420_gb300 as skp
    sizes = set()
    for symmetric, g in _graphs():
        off, nb = g.offsets.numpy(), g.nbrs.numpy()
        sizes.add(g.n + g.nnz <= LIMIT)
        d = g.to("cuda")
        with skp.Graph(d.offsets, d.nbrs) as h:
            for kw in ({}, {"symmetric": 1}, {"nosync": 1}):
                if "symmetric" in kw and not symmetric:
                    continue
                mate, pairs, count = h.skipper(pairs=True, status_bits=bits, **kw)
                h.sync()
                k = int(count)
                m, p = mate.cpu().numpy().view(np.uint32), pairs[:k].cpu().numpy().view(np.uint32)
                v = oracle.check(off, nb, m, p)
                assert v.flags == 0, (g.n, g.nnz, kw, v.as_dict())
                assert h.validate(mate, pairs[:k]).as_dict() == v.as_dict()
                if symmetric:
                    assert h.state_census() == {"acc": g.n - 2 * k, "rsvd": 0, "mchd": 2 * k, "other": 0}
                if g.n == 10001:
                    assert k == 1
                if g.n == 4003:
                    assert k == 3
    assert sizes == {True, False}


def test_an_id_out_of_range_is_reported():
    import paper_2507_04420_gb300 as skp
    off = torch.arange(41, dtype=torch.int64).cuda()
    nb = torch.full((40,), 40, dtype=torch.int32).cuda()
    with skp.Graph(off, nb, check=False) as h:
        with pytest.raises(skp.SkipperError) as e:
            h.skipper()
        assert e.value.status == "MM_ERR_BAD_GRAPH"
        nb.fill_(0)
        assert h.validate(h.skipper()).flags == 0
