"""Checks of matchings that are wrong everywhere cost about what the check of a right
one costs: faults are counted warp by warp (added to the verdict group by group, they
took four times as long), in every form of the checker."""
import time

import pytest
import torch

import graphgen as gg
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def _best(f):
    best = 1e9
    for _ in range(7):
        t0 = time.perf_counter()
        f()
        best = min(best, time.perf_counter() - t0)
    return best


def test_faults_in_every_group():
    import paper_2507_04420_gb300 as skp
    n = 20_000_000
    g = gg.path(n, device="cuda")
    own = torch.arange(n, dtype=torch.int32, device="cuda")     # every vertex its own partner
    shifted = own.roll(1)                                       # no partner names its vertex
    multi = skp.Multi()
    vb, eb = (torch.tensor([0, x], dtype=torch.int64, device="cuda") for x in (n, g.nnz))
    with skp.Graph(g.offsets, g.nbrs) as h, skp.Graph(g.offsets, g.nbrs, check=False, local_ids=True) as b:
        right = h.skipper()
        for check in (h.validate, lambda m: b.validate_batched(vb, eb, m), lambda m: multi.validate([(g.offsets, g.nbrs, m)])[0]):
            assert check(right).flags == 0
            v = check(own)
            assert (v.n_bad_range, v.n_uncovered, v.first_bad_vertex) == (n, 0, 0)
            v = check(shifted)
            assert (v.n_asym, v.n_nonedge, v.first_bad_vertex) == (n, 1, 0)   # vertex 0 names the last one
            assert _best(lambda: check(own)) <= 2 * _best(lambda: check(right))
    src, dst = gg.edge_list(g, "row")
    with skp.EdgeList(n, src.cuda(), dst.cuda()) as h:
        assert h.validate(own).n_bad_range == n
        assert _best(lambda: h.validate(own)) <= 2 * _best(lambda: h.validate(right))
