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


def test_many_rows_too_long_for_a_warp():
    """2000 rows of 17,000 entries, which a second kernel reads in pieces, against 2000
    of 1900, which it does not (an entry took ten to twenty times as long where long rows
    were read one after the other)."""
    import paper_2507_04420_gb300 as skp
    n, multi, best = 2000, skp.Multi(), {}
    for length in (1900, 17000):
        off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * length
        nb = torch.randint(0, n, (n * length,), dtype=torch.int32, device="cuda")
        none = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        loops = int((nb.view(n, length) == torch.arange(n, dtype=torch.int32, device="cuda")[:, None]).sum())
        vb, eb = (torch.tensor([0, x], dtype=torch.int64, device="cuda") for x in (n, n * length))
        with skp.Graph(off, nb) as h, skp.Graph(off, nb, check=False, local_ids=True) as b:
            checks = (lambda: h.validate(none), lambda: b.validate_batched(vb, eb, none),
                      lambda: multi.validate([(off, nb, none)])[0])
            for k, check in enumerate(checks):
                assert check().n_uncovered == n * length - loops
                best[k, length] = _best(check)
    for k in range(3):
        assert best[k, 17000] / 17000 <= 1.5 * best[k, 1900] / 1900, best


@pytest.mark.parametrize("length", [2047, 2048, 2049, 2051, 8191, 8192, 8193, 8195, 16384, 16386, 24577])
def test_rows_at_the_edges_of_pieces(length):
    import paper_2507_04420_gb300 as skp
    n = 37
    off = torch.tensor([0] + [length + (i % 3) for i in range(n)], dtype=torch.int64).cumsum(0)
    nnz = int(off[-1])
    nb = torch.randint(0, n, (nnz,), dtype=torch.int32)
    rows = torch.repeat_interleave(torch.arange(n, dtype=torch.int32), off[1:] - off[:-1])
    mate = torch.full((n,), -1, dtype=torch.int32)
    mate[3], mate[20] = 20, 3           # rows of unmatched vertices with one neighbour covered
    open_ = (rows != nb) & (mate[rows.long()] < 0) & (mate[nb.long()] < 0)
    want = (int(open_.sum()), int(open_.nonzero()[0]))
    vb, eb = (torch.tensor([0, x], dtype=torch.int64, device="cuda") for x in (n, nnz))
    off, nb, mate = off.cuda(), nb.cuda(), mate.cuda()
    with skp.Graph(off, nb) as h, skp.Graph(off, nb, check=False, local_ids=True) as b:
        for _ in range(2):
            got = h.validate(mate), b.validate_batched(vb, eb, mate), skp.Multi().validate([(off, nb, mate)] * 3)[2]
            for v in got:
                assert (v.n_uncovered, v.first_uncovered, v.n_matched) == want + (2,)
