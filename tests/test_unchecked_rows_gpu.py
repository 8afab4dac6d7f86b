"""Graphs whose row ends were never checked: ends before the first entry, past
the last one or out of order read as if they were clamped to the entries, in the
checker's three forms and in serial mode.  The entries lie in a larger buffer
whose other words name a vertex, so that a read outside them would show."""
import numpy as np
import pytest
import torch

import oracle
from tests.conftest import cuda_ok
from tests.test_checker_walk_gpu import NONE, _mate, _spoiled
from tests.test_serial_walk_gpu import _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

PAD, TAIL = 16, 512


def _inside(nbrs):
    """The entries as a 16-byte aligned slice of a device buffer of other ids."""
    full = torch.full((PAD + nbrs.size + TAIL,), 1, dtype=torch.int32, device="cuda")
    full[PAD:PAD + nbrs.size] = torch.from_numpy(nbrs.view(np.int32)).cuda()
    return full[PAD:PAD + nbrs.size]


def _verdict(ends, nbrs, mate):
    """The oracle's verdict on the rows nbrs[ends[v]:ends[v + 1]], which may overlap or be empty."""
    at = [np.arange(s, max(s, e)) for s, e in zip(ends[:-1], ends[1:])]
    off = np.concatenate([[0], np.cumsum([a.size for a in at])])
    at = np.concatenate(at)
    v = oracle.check(off, nbrs[at], mate).as_dict()
    x, y = np.repeat(np.arange(off.size - 1), np.diff(off)), nbrs[at]
    unc = at[(x != y) & (mate[x] == NONE) & (mate[y] == NONE)]
    assert unc.size == v["n_uncovered"]
    v["first_uncovered"] = int(unc.min()) if unc.size else 2 ** 64 - 1
    return v


def _graph(n, lengths, ordered):
    """(row ends as given, row ends as read, entries)"""
    g = _ragged(n, lengths, 5 * n)
    nb = g.nbrs.numpy()
    off = g.offsets.numpy().copy()
    off[0] = -12
    if n > 1:
        off[n - 1] = nb.size + 100
    off[n] = nb.size + 300
    if not ordered:
        off[n // 2] = nb.size + 50
        off[n // 3] = -3
    return off, np.clip(off, 0, nb.size), nb


SIZES = [(1, [9]), (33, [2, 5, 0]), (70, [3, 40, 600, 0]), (40, [17000, 3])]


@pytest.mark.parametrize("how", ["right", "none", "asym", "strangers"])
def test_checks_read_row_ends_clamped(how):
    import paper_2507_04420_gb300 as skp
    kept, verdicts = [], []
    for k, (n, lengths) in enumerate(SIZES):
        off, clipped, nb = _graph(n, lengths, ordered=False)
        ref = oracle.sgmm(np.maximum.accumulate(clipped), nb)[0]
        m = _spoiled(ref, n, how, k)
        v = _verdict(clipped, nb, m)
        d_off, d_nb, d_m = torch.from_numpy(off).cuda(), _inside(nb), _mate(m)
        with skp.Graph(d_off, d_nb, check=False) as h:
            assert h.validate(d_m).as_dict() == v, (n, how)
        with skp.Graph(d_off, d_nb, check=False, local_ids=True) as h:
            vb, eb = (torch.tensor([0, x], dtype=torch.int64, device="cuda") for x in (n, nb.size))
            assert h.validate_batched(vb, eb, d_m).as_dict() == v, (n, how)
        kept.append((d_off, d_nb, d_m))
        verdicts.append(v)
    assert [v.as_dict() for v in skp.Multi().validate(kept)] == verdicts


@pytest.mark.parametrize("bits", [2, 8, 32])
def test_serial_mode_reads_row_ends_clamped(bits):
    import paper_2507_04420_gb300 as skp
    kept, refs = [], []
    for n, lengths in SIZES:
        off, clipped, nb = _graph(n, lengths, ordered=True)
        ref = oracle.sgmm(clipped, nb)[0]
        d_off, d_nb = torch.from_numpy(off).cuda(), _inside(nb)
        with skp.Graph(d_off, d_nb, check=False) as h:
            assert np.array_equal(h.skipper(serial=1, status_bits=bits).cpu().numpy().view(np.uint32), ref), n
        kept.append((d_off, d_nb, torch.empty(n, dtype=torch.int32, device="cuda")))
        refs.append(ref)
    skp.Multi().run(kept, serial=1, status_bits=bits)
    for (_, _, m), ref in zip(kept, refs):
        assert np.array_equal(m.cpu().numpy().view(np.uint32), ref)


@pytest.mark.parametrize("graphs", [1, 3])
def test_overlapping_long_rows_beyond_the_queue(graphs):
    """Every other row is all the entries: many more rows of more than 16384
    entries than the queue has room for, each counted in full."""
    import paper_2507_04420_gb300 as skp
    n, nnz = 64, 40000
    r = np.random.RandomState(2)
    nb = r.randint(0, n, nnz).astype(np.uint32)
    off = np.where(np.arange(n + 1) % 2 == 0, 0, nnz).astype(np.int64)
    m = np.full(n, NONE, np.uint32)
    v = _verdict(off, nb, m)
    d_off, d_nb, d_m = torch.from_numpy(off).cuda(), torch.from_numpy(nb.view(np.int32)).cuda(), _mate(m)
    with skp.Graph(d_off, d_nb, check=False) as h:
        for _ in range(2):
            assert h.validate(d_m).as_dict() == v
    for got in skp.Multi().validate([(d_off, d_nb, d_m)] * graphs):
        assert got.as_dict() == v
