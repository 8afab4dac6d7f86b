"""Serial mode's warp walk at the sizes where it can go wrong: windows of 31 to
33 rows, rows of 0 to 500 entries that cross the 128-entry chunks at every
alignment, loops, repeats, unsorted and one-sided rows, graphs that share state
words in a batch.  Sequential greedy has one answer, so results are compared
byte for byte with the oracle's."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def _np(t):
    return t.cpu().numpy().view(np.uint32)


def _ragged(n, lengths, seed):
    """Rows of the given lengths in turn, ids drawn near the row and anywhere."""
    r = np.random.RandomState(seed)
    deg = np.array([lengths[r.randint(len(lengths))] for _ in range(n)], np.int64)
    rows = np.repeat(np.arange(n), deg)
    near = np.clip(rows + r.randint(-40, 41, rows.size), 0, n - 1)
    ids = np.where(r.rand(rows.size) < 0.5, near, r.randint(0, n, rows.size))
    off = np.concatenate([[0], np.cumsum(deg)])
    return gg.CSR(torch.from_numpy(off), torch.from_numpy(ids.astype(np.int32)))


SIZES = [1, 2, 31, 32, 33, 63, 65, 97, 1000]
LENGTHS = [[1], [0, 0, 1, 3], [4, 5, 7], [0, 127, 128, 129], [500, 0, 2]]


@pytest.mark.parametrize("bits", [2, 8, 32])
def test_ragged_graphs_alone_and_packed(bits):
    import paper_2507_04420_gb300 as skp
    graphs = [_ragged(n, ln, 7 * n + i) for n in SIZES for i, ln in enumerate(LENGTHS)]
    refs = [oracle.sgmm(g.offsets.numpy(), g.nbrs.numpy())[0] for g in graphs]
    for g, ref in zip(graphs, refs):
        d = g.to("cuda")
        with skp.Graph(d.offsets, d.nbrs) as h:
            assert np.array_equal(_np(h.skipper(serial=1, status_bits=bits)), ref), g.n
    for local in (False, True):
        packed = gg.pack(graphs, local=local)
        d, vb, eb = packed.csr.to("cuda"), packed.vbase.cuda(), packed.ebase.cuda()
        with skp.Graph(d.offsets, d.nbrs, check=False, local_ids=local) as h:
            m = _np(h.batched(vb, eb, serial=1, status_bits=bits))
        for k, ref in enumerate(refs):
            lo, hi = int(packed.vbase[k]), int(packed.vbase[k + 1])
            shift = np.uint32(0 if local else lo)
            assert np.array_equal(m[lo:hi], np.where(ref == 0xFFFFFFFF, ref, ref + shift)), (local, k)


@pytest.mark.parametrize("first_free", [True, False])
def test_an_id_out_of_range_counts_only_when_the_order_reaches_it(first_free):
    """Row 0 lists a free neighbour and the id n: greedy stops at the free one."""
    import paper_2507_04420_gb300 as skp
    n = 40
    off = torch.zeros(n + 1, dtype=torch.int64)
    off[1:] = 2
    nb = torch.tensor([5, n] if first_free else [n, 5], dtype=torch.int32)
    with skp.Graph(off.cuda(), nb.cuda(), check=False) as h:
        if first_free:
            assert int(h.skipper(serial=1)[5]) == 0
        else:
            with pytest.raises(skp.SkipperError) as e:
                h.skipper(serial=1)
            assert e.value.status == "MM_ERR_BAD_GRAPH"
