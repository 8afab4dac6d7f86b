"""Serial mode with a graph's matched bits in shared memory (batches of local
ids, many-graph calls): the largest graph whose bits fit and the smallest left
to the state array, windows that end early, an id out of range met and not
met.  One answer only, compared byte for byte with the oracle's."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
from tests.conftest import cuda_ok
from tests.test_serial_walk_gpu import _np, _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

FITS = 32768   # vertices


@pytest.mark.parametrize("bits", [2, 8, 32])
def test_at_the_size_limit(bits):
    import paper_2507_04420_gb300 as skp
    graphs = [_ragged(n, [0, 2, 5], n) for n in (FITS - 1, 1, FITS, 33, FITS + 1, 2 * FITS, 31)] + [gg.grid(181, 181)]
    refs = [oracle.sgmm(g.offsets.numpy(), g.nbrs.numpy())[0] for g in graphs]
    packed = gg.pack(graphs, local=True)
    d, vb, eb = packed.csr.to("cuda"), packed.vbase.cuda(), packed.ebase.cuda()
    with skp.Graph(d.offsets, d.nbrs, check=False, local_ids=True) as h:
        m = _np(h.batched(vb, eb, serial=1, status_bits=bits))
    multi = skp.Multi()
    bufs = [(g.offsets.cuda(), g.nbrs.cuda(), torch.empty(g.n, dtype=torch.int32, device="cuda")) for g in graphs]
    multi.run(bufs, serial=1, status_bits=bits)
    for k, ref in enumerate(refs):
        lo, hi = int(packed.vbase[k]), int(packed.vbase[k + 1])
        assert np.array_equal(m[lo:hi], ref), (graphs[k].n, "batch")
        assert np.array_equal(_np(bufs[k][2]), ref), (graphs[k].n, "multi")


@pytest.mark.parametrize("first_free", [True, False])
def test_an_id_out_of_range(first_free):
    import paper_2507_04420_gb300 as skp
    n = 40
    off = torch.zeros(n + 1, dtype=torch.int64)
    off[1:] = 2
    nb = torch.tensor([5, n] if first_free else [n, 5], dtype=torch.int32)
    mate = torch.empty(n, dtype=torch.int32, device="cuda")
    graphs = [(off.cuda(), nb.cuda(), mate)]
    if first_free:
        skp.Multi().run(graphs, serial=1)
    else:
        with pytest.raises(skp.SkipperError) as e:
            skp.Multi().run(graphs, serial=1)
        assert e.value.status == "MM_ERR_BAD_GRAPH"
    assert int(mate[0]) == 5 and int(mate[5]) == 0 and int((mate != -1).sum()) == 2
