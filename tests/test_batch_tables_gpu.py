"""The batch checker on a vertex table that does not end where the batch does: no
table is read past its end and no vertex outside the batch is reached."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
from tests.conftest import cuda_ok
from tests.test_checker_walk_gpu import _mate
from tests.test_serial_walk_gpu import _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("last", [37, 130, 300])
def test_a_last_entry_that_is_not_the_batchs_end(last):
    import paper_2507_04420_gb300 as skp
    graphs = [_ragged(40, [3, 0, 70], 1), gg.grid(9, 20), _ragged(last, [2, 5, 33], 3)]
    packed = gg.pack(graphs, local=True)
    mates = [oracle.sgmm(g.offsets.numpy(), g.nbrs.numpy())[0] for g in graphs]
    m = _mate(np.concatenate(mates))
    n = int(packed.vbase[-1])
    with skp.Graph(packed.csr.offsets.cuda(), packed.csr.nbrs.cuda(), check=False, local_ids=True) as h:
        eb = packed.ebase.cuda()
        right = h.validate_batched(packed.vbase.cuda(), eb, m).as_dict()
        assert right["flags"] == 0
        for end in (n + 1, n + 1000, 2 ** 40):
            vb = packed.vbase.clone()
            vb[-1] = end
            assert h.validate_batched(vb.cuda(), eb, m).as_dict() == right, end
        for short in (1, 20, last):
            vb = packed.vbase.clone()
            vb[-1] = n - short
            cut = mates[2][mates[2] != 0xFFFFFFFF]      # partners that the table leaves out
            got = h.validate_batched(vb.cuda(), eb, m)
            assert got.n_bad_range == int((cut >= last - short).sum()), short
            assert (got.n_asym, got.n_nonedge, got.n_uncovered) == (0, 0, 0), short
