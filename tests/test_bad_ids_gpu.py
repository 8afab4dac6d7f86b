"""An unchecked input full of ids out of range: a call that waits, whose kernels
report straight to the host, takes no longer than one that does not (crossing the
link for every bad entry, it took ten times as long)."""
import time

import pytest
import torch

import graphgen as gg
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


def test_every_id_out_of_range():
    import paper_2507_04420_gb300 as skp
    n = 4_000_000
    g = gg.uniform(n, 20_000_000, seed=7, device="cuda")
    mate = torch.empty(n, dtype=torch.int32, device="cuda")
    with skp.Graph(g.offsets, g.nbrs + n, check=False) as h:
        def run(**kw):
            t0 = time.perf_counter()
            with pytest.raises(skp.SkipperError) as e:
                h.skipper(mate=mate, **kw)
                h.sync()
            assert e.value.status == "MM_ERR_BAD_GRAPH"
            return time.perf_counter() - t0
        waiting, behind = (min(run(**kw) for _ in range(5)) for kw in ({}, {"nosync": 1}))
        assert waiting <= 3 * behind, (waiting, behind)
        assert (mate == -1).all()
