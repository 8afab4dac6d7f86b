"""A batch of lattices takes the second visits of a chunk whether its launches run
directly or as a CUDA graph: the same matching rules, and the same time (the
replay took twice as long where it ran without them)."""
import time

import pytest
import torch

import graphgen as gg
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("symmetric", [0, 1])
def test_lattices_direct_and_replayed(symmetric):
    import paper_2507_04420_gb300 as skp
    p = gg.pack([gg.grid(1000, 1000) for _ in range(20)])
    d, vb, eb = p.csr.to("cuda"), p.vbase.cuda(), p.ebase.cuda()
    best = {}
    for bits in (2, 8, 32):
        with skp.Graph(d.offsets, d.nbrs) as h:
            for use_graph in (0, 1):
                o = skp.options(status_bits=bits, symmetric=symmetric, use_graph=use_graph)
                mate = h.batched(vb, eb, opts=o)
                assert h.validate(mate).flags == 0, (bits, use_graph)
                times = []
                for _ in range(40):
                    t0 = time.perf_counter()
                    h.batched(vb, eb, mate=mate, opts=o)
                    times.append(time.perf_counter() - t0)
                best[bits, use_graph] = min(times)
    assert max(best[2, 0], best[2, 1]) <= 1.4 * min(best[2, 0], best[2, 1]), best
