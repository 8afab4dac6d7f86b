"""The pair list (u, mate[u]), u < mate[u], in ascending u, at the edges of its
tiles (16384 vertices, parts of 128), with more tiles than one look back
covers, a mate array that is not 16-byte aligned, and room for fewer pairs."""
import numpy as np
import pytest
import torch

import graphgen as gg
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n", [1, 2, 127, 129, 1025, 2047, 4097, 16383, 16384, 16385, 40000, 700001])
def test_pairs_are_the_mates_in_order(n):
    import paper_2507_04420_gb300 as skp
    p = torch.from_numpy(np.random.RandomState(n).permutation(n))
    k = n // 2
    g = gg.from_edges(n, p[:k // 2 * 1], p[k:k + k // 2])   # a random matching of about n / 4 edges, and lone vertices
    e = gg.edge_list(g)
    d = g.to("cuda")
    buf = torch.empty(n + 4, dtype=torch.int32, device="cuda")
    with skp.Graph(d.offsets, d.nbrs) as h, skp.EdgeList(n, e[0].cuda(), e[1].cuda()) as l:
        for handle in (h, l):
            for shift in (0, 1, 3):
                for kw in ({}, {"serial": 1}, {"status_bits": 32}, {"cap": max(1, k // 5)}):
                    cap = kw.get("cap")
                    mate, pairs, count = handle.skipper(mate=buf[shift:shift + n], pairs=True, **kw)
                    m = mate.cpu().numpy()
                    u = np.flatnonzero(m > np.arange(n))
                    assert int(count) == u.size == g.nnz // 2
                    got = pairs.cpu().numpy()[:min(u.size, cap or u.size)]
                    assert np.array_equal(got, np.stack([u, m[u]], 1)[:len(got)])
