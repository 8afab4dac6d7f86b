"""Grain 0 by the length of rows, seen through the units a call reports: at most
4096 rows + entries a unit where units are dispersed, 2048 below 16 rows +
entries a row, 1024 below 8 (word states: 6), 8192 in ascending order."""
import pytest
import torch

import graphgen as gg
from tests.conftest import cuda_ok

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

ROWS = [(8_000_000, 16_000_000, 4), (6_000_000, 18_000_000, 6), (6_000_000, 27_000_000, 9), (5_000_000, 80_000_000, 32)]  # vertices, edges, entries a row


@pytest.mark.parametrize("n,m,row", ROWS)
def test_the_cap_follows_the_rows(n, m, row):
    import paper_2507_04420_gb300 as skp
    g = gg.uniform(n, m, seed=3, device="cuda")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items = g.n + g.nnz
    assert items // g.n in (row, row + 1)
    mate = torch.empty(g.n, dtype=torch.int32, device="cuda")
    with skp.Graph(g.offsets, g.nbrs) as h:
        for bits in (2, 8, 32):
            for order in (0, 1):
                short = 1024 if row < (6 if bits == 32 else 8) else 2048 if row < 16 else 4096
                most = 8192 if order == 1 else short
                grain = 512
                while grain < most and grain * 1414 < items // (2 * sms * 64) * 1000:
                    grain *= 2
                h.skipper(mate=mate, status_bits=bits, unit_order=order, timing=1)
                assert h.timing()["units"] == -(-items // grain), (row, bits, order)
