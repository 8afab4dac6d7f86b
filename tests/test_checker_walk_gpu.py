"""The checker's walk at the sizes where it can go wrong: rows read by one lane
(up to 32 entries at any alignment), by a warp (256 entries a step) and by the
whole grid (more than 16384 entries), in groups of 32 vertices that end early or
span graphs, on one-sided CSRs with loops and repeats, for right and for wrong
matchings.  Every field of the verdict must be the oracle's."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle
from tests.conftest import cuda_ok
from tests.test_serial_walk_gpu import _ragged

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

NONE = 0xFFFFFFFF


def _spoiled(ref, n, how, seed):
    """A copy of the matching `ref` with faults of one kind."""
    r, m = np.random.RandomState(seed), ref.copy()
    some = r.rand(n) < 0.2
    if how == "none":
        m[:] = NONE
    elif how == "dropped":      # both ends of some pairs: uncovered entries
        for v in np.flatnonzero(some):
            if m[v] != NONE:
                m[m[v]] = NONE
                m[v] = NONE
    elif how == "asym":
        m[some] = NONE
    elif how == "range":
        m[some] = r.choice([n, n + 7, NONE - 1], some.sum())
    elif how == "self":
        m[some] = np.flatnonzero(some)
    elif how == "strangers":    # symmetric pairs drawn blindly, few of them edges
        p = r.permutation(n)[: n // 2 * 2]
        m[p[0::2]], m[p[1::2]] = p[1::2], p[0::2]
    return m


HOW = ["right", "none", "dropped", "asym", "range", "self", "strangers"]
GRAPHS = [(1, [0, 1]), (31, [1, 3, 4]), (33, [28, 29, 33]), (65, [31, 32, 36, 40]), (97, [0, 255, 256, 257]),
          (70, [600, 2, 0]), (40, [16383, 16384, 16385, 5]), (3, [50000, 20001, 1]), (1000, [0, 1, 2, 5, 9, 35])]


def _mate(m):
    return torch.from_numpy(m.view(np.int32)).cuda()


@pytest.mark.parametrize("how", HOW)
def test_verdicts_are_the_oracles(how):
    import paper_2507_04420_gb300 as skp
    graphs = [_ragged(n, ln, 3 * n) for n, ln in GRAPHS] + [gg.star(40000), gg.grid(17, 33)]
    mates, verdicts, kept = [], [], []
    for k, g in enumerate(graphs):
        off, nb = g.offsets.numpy(), g.nbrs.numpy()
        m = _spoiled(oracle.sgmm(off, nb)[0], g.n, how, k)
        mates.append(m)
        verdicts.append(oracle.check(off, nb, m).as_dict())
        d = g.to("cuda")
        kept.append((d.offsets, d.nbrs, _mate(m)))
        with skp.Graph(d.offsets, d.nbrs, check=False) as h:
            for _ in range(2):  # the second check starts from the counters the first one left
                assert h.validate(kept[-1][2]).as_dict() == verdicts[k], (k, how)
    multi = skp.Multi()
    for _ in range(2):
        for k, v in enumerate(multi.validate(kept)):
            assert v.as_dict() == verdicts[k], (k, how)
    packed = gg.pack(graphs, local=True)
    vb, eb = packed.vbase.numpy(), packed.ebase.numpy()
    with skp.Graph(packed.csr.offsets.cuda(), packed.csr.nbrs.cuda(), check=False, local_ids=True) as h:
        got = h.validate_batched(packed.vbase.cuda(), packed.ebase.cuda(), _mate(np.concatenate(mates))).as_dict()
    for f in ("n_matched", "n_pairs", "n_bad_range", "n_asym", "n_nonedge", "n_uncovered"):
        assert got[f] == sum(v[f] for v in verdicts), f
    none = 2 ** 64 - 1
    for f, base in (("first_bad_vertex", vb), ("first_uncovered", eb)):
        assert got[f] == min([int(base[k]) + v[f] for k, v in enumerate(verdicts) if v[f] != none] + [none]), f
