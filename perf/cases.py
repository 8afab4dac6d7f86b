"""The work that a user of this library has it do, as cases that can be timed.

What a pass returns.  A parallel pass finds *a* maximal matching; which one
depends on timing (``skipper.h``, mm_skipper), so its mates cannot be compared
from one run to the next.  What every correct pass has in common is returned
instead: where the checker is part of the work, its verdict (whole numbers:
violation flags and counts), and where it is not, the share of the vertices that
found a partner, in the few digits (float16) that timing leaves alone; beside
either, the number of entries that the answer is about.  Serial mode is sequential greedy, one answer
only, so its mates come back whole.

A case is one of these kinds (``kind``):
  csr    one CSR in device memory: the pass, with its pair list or the checker
  host   one CSR in page-locked host memory, read in place: pass and pair list
  list   one edge list in device memory: the pass and its pair list
  batch  many graphs packed block-diagonally, replayed as a CUDA graph and checked
  multi  many graphs in buffers of their own, matched in one launch and checked
  order  many packed graphs in serial mode, one reproducible answer a graph
"""
import math

import numpy as np
import torch

import paper_2507_04420_gb300 as skp

DEV = "cuda"


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 12345)
    return g


def _levels_table():
    """Three R-MAT levels at once: 2^16 slots, each quadrant path (a, b, c, d =
    .57, .19, .19, .05 a level) in about as many slots as its probability."""
    p = np.array([0.57, 0.19, 0.19, 0.05])
    q = np.einsum("i,j,k->ijk", p, p, p).reshape(-1)
    edge = np.rint(np.cumsum(q) * 65536).astype(np.int64)
    code = np.searchsorted(edge, np.arange(65536), side="right")
    u, v = np.zeros(65536, np.int32), np.zeros(65536, np.int32)
    for lvl in range(3):
        quad = code >> (2 * (2 - lvl)) & 3
        u, v = u << 1 | (quad >> 1), v << 1 | (quad & 1)
    return torch.from_numpy(u.astype(np.int32)).to(DEV), torch.from_numpy(v.astype(np.int32)).to(DEV)


def _rmat_draws(m, levels, rng):
    """m endpoint pairs of `levels` R-MAT levels (a multiple of 3 or more is cut), int32."""
    tu, tv = _levels_table()
    us, vs = [], []
    for at in range(0, m, 1 << 26):
        k = min(1 << 26, m - at)
        u = torch.zeros(k, dtype=torch.int32, device=DEV)
        v = torch.zeros(k, dtype=torch.int32, device=DEV)
        groups = -(-levels // 3)
        for i in range(groups):
            if i % 3 == 0:
                r = torch.randint(0, 1 << 48, (k,), generator=rng, device=DEV)
            s = (r >> (16 * (i % 3)) & 0xFFFF).to(torch.int32)
            u, v = u << 3 | tu[s], v << 3 | tv[s]
        cut = 3 * groups - levels
        us.append(u >> cut)
        vs.append(v >> cut)
    return torch.cat(us), torch.cat(vs)


def _edges(case, rng):
    """Endpoint pairs of one graph: (n, u, v), int32, loops and repeats as drawn."""
    if case["family"] == "grid":  # a road-like lattice in row-major order, a few edges missing
        rows, cols = case["rows"], case["cols"]
        ids = torch.arange(rows * cols, dtype=torch.int32, device=DEV).reshape(rows, cols)
        u = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
        v = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
        keep = torch.rand(u.numel(), generator=rng, device=DEV) < 0.97
        return rows * cols, u[keep], v[keep]
    n, m = case["n"], case["m"]
    if case["family"] == "uniform":
        u = torch.randint(0, n, (m,), generator=rng, device=DEV, dtype=torch.int32)
        v = torch.randint(0, n, (m,), generator=rng, device=DEV, dtype=torch.int32)
        return n, u, v
    scale = max(1, (n - 1).bit_length())  # rmat, ids in random order
    u, v = _rmat_draws(m, scale, rng)
    ids = (torch.randperm(1 << scale, generator=rng, device=DEV) % n).to(torch.int32)
    return n, ids[u], ids[v]


def _csr(n, u, v):
    """Symmetric CSR, rows sorted, loops and repeats dropped; by ranges of rows
    so that the sort of a large graph takes little memory."""
    parts, deg = [], torch.zeros(n, dtype=torch.int64, device=DEV)
    step = max(1, -(-n // max(1, -(-u.numel() // (1 << 27)))))
    for lo in range(0, n, step):
        hi = min(n, lo + step)
        keys = []
        for a, b in ((u, v), (v, u)):
            at = (a != b) if step >= n else (a >= lo) & (a < hi) & (a != b)
            keys.append((a[at].long() - lo) * n + b[at])
        key = torch.unique(torch.cat(keys))
        del keys
        row = torch.div(key, n, rounding_mode="floor")
        deg[lo:hi] = torch.bincount(row, minlength=hi - lo)
        parts.append((key - row * n).to(torch.int32))
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(deg, 0, out=off[1:])
    return off, parts[0] if len(parts) == 1 else torch.cat(parts)


def _packed(case, seed):
    """`graphs` graphs with edge counts log-uniform in [m_lo, m_hi], uniform,
    R-MAT and lattice in turn, side by side: (offsets, global ids, vbase, ebase).
    The sizes are the case's own, the edges of the random graphs the seed's."""
    rng, G = _rng(seed), case["graphs"]
    r = np.random.RandomState(G + case["m_hi"])
    m = np.exp(r.uniform(math.log(case["m_lo"]), math.log(case["m_hi"]), G)).astype(np.int64)
    ef = r.randint(8, 33, G)
    kind = np.arange(G) % 3
    scale = np.maximum(4, np.rint(np.log2(m / ef))).astype(np.int64)
    side = np.maximum(2, np.rint(np.sqrt(m / 2))).astype(np.int64)
    n = np.where(kind == 0, np.maximum(16, 2 * m // ef), np.where(kind == 1, 1 << scale, side * side))
    vbase = torch.from_numpy(np.concatenate([[0], np.cumsum(n)])).to(DEV)

    def spread(which, count):  # the graph of each edge, and a column of its values
        g = torch.from_numpy(np.flatnonzero(which)).to(DEV)
        return torch.repeat_interleave(g, torch.from_numpy(count[which]).to(DEV))

    us, vs = [], []
    g = spread(kind == 0, m)
    nn = torch.from_numpy(n).to(DEV)[g]
    for out in (us, vs):
        out.append((torch.rand(g.numel(), generator=rng, device=DEV, dtype=torch.float64) * nn).long() + vbase[g])
    g = spread(kind == 1, m)
    if g.numel():
        top = int(scale[kind == 1].max())
        cut = top - torch.from_numpy(scale).to(DEV)[g]
        for x, out in zip(_rmat_draws(g.numel(), top, rng), (us, vs)):
            x = (x.long() >> cut) * 0x9E3779B1 & ((1 << (top - cut)) - 1)  # ids out of order
            out.append(x + vbase[g])
    for step_r, step_c in ((0, 1), (1, 0)):
        count = side * (side - 1)
        g = spread(kind == 2, count)
        if g.numel() == 0:
            continue
        sd = torch.from_numpy(side).to(DEV)[g]
        first = torch.from_numpy(np.cumsum(np.where(kind == 2, count, 0)) - np.where(kind == 2, count, 0)).to(DEV)[g]
        i = torch.arange(g.numel(), device=DEV) - first
        width = sd - step_c
        a = i // width * sd + i % width
        us.append(a + vbase[g])
        vs.append(a + step_r * sd + step_c + vbase[g])
    off, nbrs = _csr(int(vbase[-1]), torch.cat(us), torch.cat(vs))
    return off, nbrs, vbase, off[vbase].contiguous()


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one small request: a call is launches and waits more than work
        dict(name="call-1k-edges", kind="csr", family="uniform", n=100, m=1000, bits=8, symmetric=0, check=True),
        # a graph of a few million edges, the pairs wanted as a list
        dict(name="rmat18-pairs", kind="csr", family="rmat", n=1 << 18, m=1 << 22, bits=8, symmetric=0, check=False),
        # a social-network-like graph in the layout whose states are the mates, matched and checked
        dict(name="rmat22-word-check", kind="csr", family="rmat", n=1 << 22, m=1 << 26, bits=32, symmetric=0, check=True),
        # the benchmark's headline: R-MAT 27, edge factor 16, a byte a vertex (2 bits and words are in the draws)
        dict(name="rmat27-pairs", kind="csr", family="rmat", n=1 << 27, m=1 << 31, bits=8, symmetric=0, check=False),
        # low locality, most rows open when their turn comes; 2-bit states, the CSR declared symmetric
        dict(name="uniform-2bit-sym", kind="csr", family="uniform", n=20000003, m=200000000, bits=2, symmetric=1, check=False),
        # ids with locality (road networks, meshes): reservations meet; matched and checked
        dict(name="grid-check", kind="csr", family="grid", rows=4096, cols=4096, bits=8, symmetric=0, check=True),
        # coordinate input in generator order, each edge once, repeats and loops as drawn
        dict(name="list-rmat24", kind="list", family="rmat", n=1 << 24, m=1 << 28, bits=2),
        # the packed batch of the batched benchmark with graphs up to 1e5 edges, replayed, the result checked
        dict(name="batch-4096-check", kind="batch", graphs=4096, m_lo=1000, m_hi=100000, bits=8, local=False),
        # what the server launches and checks at once: requests in buffers of their own
        dict(name="multi-171-check", kind="multi", graphs=171, m_lo=1000, m_hi=1000000, bits=8),
        # reproducible results: sequential greedy on every graph of a batch
        dict(name="order-4096", kind="order", graphs=4096, m_lo=100, m_hi=10000, bits=8, local=True),
        # the graph stays in host memory and is read in place
        dict(name="host-rmat22", kind="host", family="rmat", n=1 << 22, m=1 << 26, bits=8, symmetric=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["csr", "csr", "csr", "host", "list", "batch", "multi", "order"])
    bits = rng.choice([8, 8, 2, 32])
    if kind in ("batch", "multi", "order"):
        top = {"batch": 100000, "multi": 1000000, "order": 10000}[kind]
        lo = _log(rng, 100, top / 30)
        c = dict(kind=kind, graphs=_log(rng, 8 if kind == "multi" else 64, 400 if kind == "multi" else 4096),
                 m_lo=lo, m_hi=_log(rng, 10 * lo, top), bits=bits)
        return c if kind == "multi" else dict(c, local=rng.random() < 0.5)
    family = rng.choice(["rmat", "uniform"] if kind == "list" else ["rmat", "uniform", "grid"])
    m = _log(rng, 1000 if kind == "csr" else 1 << 20, 1 << 28 if kind == "list" else 1 << 26 if kind == "host" else 3 << 26)
    c = dict(kind=kind, family=family)
    if family == "grid":
        cols = max(8, int(math.sqrt(m / 2) * rng.uniform(0.5, 2)))
        c.update(rows=max(8, m // (2 * cols)), cols=cols)
    else:
        c.update(n=max(16, int(m / rng.uniform(4, 32))), m=m)
    c["bits"] = bits
    if kind != "list":
        c["symmetric"] = int(rng.random() < 0.3)
    if kind == "csr":  # timing moves the size of a small graph's or a lattice's matching too much
        c["check"] = m < 500000 or family == "grid" or rng.random() < 0.4
    return c


def prepare(case, seed):
    kind = case["kind"]
    opts = dict(status_bits=case["bits"])
    if kind in ("batch", "order", "multi"):
        off, nbrs, vbase, ebase = _packed(case, seed)
        if kind == "multi":
            v, e = vbase.tolist(), ebase.tolist()
            graphs = []
            for i in range(case["graphs"]):
                o = off[v[i]:v[i + 1] + 1] - e[i]
                graphs.append((o, nbrs[e[i]:e[i + 1]] - v[i], torch.empty(o.numel() - 1, dtype=torch.int32, device=DEV)))
            return dict(kind=kind, handle=skp.Multi(), graphs=graphs, entries=nbrs.numel(), opts=skp.options(**opts))
        if case["local"]:
            nbrs -= torch.repeat_interleave(vbase[:-1], ebase[1:] - ebase[:-1]).to(torch.int32)
        opts["use_graph"] = 1
        opts["serial"] = int(kind == "order")
        handle = skp.Graph(off, nbrs, check=not case["local"], local_ids=case["local"])
        mate = torch.empty(off.numel() - 1, dtype=torch.int32, device=DEV)
        return dict(kind=kind, handle=handle, vbase=vbase, ebase=ebase, mate=mate, entries=nbrs.numel(),
                    opts=skp.options(**opts))
    n, u, v = _edges(case, _rng(seed))
    mate = torch.empty(n, dtype=torch.int32, device=DEV)
    state = dict(kind=kind, mate=mate, check=case.get("check", False))
    if kind == "list":
        state.update(handle=skp.EdgeList(n, u, v), entries=int((u != v).sum()))
    else:
        opts["symmetric"] = case["symmetric"]
        off, nbrs = _csr(n, u, v)
        del u, v
        if kind == "host":
            off, nbrs = off.cpu().pin_memory(), nbrs.cpu().pin_memory()
        state.update(handle=skp.Graph(off, nbrs, host_mapped=kind == "host"), entries=nbrs.numel())
    state["opts"] = skp.options(**opts)
    return state


def _faults(v):
    return [int(v.flags), int(v.n_bad_range), int(v.n_asym), int(v.n_nonedge), int(v.n_uncovered)]


def run(state):
    kind, handle, opts = state["kind"], state["handle"], state["opts"]
    if kind == "multi":
        handle.run(state["graphs"], opts=opts)
        verdicts = handle.validate(state["graphs"])
        return dict(entries=state["entries"], flags=np.array([v.flags for v in verdicts], dtype=np.int64))
    if kind == "order":
        return dict(mate=handle.batched(state["vbase"], state["ebase"], mate=state["mate"], opts=opts))
    if kind == "batch":
        mate = handle.batched(state["vbase"], state["ebase"], mate=state["mate"], opts=opts)
        verdict = handle.validate_batched(state["vbase"], state["ebase"], mate)
        return dict(entries=state["entries"], faults=_faults(verdict))
    if state["check"]:
        mate = handle.skipper(mate=state["mate"], opts=opts)
        return dict(entries=state["entries"], faults=_faults(handle.validate(mate)))
    mate, _, count = handle.skipper(mate=state["mate"], pairs=True, opts=opts)
    return dict(entries=state["entries"], share=(count / mate.numel()).to(torch.float16))


def work(case):
    """The input read once (row ends 8 bytes, an entry 4, both directions of an
    edge stored; a listed edge 8) and the mates and the pairs written once."""
    kind = case["kind"]
    if kind in ("batch", "multi", "order"):
        lo, hi = case["m_lo"], case["m_hi"]
        m = case["graphs"] * (hi - lo) / math.log(hi / lo)  # the mean of log-uniform edge counts
        n = m * (1 / 10 + 1 / 20 + 1 / 2) / 3
        return dict(bytes=8 * n + 8 * m + 4 * n, flops=0)
    if case["family"] == "grid":
        n, m = case["rows"] * case["cols"], 2 * case["rows"] * case["cols"] * 0.97
    else:
        n, m = case["n"], case["m"]
    pairs = 0 if case.get("check") else 8 * 0.3 * n
    return dict(bytes=(0 if kind == "list" else 8 * n) + 8 * m + 4 * n + pairs, flops=0)


def exact(case, seed):
    """Every output is a whole number or depends on timing (above): none has a 64-bit value to be held to."""
    return None
