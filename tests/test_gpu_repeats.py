"""Index files whose rows name a neighbour more than once. The loader takes them, and the
paper's algorithms pass over the repetition (visited already): every walk has to meet the
oracle's answers. Integer-valued vectors, so that every distance is exact."""
import os

import numpy as np
import pytest
from index_writer import _CODES, write_index

pytestmark = pytest.mark.gpu

N, D, NQ = 3000, 24, 41
_TYPES = {c: t for t, c in _CODES.items()}


def _sections(path):
    b = open(path, "rb").read()
    out = {}
    for i in range(int.from_bytes(b[12:16], "little")):
        e = b[16 + 96 * i:16 + 96 * (i + 1)]
        code, ndim = np.frombuffer(e[24:32], "<u4")
        shape = np.frombuffer(e[32:64], "<u8")[:ndim].astype(int)
        off, size = np.frombuffer(e[64:80], "<u8")
        out[e[:24].rstrip(b"\0").decode()] = np.frombuffer(b, _TYPES[int(code)], count=int(np.prod(shape)),
                                                           offset=int(off)).reshape(shape).copy()
    return out


def _repeat(adj, gmask, rng):
    """In about half of the chunks of (rows, S, M) slots: the first slot's id in the last
    taken slot or in the first free one, and both marked if one of them is."""
    rows, S, M = adj.shape
    for r in range(rows):
        for j in np.flatnonzero(rng.random(S) < 0.5):
            c = int((adj[r, j] >= 0).sum())
            if c < 1:
                continue
            s = c if c < M and rng.random() < 0.5 else max(c - 1, 0)
            if s == 0:
                continue
            adj[r, j, s] = adj[r, j, 0]
            p, p2 = j * M, j * M + s
            if (gmask[r, p // 32] >> np.uint32(p % 32)) & 1 or (gmask[r, p2 // 32] >> np.uint32(p2 % 32)) & 1:
                gmask[r, p // 32] |= np.uint32(1) << np.uint32(p % 32)
                gmask[r, p2 // 32] |= np.uint32(1) << np.uint32(p2 % 32)


@pytest.fixture(scope="module", params=[(16, 16), (3, 64)], ids=["16x16", "3x64"])
def repeated(request, tmp_path_factory):
    import hsig_build
    import oracle
    import paper_2412_02448_gb300 as U
    S, M = request.param
    rng = np.random.default_rng([S, M, 5])
    c = rng.integers(0, 200, (30, D))
    x = np.clip(c[rng.integers(0, 30, N)] + rng.integers(-25, 26, (N, D)), 0, 255).astype(np.float32)
    q = np.clip(c[rng.integers(0, 30, NQ)] + rng.integers(-25, 26, (NQ, D)), 0, 255).astype(np.float32)
    attr = rng.integers(0, 2000, N).astype(np.int64)
    w = np.rint(2000 * np.array([0.05, 0.3, 0.9])[np.arange(NQ) % 3]).astype(np.int64)
    lo = (rng.random(NQ) * (2000 - w)).astype(np.int64)
    d = tmp_path_factory.mktemp("repeats")
    hsig_build.build_index(x, attr, str(d / "a.idx"), S, M, 80, seed=3)
    s = _sections(str(d / "a.idx"))
    for a, g in (("adj0", "gmask0"), ("adjU", "gmaskU")):
        _repeat(s[a].reshape(-1, S, M), s[g], rng)
    path = write_index(str(d / "b.idx"), s)
    ix, oi = U.Index(path, device=0), oracle.OracleIndex(path)
    yield q, lo, lo + w - 1, ix, oi
    ix.close()
    oi.close()


@pytest.mark.parametrize("strategy,sel,ef,m", [("hybrid", 2, 40, 48), ("hybrid", 2, 90, 192), ("hybrid", 1, 40, 40),
                                               ("hybrid", 1, 64, 64), ("post", 2, 60, 16)])
@pytest.mark.parametrize("visited", [64, 4096])
def test_walk_over_repeated_neighbours(repeated, strategy, sel, ef, m, visited):
    """A small visited filter forgets ids between the two places of one."""
    import paper_2412_02448_gb300 as U
    import torch
    q, lo, hi, ix, oi = repeated
    p = U.Params.defaults(ef=ef, ef_post=ef, m=m, selection=sel, cand_cap=4096, visited_cap=visited)
    r = ix.search(q, lo, hi, 10, strategy=strategy, params=p, counters=True)
    torch.cuda.synchronize()
    r = {k: v.cpu().numpy() for k, v in r.items()}
    o = oi.search(q, lo, hi, 10, ef=ef, ef_post=ef, m=m, strategy=strategy, selection=sel)
    assert not r["status"].any()
    np.testing.assert_array_equal(r["ids"], o["ids"])
    np.testing.assert_array_equal(r["count"], o["count"])
    np.testing.assert_array_equal(r["counters"][:, 1], o["n_exp"])
    for row in r["ids"]:
        found = row[row >= 0]
        assert len(found) == len(set(found.tolist()))
