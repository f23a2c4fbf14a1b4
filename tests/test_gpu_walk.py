"""The search kernel at the edges of its layout: row widths that fill a part of a chunk
group, more selected slots than the slot table holds, beams at the edges of a 32-entry
block, and pre-filter ranges cut into many or few work items. Integer-valued vectors
whose squared distances stay below 2^24, so every float32 distance is exact and the
oracle's answers are met bit for bit."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

S, M, N, NQ = 16, 16, 3000, 37


def _table(d):
    """N vectors of d integer coordinates (d * span^2 < 2^24) around 40 centres."""
    rng = np.random.default_rng([d, 21])
    span = int(min(255, np.sqrt((1 << 24) / d) - 1))
    c = rng.uniform(0, span, size=(40, d))
    x = np.clip(np.rint(c[rng.integers(0, 40, N)] + span / 12 * rng.standard_normal((N, d))), 0, span)
    q = np.clip(np.rint(c[rng.integers(0, 40, NQ)] + span / 12 * rng.standard_normal((NQ, d))), 0, span)
    attr = rng.integers(0, 2000, N).astype(np.int64)
    w = np.rint(2000 * np.array([0.01, 0.08, 0.3, 0.9])[np.arange(NQ) % 4]).astype(np.int64)
    lo = (rng.random(NQ) * (2000 - w)).astype(np.int64)
    return x.astype(np.float32), attr, q.astype(np.float32), lo, lo + w - 1


@pytest.fixture(scope="module", params=[3, 17, 32, 100, 129, 200, 300, 515])
def table(request, tmp_path_factory):
    import hsig_build
    import oracle
    import paper_2412_02448_gb300 as U
    d = request.param
    x, attr, q, lo, hi = _table(d)
    path = os.path.join(str(tmp_path_factory.mktemp("walk")), "t.idx")
    hsig_build.build_index(x, attr, path, S, M, 40, seed=3)
    ix, oi = U.Index(path, device=0), oracle.OracleIndex(path)
    yield x, attr, q, lo, hi, ix, oi
    ix.close()
    oi.close()


def _np(r):
    import torch
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in r.items()}


@pytest.mark.parametrize("strategy,ef,m", [("hybrid", 1, 3), ("hybrid", 33, 97), ("hybrid", 200, 256),
                                           ("post", 1, 16), ("post", 32, 16), ("post", 129, 16)])
def test_walk_equals_oracle(table, strategy, ef, m):
    """Widths, beams and selections (m up to every slot: the slot table is refilled within
    an expansion); the candidate buffer holds every visited object of these tables. k stays
    within the beam (the library widens a beam below k, the oracle does not)."""
    import paper_2412_02448_gb300 as U
    x, attr, q, lo, hi, ix, oi = table
    k = min(7, ef)
    p = U.Params.defaults(ef=ef, ef_post=ef, m=m, cand_cap=4096, visited_cap=512)
    r = _np(ix.search(q, lo, hi, k, strategy=strategy, params=p, counters=True))
    o = oi.search(q, lo, hi, k, ef=ef, ef_post=ef, m=m, strategy=strategy)
    assert not r["status"].any()
    np.testing.assert_array_equal(r["ids"], o["ids"])
    np.testing.assert_array_equal(r["count"], o["count"])
    ok = r["ids"] >= 0
    np.testing.assert_array_equal(r["dist"][ok], o["dist"][ok].astype(np.float32))
    np.testing.assert_array_equal(r["counters"][:, 1], o["n_exp"])


@pytest.mark.parametrize("nq,k,scan_rows", [(1, 1, 8192), (2, 10, 8192), (37, 10, 8192), (37, 10, 32), (37, 100, 8192),
                                            (37, 256, 32)])
def test_scan_items_equal_exact(table, nq, k, scan_rows):
    """Pre-filter ranges cut into items by the size of the batch, merged list by list."""
    import oracle
    import paper_2412_02448_gb300 as U
    x, attr, q, lo, hi, ix, oi = table
    ids, dist, cnt = oracle.exact_knn(x, attr, q[:nq], lo[:nq], hi[:nq], k)
    for dtype in (U.FP32, U.BF16) if x.max() <= 255 and k <= 100 else (U.FP32,):
        r = _np(ix.search(q[:nq], lo[:nq], hi[:nq], k, strategy="pre",
                          params=U.Params.defaults(scan_rows=scan_rows, dtype=dtype)))
        np.testing.assert_array_equal(r["ids"], ids)
        np.testing.assert_array_equal(r["count"], cnt)


@pytest.mark.parametrize("d", [17, 96, 128, 300, 600])
def test_narrow_rows_equal_oracle(d, tmp_path):
    """BF16 and FP8 storage on vectors that both hold exactly (integers 0..7, every vector's
    largest coordinate 7: the FP8 scale is 1/64 and every code exact), both selections: the
    rows of float32 storage, which are the oracle's."""
    import hsig_build
    import oracle
    import paper_2412_02448_gb300 as U
    x, attr, q, lo, hi = _table(d)
    top = float(max(x.max(), q.max(), 1.0))
    x, q = np.rint(x * (7.0 / top)), np.rint(q * (7.0 / top))
    x[np.arange(N), np.arange(N) % d] = 7.0
    x, q = x.astype(np.float32), q.astype(np.float32)
    path = str(tmp_path / "t.idx")
    hsig_build.build_index(x, attr, path, S, M, 40, seed=5)
    ix, oi = U.Index(path, device=0), oracle.OracleIndex(path)
    for strategy, sel, m in (("hybrid", 2, 48), ("hybrid", 1, 40), ("post", 2, 16), ("pre", 2, 16)):
        o = oi.search(q, lo, hi, 10, ef=64, ef_post=64, m=m, strategy=strategy, selection=sel)
        for dtype in (U.FP32, U.BF16, U.FP8E4M3):
            p = U.Params.defaults(ef=64, ef_post=64, m=m, selection=sel, dtype=dtype, cand_cap=4096)
            r = _np(ix.search(q, lo, hi, 10, strategy=strategy, params=p))
            assert not r["status"].any()
            np.testing.assert_array_equal(r["ids"], o["ids"], err_msg=f"{strategy} S{sel} dtype {dtype}")
            np.testing.assert_array_equal(r["count"], o["count"])
    ix.close()
    oi.close()
