"""Pre-filter batches on a handle whose scratch is larger than they need, and at the ends of
the scan's parameters. Integer-valued vectors: every distance is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(ix, w, rows, k, **kw):
    import paper_2412_02448_gb300 as U
    import torch
    r = ix.search(w.queries[rows], w.lo[rows], w.hi[rows], k, strategy="pre", params=U.Params.defaults(**kw))
    torch.cuda.synchronize()
    return {n: v.cpu().numpy() for n, v in r.items()}


@pytest.mark.parametrize("nq", [1, 9, 150])
def test_small_tensor_core_batch_after_a_large_one(nq, c2_small_index):
    """The tables of the tensor-core scan are those of the largest batch so far: more CTAs
    clear them than the batch has queries."""
    import oracle
    import paper_2412_02448_gb300 as U
    w, path = c2_small_index
    big = np.arange(30_000) % len(w.queries)
    ids, _, cnt = oracle.exact_knn(w.vectors, w.attrs, w.queries, w.lo, w.hi, 10)
    ix = U.Index(path, device=0)
    for rows in (big, np.arange(nq), big[:700], np.arange(nq)[::-1].copy()):
        r = _run(ix, w, rows, 10, tc_scan=1)
        np.testing.assert_array_equal(r["ids"], ids[rows])
        np.testing.assert_array_equal(r["count"], cnt[rows])
    ix.close()


@pytest.mark.parametrize("k,mult", [(1, 1), (33, 4), (256, 16)])
def test_pre_filter_lists_without_walk_buffers(k, mult, c2_small_index):
    """A forced pre-filter batch gets shared memory for its lists alone, whatever the walks'
    parameters: up to 4,096 candidates re-ranked, the smallest and a large beam."""
    import oracle
    import paper_2412_02448_gb300 as U
    w, path = c2_small_index
    rows = np.arange(60)
    ids, _, cnt = oracle.exact_knn(w.vectors, w.attrs, w.queries[rows], w.lo[rows], w.hi[rows], k)
    ix = U.Index(path, device=0)
    for dtype in (U.FP32, U.BF16):  # coordinates up to 255 are exact in both
        for kw in (dict(visited_cap=64, cand_cap=32, ef=1), dict(visited_cap=8192, cand_cap=2048, ef=300)):
            r = _run(ix, w, rows, k, dtype=dtype, rerank_mult=mult, warps_per_block=2, **kw)
            np.testing.assert_array_equal(r["ids"], ids)
            np.testing.assert_array_equal(r["count"], cnt)
    ix.close()


@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_routed_scans_in_every_build(dtype, c2_small_index):
    """Pre-filter items of a routed batch in the builds of 128, 96 and 80 registers (which load
    narrow rows in two ways), next to walks: the same rows. Small buffers let the smaller
    builds be taken, larger ones take 128 registers for every budget."""
    import paper_2412_02448_gb300 as U
    import torch
    w, path = c2_small_index
    ix = U.Index(path, device=0)
    out = []
    for regs, vis in ((128, 1024), (80, 1024), (64, 1024), (64, 8192), (80, 8192)):
        p = U.Params.defaults(dtype=dtype, reg_budget=regs, tau_a=w.n // 10, tau_b=w.n // 2, rerank_mult=2, ef=32,
                              cand_cap=1024 if vis > 1024 else 256, visited_cap=vis)
        r = ix.search(w.queries, w.lo, w.hi, 10, strategy="auto", params=p)
        torch.cuda.synchronize()
        out.append({n: v.cpu().numpy() for n, v in r.items()})
    for r in out[1:]:
        ok = (r["status"] | out[0]["status"]) == 0  # a full candidate buffer drops its worst entries
        for n in ("ids", "dist", "count"):
            np.testing.assert_array_equal(r[n][ok], out[0][n][ok])
    assert ok.mean() > 0.5
    ix.close()
