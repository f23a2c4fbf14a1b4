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
