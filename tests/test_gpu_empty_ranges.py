"""Queries whose range holds nothing: no walk, no distance evaluation, an empty row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strategy", ["post", "hybrid", "pre", "auto"])
def test_counters_of_empty_ranges(strategy, c2_small_index):
    """lo > hi, and ranges between and beyond the attribute values, among ordinary queries:
    the counters of a query without a walk are the oracle's (0, 0)."""
    import oracle
    import paper_2412_02448_gb300 as U
    import torch
    w, path = c2_small_index
    q, lo, hi = w.queries[:12], w.lo[:12].copy(), w.hi[:12].copy()
    lo[[1, 4]], hi[[1, 4]] = 50, 40
    top = int(w.attrs.max())
    lo[[7, 9]], hi[[7, 9]] = top + 10, top + 20
    ix, oi = U.Index(path, device=0), oracle.OracleIndex(path)
    tau = dict(tau_a=w.n // 100, tau_b=w.n // 2)
    r = ix.search(q, lo, hi, 5, strategy=strategy, counters=True,
                  params=U.Params.defaults(ef=32, cand_cap=4096, visited_cap=4096, **tau))
    torch.cuda.synchronize()
    r = {k: v.cpu().numpy() for k, v in r.items()}
    o = oi.search(q, lo, hi, 5, ef=32, m=16, strategy=strategy, **tau)
    np.testing.assert_array_equal(r["count"], o["count"])
    none = o["n_exp"] + o["n_dist"] == 0
    assert none.sum() >= 2
    np.testing.assert_array_equal(r["counters"][none, :2], 0)
    assert (r["ids"][none] == -1).all() and np.isinf(r["dist"][none]).all()
    ix.close()
    oi.close()
