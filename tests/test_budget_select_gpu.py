"""Budget cut (rule 2) by clusters of one to eight blocks, against the FP64 oracle:
few queries with many keys, more queries, a budget at the range set's size, ties of
the projected distance at the cut."""
import math

import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2107_05537_gb300 as pm  # noqa: E402


@pytest.mark.parametrize("n,nq,beta,kind", [
    (150_000, 3, 0.3, "mixture"),    # eight blocks per query
    (150_000, 40, 0.3, "mixture"),   # fewer
    (60_000, 5, 0.9, "mixture"),
    (3_000, 30, 0.2, "mixture"),     # one
    (40_000, 6, 0.5, "copies"),      # every projected distance twenty times
])
def test_cut(n, nq, beta, kind):
    X, Q, _, _ = datagen.mixture(n if kind == "mixture" else n // 20, 16, 4, 2.0, seed=n, nq=nq)
    if kind == "copies":
        X = np.repeat(X, 20, axis=0)
    A = oracle.gen_projection(7, 12, 16).astype(np.float32)
    t, _, _ = oracle.params(12, 1.5, 1 / math.e)
    r = 60.0   # every point is in range
    ix = pm.Index(torch.from_numpy(X).cuda(), m=12, leaf_size=128, proj=A)
    ref = oracle.knn(X, A, Q, 5, 1.5, t, oracle.budget(len(X), beta, 5), r, 0)
    assert (ref["rule"] == 2).any()
    for stats in (True, False):
        got = ix.knn(torch.from_numpy(Q).cuda(), k=5, beta=beta, r_min=r, t=t, with_stats=stats)
        assert np.array_equal(got["ids"].cpu().numpy(), ref["ids"])
        assert np.array_equal(got["dists"].cpu().numpy(), ref["dists"].astype(np.float32))
        if stats:
            assert np.array_equal(got["stats"]["rule"], ref["rule"])
            assert np.array_equal(got["stats"]["ncand"], ref["ncand"])
    ix.close()
