"""The host bisection gives one layout whatever the number of threads."""
import os

import numpy as np
import pytest

import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2107_05537_gb300 as pm  # noqa: E402


# below and above the sizes that a team splits together, a degenerate top level (one
# far cluster), and points that coincide
@pytest.mark.parametrize("kind,n,leaf", [("mixture", 700, 16), ("mixture", 30_000, 16), ("mixture", 60_000, 256),
                                         ("far", 20_000, 64), ("copies", 9_000, 32)])
def test_one_thread_and_many(kind, n, leaf):
    if kind == "mixture":
        X, _, _, _ = datagen.mixture(n, 24, 40, (0.5, 2.0), seed=n)
    elif kind == "far":
        X = datagen.gaussian(n, 24, seed=3)
        X[:50] += 1000.0
    else:
        X = np.repeat(datagen.gaussian(n // 30, 24, seed=4), 30, axis=0)
    T = torch.from_numpy(X).cuda()
    cpus = os.sched_getaffinity(0)

    def build():
        ix = pm.Index(T, leaf_size=leaf, seed=1)
        lay = ix.layout()
        ix.close()
        return lay

    many = build()
    try:
        os.sched_setaffinity(0, {min(cpus)})
        one = build()
    finally:
        os.sched_setaffinity(0, cpus)
    for f in many:
        assert np.array_equal(many[f], one[f]), f
