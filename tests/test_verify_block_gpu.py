"""Verification by a block per query (smaller batches) and by a warp per query
(larger ones) at the sizes where they can go wrong, against the FP64 oracle: ids
equal, distances the FP32 rounding of the FP64 values (exact), the trace equal."""
import math

import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2107_05537_gb300 as pm  # noqa: E402


def _check(X, Q, A, k, leaf=64, beta=0.2809, precision=0, copies=1, with_stats=True, r_min=0.0):
    ix = pm.Index(torch.from_numpy(X).cuda(), m=A.shape[0], leaf_size=leaf, proj=A)
    t, _, _ = oracle.params(A.shape[0], 1.5, 1 / math.e)
    got = ix.knn(torch.from_numpy(np.tile(Q, (copies, 1))).cuda(), k=k, beta=beta, t=t, precision=precision,
                 with_stats=with_stats, r_min=r_min)
    torch.cuda.synchronize()
    ix.close()
    r0 = r_min if r_min > 0 else oracle.rmin_auto(X, beta, k, 1.5, 3)
    ref = oracle.knn(X, A, Q, k, 1.5, t, oracle.budget(len(X), beta, k), r0, 0)
    ids = got["ids"].cpu().numpy().reshape(copies, len(Q), k)
    dd = got["dists"].cpu().numpy().reshape(copies, len(Q), k)
    assert (ids == ref["ids"][None]).all()
    assert (dd == ref["dists"].astype(np.float32)[None]).all()
    if with_stats:
        for f in ("rounds", "rule", "ncand"):
            assert (got["stats"][f].reshape(copies, -1) == ref[f][None]).all()


# rows of 1 to 9 steps of 32 coordinates (whole and partial load steps), 8 warps
# per block (up to two blocks per SM) and 4
@pytest.mark.parametrize("d", [1, 32, 33, 64, 96, 100, 128, 160, 192, 250, 288])
@pytest.mark.parametrize("copies", [1, 13])
def test_row_lengths(d, copies):
    X, Q, _, _ = datagen.mixture(3000, d, 9, 1.0, seed=d, nq=29)
    A = oracle.gen_projection(3, 15, d).astype(np.float32)
    _check(X, Q, A, 10, copies=copies)


# guard sets of one warp's rows, of two, and of several turns of the buffer; leaves
# of a few and of a thousand points (one leaf per group, many leaves per group)
@pytest.mark.parametrize("k", [1, 31, 33, 64, 65, 129, 256])
@pytest.mark.parametrize("leaf", [16, 1024])
def test_neighbours_and_leaf_sizes(k, leaf):
    X, Q, _, _ = datagen.mixture(5000, 40, 3, 1.0, seed=k, nq=20)
    A = oracle.gen_projection(4, 15, 40).astype(np.float32)
    _check(X, Q, A, k, leaf=leaf)
    _check(X, Q, A, k, leaf=leaf, with_stats=False, beta=0.02)


# coordinates whose squares the integer arithmetic takes and those it leaves to the
# FP64 pipe: exponents far apart, zeros of both signs, subnormals, small integers
@pytest.mark.parametrize("kind", ["spread", "integers", "sparse", "subnormal"])
def test_exact_squares(kind):
    rng = np.random.default_rng(5)
    n, d = 2000, 48
    if kind == "spread":
        Y = rng.standard_normal((n + 24, d)) * 2.0 ** rng.integers(-12, 12, (n + 24, d))
    elif kind == "integers":
        Y = rng.integers(0, 256, (n + 24, d)).astype(np.float64)
    elif kind == "sparse":
        Y = rng.standard_normal((n + 24, d)) * (rng.random((n + 24, d)) < 0.3)
        Y[::2] *= -1.0
    else:
        Y = rng.standard_normal((n + 24, d))
        Y[:, ::3] *= 1e-40
    Y = Y.astype(np.float32)
    A = oracle.gen_projection(5, 15, d).astype(np.float32)
    for k in (5, 60):
        _check(Y[:n], Y[n:], A, k)


def test_ties_beyond_k():
    X = np.repeat(datagen.gaussian(300, 24, seed=7), 7, axis=0)   # seven copies of each point
    A = oracle.gen_projection(6, 15, 24).astype(np.float32)
    _check(X, X[:40] + np.float32(0.25), A, 20)
    _check(X, X[:40].copy(), A, 20)


# a warp per query: batches above the block form's limit (16 queries per SM at 32
# coordinates), whole and partial load steps, FP32 rows and the BF16 first pass
@pytest.mark.parametrize("precision", [0, 2, 3])
@pytest.mark.parametrize("d,k", [(20, 10), (32, 40)])
def test_large_batch(d, k, precision):
    X, Q, _, _ = datagen.mixture(1500, d, 6, 1.0, seed=d, nq=64)
    A = oracle.gen_projection(8, 15, d).astype(np.float32)
    _check(X, Q, A, k, copies=80, precision=precision, with_stats=precision != 3)


# squared distances far below and above 1 (at 1e16, above 1e33)
@pytest.mark.parametrize("scale", [1e-6, 1e13, 1e16])
@pytest.mark.parametrize("nq", [2, 130])
def test_scales(scale, nq):
    X, Q, _, _ = datagen.mixture(2503, 24, 2, 4.0, seed=9, nq=nq)
    A = oracle.gen_projection(2, 13, 24).astype(np.float32)
    _check((X * np.float32(scale)).astype(np.float32), (Q * np.float32(scale)).astype(np.float32), A, 3, leaf=100,
           beta=0.9, r_min=25.0 * scale)
