"""Per-point range count on the CUDA cores (a warp per leaf, points in packed pairs)
at the sizes where it can go wrong, against the FP64 oracle: |C|, rounds and stop
rule equal for every query."""
import math

import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2107_05537_gb300 as pm  # noqa: E402


# leaves below, at and past 32, 64 and 128 points; one query, a block of 64, and one
# more than several blocks; radii that cut through the leaves
@pytest.mark.parametrize("leaf", [16, 32, 64, 129, 1024])
@pytest.mark.parametrize("nq", [1, 64, 193])
def test_counts_by_leaf_size(leaf, nq):
    X, Q, _, _ = datagen.mixture(2600, 24, 2, 4.0, seed=leaf, nq=nq)
    A = oracle.gen_projection(2, 13, 24).astype(np.float32)
    t, _, _ = oracle.params(13, 1.5, 1 / math.e)
    ix = pm.Index(torch.from_numpy(X).cuda(), m=13, leaf_size=leaf, proj=A)
    for r in (3.0, 12.0, 25.0):
        got = ix.knn(torch.from_numpy(Q).cuda(), k=3, beta=0.9, r_min=r, t=t)
        ref = oracle.knn(X, A, Q, 3, 1.5, t, oracle.budget(len(X), 0.9, 3), r, 0)
        assert np.array_equal(got["ids"].cpu().numpy(), ref["ids"])
        for f in ("ncand", "rounds", "rule"):
            assert np.array_equal(got["stats"][f], ref[f])
    ix.close()


# the same far from the origin, where norms dwarf the distances, and at scales whose
# squared norms are tiny or too large for the expanded form; a last leaf of few points
@pytest.mark.parametrize("scale,offset", [(1.0, 1000.0), (1.0, -40.0), (1e-6, 0.0), (1e16, 0.0)])
@pytest.mark.parametrize("nq", [2, 130])
def test_counts_by_scale_and_offset(scale, offset, nq):
    X, Q, _, _ = datagen.mixture(2500 + 3, 24, 2, 4.0, seed=9, nq=nq)
    X = ((X + np.float32(offset)) * np.float32(scale)).astype(np.float32)
    Q = ((Q + np.float32(offset)) * np.float32(scale)).astype(np.float32)
    A = oracle.gen_projection(2, 13, 24).astype(np.float32)
    t, _, _ = oracle.params(13, 1.5, 1 / math.e)
    ix = pm.Index(torch.from_numpy(X).cuda(), m=13, leaf_size=100, proj=A)
    for r in (3.0 * scale, 12.0 * scale, 25.0 * scale):
        got = ix.knn(torch.from_numpy(Q).cuda(), k=3, beta=0.9, r_min=r, t=t, precision=pm.PMLSH_FP32_PLAIN)
        ref = oracle.knn(X, A, Q, 3, 1.5, t, oracle.budget(len(X), 0.9, 3), r, 0)
        assert np.array_equal(got["ids"].cpu().numpy(), ref["ids"])
        for f in ("ncand", "rounds", "rule"):
            assert np.array_equal(got["stats"][f], ref[f])
    ix.close()


# tensor cores: one M-tile, exactly one, and two of them per leaf (128 queries each), as
# well as leaves that alternate between the two; leaves below, at and past a tile of
# 128 points.  Every query of a tight bundle covers the same leaves partially.
@pytest.mark.parametrize("leaf", [16, 128, 129, 600])
@pytest.mark.parametrize("nq", [1, 127, 128, 129, 256, 257, 400])
def test_tensor_counts_by_queries_per_leaf(leaf, nq):
    X, Q, _, _ = datagen.mixture(2600, 24, 2, 4.0, seed=leaf, nq=nq)
    rng = np.random.default_rng(nq)
    Q[: (nq + 1) // 2] = Q[0] + rng.standard_normal(((nq + 1) // 2, 24)).astype(np.float32) * np.float32(0.01)
    A = oracle.gen_projection(2, 13, 24).astype(np.float32)
    t, _, _ = oracle.params(13, 1.5, 1 / math.e)
    ix = pm.Index(torch.from_numpy(X).cuda(), m=13, leaf_size=leaf, proj=A)
    for r in (3.0, 12.0, 25.0):
        got = ix.knn(torch.from_numpy(Q).cuda(), k=3, beta=0.9, r_min=r, t=t, precision=pm.PMLSH_BF16_TENSOR)
        ref = oracle.knn(X, A, Q, 3, 1.5, t, oracle.budget(len(X), 0.9, 3), r, 0)
        assert np.array_equal(got["ids"].cpu().numpy(), ref["ids"])
        for f in ("ncand", "rounds", "rule"):
            assert np.array_equal(got["stats"][f], ref[f])
    ix.close()


# points around the place of the leaf test's stand-in for queries beyond the batch
# (+1e18 on every coordinate): a block's absent queries take part in nothing
@pytest.mark.parametrize("nq", [3, 65, 300])
@pytest.mark.parametrize("precision", [pm.PMLSH_FP32_PLAIN, pm.PMLSH_BF16_TENSOR])
def test_points_at_the_absent_queries(nq, precision):
    rng = np.random.default_rng(5)
    X = (1e18 + 1e16 * rng.standard_normal((2500, 15))).astype(np.float32)
    Q = (1e18 + 1e16 * rng.standard_normal((nq, 15))).astype(np.float32)
    A = np.eye(15, dtype=np.float32)
    t, _, _ = oracle.params(15, 1.5, 1 / math.e)
    ix = pm.Index(torch.from_numpy(X).cuda(), leaf_size=64, proj=A)
    for r in (1e16, 2e16):
        got = ix.knn(torch.from_numpy(Q).cuda(), k=3, beta=0.9, r_min=r, t=t, precision=precision)
        ref = oracle.knn(X, A, Q, 3, 1.5, t, oracle.budget(len(X), 0.9, 3), r, 0)
        assert np.array_equal(got["ids"].cpu().numpy(), ref["ids"])
        for f in ("ncand", "rounds", "rule"):
            assert np.array_equal(got["stats"][f], ref[f])
    ix.close()
