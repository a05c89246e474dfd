"""Closest-pair kernels at the sizes where their tiling can go wrong, against
the FP64 oracle (pairs equal, distances the rounded FP64 values: exact, since
FP32 values only choose which pairs are recomputed in FP64)."""
import math

import numpy as np
import pytest

import datagen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2107_05537_gb300 as pm  # noqa: E402


def _check(X, A, k, gamma, T, leaf):
    ix = pm.Index(torch.from_numpy(X).cuda(), m=A.shape[0], leaf_size=leaf, proj=A)
    t, _, _ = oracle.params(A.shape[0], 1.5, 1 / math.e)
    got = ix.closest_pairs(k=k, gamma=gamma, T=T, t=t)
    lay = ix.layout()
    ix.close()
    ref = oracle.cp_radius_filter(X, A, lay, k, t, gamma, T)
    assert got["pairs"].tolist() == ref["pairs"].tolist()
    assert np.array_equal(got["dists"], ref["dists"].astype(np.float32))
    for f, g in (("count", "count"), ("lca_nodes", "nodes"), ("nodes_done", "nodes_done")):
        assert got["stats"][f] == ref[g]
    return got


# rows of 1 to 9 steps of 32 coordinates: below, at and past a four-step round
@pytest.mark.parametrize("d", [1, 31, 33, 96, 97, 128, 129, 257])
def test_pair_distance_row_lengths(d):
    X, _, _, _ = datagen.mixture(700, d, 7, 1.0, seed=d)
    A = oracle.gen_projection(3, 15, d).astype(np.float32)
    _check(X, A, 9, 2.0, 10 ** 9, 16)


# nodes of one tile of 64 x 64 positions, at its edges and of several tiles;
# one cluster makes one large node
@pytest.mark.parametrize("n,clusters,leaf,k,gamma,T", [
    (64, 1, 16, 3, math.inf, 10 ** 9),
    (65, 1, 16, 3, math.inf, 10 ** 9),
    (129, 1, 16, 3, math.inf, 10 ** 9),
    (1000, 9, 16, 12, 1.4, 10 ** 9),
    (1000, 9, 16, 400, 1.4, 10 ** 9),    # ub is infinite at the start: fewer self pairs than k
    (1000, 9, 32, 12, 3.0, 6000),        # the budget cut inside a node
    (6000, 40, 16, 1000, 2.5, 10 ** 9),  # many nodes, ub falls often
])
def test_node_tiles_and_replay(n, clusters, leaf, k, gamma, T):
    X, _, _, _ = datagen.mixture(n, 20, clusters, 1.0, seed=n + k)
    A = oracle.gen_projection(4, 15, 20).astype(np.float32)
    _check(X, A, k, gamma, T, leaf)


def test_more_entrants_than_the_list_holds():
    # the ten self pairs that set ub are farther apart than most of the pairs
    # between leaves, so one ub admits more than 4,096 of them
    rng = np.random.default_rng(3)
    X = rng.standard_normal((900, 6)).astype(np.float32)
    A = oracle.gen_projection(4, 6, 6).astype(np.float32)
    _check(X, A, 1024, math.inf, 10 ** 9, 16)


def _bnb(X, A, k, T, leaf):
    ix = pm.Index(torch.from_numpy(X).cuda(), m=A.shape[0], leaf_size=leaf, proj=A)
    got = ix.closest_pairs_bnb(k=k, T=T)
    ix.close()
    rp, rd = oracle.cp_bnb(X, A, T, k)[:2]
    return got, np.asarray(rp), np.asarray(rd)


# leaf counts around the 128 x 32 tiles of Mindist; T below, at and above the self
# pairs (a first cut, none, cuts in the batches)
@pytest.mark.parametrize("n,clusters,leaf,T", [
    (40, 2, 16, 30), (300, 5, 16, 200), (700, 3, 16, 1500), (1500, 6, 16, 4000), (1500, 6, 128, 4000),
])
def test_branch_and_bound_tiles(n, clusters, leaf, T):
    X, _, _, _ = datagen.mixture(n, 10, clusters, 1.0, seed=n)
    A = oracle.gen_projection(6, 15, 10).astype(np.float32)
    got, rp, rd = _bnb(X, A, 12, T, leaf)
    assert got["pairs"].tolist() == rp.tolist()
    assert np.array_equal(got["dists"], rd.astype(np.float32))
    assert got["stats"]["count"] == T


# the FP32 window around the wanted rank, and the data that leave it: equal ratios by
# the thousand (copies, a grid), ranks at both ends
@pytest.mark.parametrize("kind", ["mixture", "copies", "grid", "line"])
@pytest.mark.parametrize("pr", [1e-9, 0.02, 0.5, 0.85, 1.0])
def test_gamma_rank(kind, pr):
    if kind == "mixture":
        X, _, _, _ = datagen.mixture(900, 12, 9, 1.0, seed=3)
    elif kind == "copies":
        X = np.repeat(datagen.gaussian(60, 12, seed=5), 15, axis=0)
    elif kind == "grid":
        X = np.stack(np.meshgrid(*[np.arange(6.0)] * 3), -1).reshape(-1, 3).astype(np.float32)
        X = np.concatenate([X, np.zeros((len(X), 9), np.float32)], 1)
    else:
        X = np.zeros((700, 12), np.float32)
        X[:, 0] = 2.0 ** np.arange(700).clip(0, 60) + np.arange(700)
    A = oracle.gen_projection(2, 15, 12).astype(np.float32)
    ix = pm.Index(torch.from_numpy(X).cuda(), leaf_size=16, proj=A)
    got = ix.gamma_calibrate(pr=pr)
    ref = oracle.gamma_calibrate(ix.projected(), ix.layout(), pr)
    ix.close()
    assert got == ref or (math.isinf(got) and math.isinf(ref))
