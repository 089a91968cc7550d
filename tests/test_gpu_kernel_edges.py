"""Sizes at the edges of the coarsening kernels' tiles and dispatch rules,
bit-exact against the oracle: entry tiles (2,048), compaction tiles and the
one-block radix sort (4,096), rows that change the assignment kernel (256 and
1,024 incidences, 16,384 for rows cut into parts), and member lists around the
mean kernels' bounds (64) and tiles (128)."""

import numpy as np
import pytest

import hypergen
from oracle import hnv_oracle as O

from _helpers import assert_hierarchy_equal, oracle_level0

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2103_09660_gb300 import build
    build.build()
    import paper_2103_09660_gb300 as mod
    import torch
    assert torch.cuda.is_available()
    return mod


def _hypergraph(n, edges, seed=0):
    rng = np.random.default_rng(seed)
    ptr = np.concatenate([[0], np.cumsum([len(e) for e in edges])]).astype(np.int64)
    return hypergen.Hypergraph(n=n, m=len(edges), edge_ptr=ptr,
                               edge_nodes=np.concatenate(edges).astype(np.int32),
                               weights=rng.uniform(0.5, 2.0, len(edges)).astype(np.float32))


@pytest.mark.parametrize("nnz", [1, 31, 2047, 2048, 2049, 4095, 4096, 4097, 8193])
def test_entry_and_compaction_tiles(H, nnz):
    """nnz incidences in hyperedges of 1-3 members, one of them long."""
    rng = np.random.default_rng(nnz)
    n, edges, left = 500, [], nnz
    if nnz > 1000:
        edges.append(rng.integers(0, n, 700))         # repeats, removed by the build
        left -= 700
    while left > 0:
        k = min(left, int(rng.integers(1, 4)))
        edges.append(rng.choice(n, k, replace=False))
        left -= k
    hg = _hypergraph(n, edges, nnz)
    for policy in (O.ASSIGN_HASH, O.ASSIGN_HIGH_WEIGHT):
        h = O.coarsen(oracle_level0(hg), O.CoarsenParams(policy=policy, min_nodes=2, max_levels=4,
                                                         seed=nnz))
        with H.Graph.from_hypergraph(hg) as G:
            G.coarsen(policy=policy, min_nodes=2, max_levels=4, seed=nnz)
            assert_hierarchy_equal(G, h)


@pytest.mark.parametrize("hub", [256, 257, 1024, 1025, 4097, 16384, 16385, 40000])
@pytest.mark.parametrize("dense", [False, True])
def test_hub_rows(H, hub, dense):
    """Node 0 in `hub` hyperedges, among nodes of few (8 lanes per node) or
    many (32 lanes) incidences."""
    rng = np.random.default_rng(hub)
    n = 60 if dense else 30000
    a = rng.integers(1, n, (hub, 2))
    edges = [[0, int(x), int(y)] for x, y in a]
    hg = _hypergraph(n, edges, hub)
    h = O.coarsen(oracle_level0(hg), O.CoarsenParams(min_nodes=2, max_levels=2, seed=hub))
    with H.Graph.from_hypergraph(hg) as G:
        G.coarsen(min_nodes=2, max_levels=2, seed=hub)
        assert_hierarchy_equal(G, h)


@pytest.mark.parametrize("k", [1, 31, 32, 33, 65])
def test_means_and_cosines(H, k):
    """Hyperedges of 63 .. 385 members (means, and coarse nodes that merge as
    many nodes), feature widths around the 32-wide slabs."""
    rng = np.random.default_rng(k)
    n = 3000
    edges = [rng.choice(n, s, replace=False) for s in (63, 64, 65, 127, 128, 129, 256, 257, 384, 385)]
    edges += [rng.choice(n, 3, replace=False) for _ in range(40)]
    hg = _hypergraph(n, edges, k)
    X = rng.standard_normal((n, k)).astype(np.float32)
    kw = dict(min_nodes=2, max_levels=2, seed=k)
    h = O.coarsen(oracle_level0(hg), O.CoarsenParams(policy=O.ASSIGN_COSINE, features=X, **kw))
    with H.Graph.from_hypergraph(hg) as G:
        G.set_node_features(X)
        G.coarsen(policy=H.ASSIGN_COSINE, **kw)
        assert_hierarchy_equal(G, h)
        for ell, F in enumerate(h.features):
            np.testing.assert_array_equal(G.level_features(ell), F)
