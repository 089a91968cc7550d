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


def test_build_with_an_allocator_of_small_blocks(H):
    """An allocator hook that grants no request above 64 KB: the temporaries of
    a small graph, which share slabs where those can be had, need no more."""
    import ctypes
    import torch
    held, refused = [], []

    def alloc(nbytes, s, ctx):
        if nbytes > 65536:
            refused.append(nbytes)
            return None
        held.append(torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
        return held[-1].data_ptr()
    AF = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
    FF = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
    fns = AF(alloc), FF(lambda p, s, ctx: None)
    hg = hypergen.random_small_hypergraph(np.random.default_rng(3), 200, 150, 6)
    X = np.random.default_rng(4).standard_normal((200, 5)).astype(np.float32)
    assert H.lib().hnv_set_allocator(*[ctypes.cast(f, ctypes.c_void_p) for f in fns], None) == 0
    try:
        for policy in (O.ASSIGN_HASH, O.ASSIGN_COSINE):
            h = O.coarsen(oracle_level0(hg), O.CoarsenParams(
                policy=policy, features=X if policy == O.ASSIGN_COSINE else None, min_nodes=5,
                max_levels=4, seed=1))
            with H.Graph.from_hypergraph(hg) as G:
                if policy == O.ASSIGN_COSINE:
                    G.set_node_features(X)
                G.coarsen(policy=policy, min_nodes=5, max_levels=4, seed=1)
                assert_hierarchy_equal(G, h)
        torch.cuda.synchronize()
    finally:
        assert H.lib().hnv_set_allocator(None, None, None) == 0
    assert set(refused) == {512 * 1024}          # slabs only
