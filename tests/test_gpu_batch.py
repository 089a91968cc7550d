"""Batched V-cycle (hnv_batch_*) against the per-graph V-cycle and the
oracle. Per row, the batched kernels sum the same incidences in the same
order as the single-graph kernels (the order does not depend on lanes per
row, row-class boundaries or the graph's position in the batch), so the
batched results equal the per-graph ones bit for bit."""

import os

import numpy as np
import pytest

import hypergen
from oracle import hnv_oracle as O

from _helpers import FP32_TOL, oracle_level0, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2103_09660_gb300 import build
    build.build()
    import paper_2103_09660_gb300 as mod
    import torch
    assert torch.cuda.is_available()
    return mod


def _graphs(H, count, seed, weighted=True):
    rng = np.random.default_rng(seed)
    hgs, Gs = [], []
    for i in range(count):
        n = int(np.exp(rng.uniform(np.log(200), np.log(6000))))
        hg = hypergen.planted_hypergraph(n, int(0.8 * n), C=8, alpha=2.0, cap=300, p_in=0.8,
                                         weighted=weighted, seed=seed * 1000 + i)
        G = H.Graph.from_hypergraph(hg)
        G.coarsen(min_nodes=max(50, hg.n // 50), seed=i)
        hgs.append(hg)
        Gs.append(G)
    return hgs, Gs


def _run_single(H, G, zc_i, d, dt, sweeps):
    import torch
    n0, m0, _ = G.level_info(0)
    zv = torch.empty((n0, d), dtype=dt, device="cuda")
    ze = torch.empty((m0, d), dtype=dt, device="cuda")
    G.vcycle(zc_i, zv, ze, 0.5, sweeps)
    return zv, ze


@pytest.mark.parametrize("dtname,d", [("f32", 32), ("f32", 64), ("bf16", 64), ("f32", 128)])
def test_batch_equals_per_graph(H, dtname, d):
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hgs, Gs = _graphs(H, 12, seed=3 + d)
    depths = {G.num_levels for G in Gs}
    assert len(depths) > 1            # graphs of different depth in one batch
    with H.Batch(Gs) as B:
        assert B.kernel == H.BATCH_KERNEL_PER_CLASS           # the default
        co, vo, eo = B.offsets()
        zc = torch.randn((int(co[-1]), d), device="cuda").to(dt)
        zv = torch.empty((int(vo[-1]), d), dtype=dt, device="cuda")
        ze = torch.empty((int(eo[-1]), d), dtype=dt, device="cuda")
        # both half-sweep kernels; direct launches, capture, replay, and a
        # switch back to the first kernel (re-capture)
        for kernel, use_graph in ((H.BATCH_KERNEL_PERSISTENT, False),
                                  (H.BATCH_KERNEL_PERSISTENT, True),
                                  (H.BATCH_KERNEL_PERSISTENT, True),
                                  (H.BATCH_KERNEL_PER_CLASS, False),
                                  (H.BATCH_KERNEL_PER_CLASS, True),
                                  (H.BATCH_KERNEL_PERSISTENT, True)):
            B.kernel = kernel
            zv.fill_(float("nan"))
            ze.fill_(float("nan"))
            B.vcycle(zc, zv, ze, 0.5, 4, use_cuda_graph=use_graph)
            torch.cuda.synchronize()
            for G in Gs:
                G.sync_status()          # no work item was out of bounds
            for i, G in enumerate(Gs):
                sv, se = _run_single(H, G, zc[co[i]:co[i + 1]].contiguous(), d, dt, 4)
                assert torch.equal(sv, zv[vo[i]:vo[i + 1]]) and torch.equal(se, ze[eo[i]:eo[i + 1]])
        with pytest.raises(H.HNVError):
            B.kernel = 7
    for G in Gs:
        G.close()


def test_batch_autotune_keeps_results_and_matches_oracle(H):
    import torch
    d = 64
    hgs, Gs = _graphs(H, 10, seed=11)
    with H.Batch(Gs) as B:
        co, vo, eo = B.offsets()
        zc = torch.randn((int(co[-1]), d), device="cuda")
        zv = torch.empty((int(vo[-1]), d), device="cuda")
        ze = torch.empty((int(eo[-1]), d), device="cuda")
        B.vcycle(zc, zv, ze, 0.5, 3)
        before = (zv.clone(), ze.clone())
        t = B.autotune(H.F32, d)
        assert t["a_max"] < t["b_max"] < t["c_max"] and t["lanes_a"] >= 1
        assert t["kernel"] == B.kernel and t["persistent_ms"] > 0 and t["best_ms"] > 0
        assert t["best_ms"] <= t["persistent_ms"]
        B.vcycle(zc, zv, ze, 0.5, 3)
        torch.cuda.synchronize()
        assert torch.equal(before[0], zv) and torch.equal(before[1], ze)
        t2 = B.autotune(H.F32, d)
        assert t2["from_cache"] == 1 and t2["a_max"] == t["a_max"]
        assert t2["kernel"] == t["kernel"] == B.kernel
        # two graphs against the FP64 oracle
        for i in (0, len(Gs) - 1):
            lv0 = oracle_level0(hgs[i])
            h = O.coarsen(lv0, O.CoarsenParams(min_nodes=max(50, hgs[i].n // 50), seed=i))
            ref = O.vcycle(h, zc[co[i]:co[i + 1]].double().cpu().numpy(), 0.5, 3)
            assert rel_err(zv[vo[i]:vo[i + 1]].double().cpu().numpy(), ref.z_v) < FP32_TOL
            assert rel_err(ze[eo[i]:eo[i + 1]].double().cpu().numpy(), ref.z_e) < FP32_TOL
    for G in Gs:
        G.close()


def test_batch_rejects_bad_arguments(H):
    import torch
    hgs, Gs = _graphs(H, 2, seed=5)
    with H.Batch(Gs) as B:
        co, vo, eo = B.offsets()
        zc = torch.zeros((int(co[-1]), 12), device="cuda")
        zv = torch.zeros((int(vo[-1]), 12), device="cuda")
        ze = torch.zeros((int(eo[-1]), 12), device="cuda")
        with pytest.raises(H.HNVError) as ei:
            B.vcycle(zc, zv, ze)
        assert ei.value.code == -7
    for G in Gs:
        G.close()


def _hub_graph(n, hub_edges, seed):
    """A hypergraph whose node 0 is in `hub_edges` hyperedges (a split row of
    many chunks on the node side), plus random small hyperedges."""
    rng = np.random.default_rng(seed)
    edges = [[0, 1 + (i % (n - 2)), 2 + (i % (n - 2))] for i in range(hub_edges)]
    edges += [sorted(rng.choice(np.arange(1, n), 3, replace=False).tolist()) for _ in range(n)]
    ptr = np.concatenate([[0], np.cumsum([len(e) for e in edges])]).astype(np.int64)
    return hypergen.Hypergraph(n=n, m=len(edges), edge_ptr=ptr,
                               edge_nodes=np.concatenate(edges).astype(np.int32),
                               weights=rng.uniform(0.5, 2.0, len(edges)).astype(np.float32))


@pytest.mark.parametrize("dtname,d", [("bf16", 8), ("f32", 1024)])
def test_batch_edge_shapes(H, dtname, d):
    """Width extremes (one 16-byte vector per row; 256 per row), a graph that
    is not coarsened at all next to deeper ones, a node in 9,000 hyperedges
    (split rows with many chunks), zero sweeps and omega = 0 (identity)."""
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hgs = [_hub_graph(3000, 9000, 1),
           hypergen.generate(hypergen.CONFIGS["small_2k"]),
           hypergen.random_small_hypergraph(np.random.default_rng(2), 30, 20, 5)]
    Gs = []
    for i, hg in enumerate(hgs):
        G = H.Graph.from_hypergraph(hg)
        G.coarsen(min_nodes=10 ** 9 if i == 2 else 100, seed=i)   # graph 2: one level
        Gs.append(G)
    assert Gs[2].num_levels == 1 and Gs[0].num_levels > 1
    with H.Batch(Gs) as B:
        co, vo, eo = B.offsets()
        zc = torch.randn((int(co[-1]), d), device="cuda").to(dt)
        zv = torch.empty((int(vo[-1]), d), dtype=dt, device="cuda")
        ze = torch.empty((int(eo[-1]), d), dtype=dt, device="cuda")
        for kernel, omega, sweeps in ((H.BATCH_KERNEL_PERSISTENT, 0.5, 3),
                                      (H.BATCH_KERNEL_PER_CLASS, 0.5, 3),
                                      (H.BATCH_KERNEL_PERSISTENT, 0.5, 0),
                                      (H.BATCH_KERNEL_PERSISTENT, 0.0, 2)):
            B.kernel = kernel
            B.vcycle(zc, zv, ze, omega, sweeps)
            torch.cuda.synchronize()
            for i, G in enumerate(Gs):
                G.sync_status()
                n0, m0, _ = G.level_info(0)
                sv = torch.empty((n0, d), dtype=dt, device="cuda")
                se = torch.empty((m0, d), dtype=dt, device="cuda")
                G.vcycle(zc[co[i]:co[i + 1]].contiguous(), sv, se, omega, sweeps)
                assert torch.equal(sv, zv[vo[i]:vo[i + 1]]) and torch.equal(se, ze[eo[i]:eo[i + 1]])
    for G in Gs:
        G.close()


def test_batch_goes_stale_when_a_graph_is_coarsened_again(H):
    import torch
    hgs, Gs = _graphs(H, 3, seed=9)
    with H.Batch(Gs) as B:
        co, vo, eo = B.offsets()
        zc = torch.zeros((int(co[-1]), 16), device="cuda")
        zv = torch.zeros((int(vo[-1]), 16), device="cuda")
        ze = torch.zeros((int(eo[-1]), 16), device="cuda")
        B.vcycle(zc, zv, ze)
        Gs[1].coarsen(min_nodes=5, seed=1)
        with pytest.raises(H.HNVError) as ei:
            B.vcycle(zc, zv, ze)
        assert ei.value.code == -8
    for G in Gs:
        G.close()


def _buffers(B, d, dt, seed=0):
    import torch
    co, vo, eo = B.offsets()
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    zc = torch.randn((int(co[-1]), d), generator=g, device="cuda").to(dt)
    return zc, torch.empty((int(vo[-1]), d), dtype=dt, device="cuda"), \
        torch.empty((int(eo[-1]), d), dtype=dt, device="cuda")


def _launches(H, f):
    import torch
    before = H.kernel_launch_count()
    f()
    torch.cuda.synchronize()
    return H.kernel_launch_count() - before


# another gather asked for in the environment turns the teams off
needs_teams = pytest.mark.skipif(
    bool(os.environ.get("HNV_PANELS")) or os.environ.get("HNV_GATHER") == "tma",
    reason="no teams with this environment")


class _StepLists:
    """Phase timing selects a launch per half-sweep: every graph in the step
    lists of the batch, and the per-launch path for a single graph."""

    def __init__(self, H):
        self.H = H

    def __enter__(self):
        self.H.timing_enable(True)

    def __exit__(self, *exc):
        self.H.timing_enable(False)
        self.H.timing_reset()


@needs_teams
@pytest.mark.parametrize("dtname,d", [("f32", 8), ("f32", 64), ("bf16", 64), ("bf16", 512)])
def test_teams_and_step_lists_give_the_same_bits(H, dtname, d):
    """Small graphs run by teams in one launch, and lined up in the step lists
    of the per-class kernels (direct, captured, replayed, and with the row
    classes and lanes of the autotuner)."""
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hgs, Gs = _graphs(H, 9, seed=40 + d)
    with H.Batch(Gs) as B:
        zc, zv, ze = _buffers(B, d, dt)

        def run(graph):
            zv.fill_(float("nan"))
            ze.fill_(float("nan"))
            n = _launches(H, lambda: B.vcycle(zc, zv, ze, 0.5, 4, use_cuda_graph=graph))
            for G in Gs:
                G.sync_status()
            return n, zv.clone(), ze.clone()
        want = run(False)
        assert want[0] == 1
        for graph in (True, True):
            got = run(graph)
            assert got[0] == 1 and torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
        for tuned in (False, True):
            if tuned:
                B.autotune(H.F32 if dtname == "f32" else H.BF16, d)
                B.kernel = H.BATCH_KERNEL_PER_CLASS
            for graph in (False, True, True):
                with _StepLists(H):
                    got = run(graph)
                assert got[0] > 8 and torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
        got = run(True)
        assert got[0] == 1 and torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    for G in Gs:
        G.close()


@needs_teams
@pytest.mark.parametrize("dtname,d", [("f32", 256), ("bf16", 512)])
def test_batch_of_teams_and_stepped_graphs(H, dtname, d):
    """One graph too large for a team among small ones; calls of more sweeps
    than a team's launch takes in between, on the same buffers. A caller's
    captured V-cycle stays valid through them (the lists it uses are kept)."""
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hgs, Gs = _graphs(H, 4, seed=7)
    big = hypergen.planted_hypergraph(60_000, 50_000, C=8, alpha=1.8, cap=500, p_in=0.8,
                                      weighted=True, seed=1)
    G = H.Graph.from_hypergraph(big)
    G.coarsen(min_nodes=3000, max_levels=2)
    assert G.level_info(0)[2] * 1024 > 250_000_000
    Gs.insert(2, G)
    with H.Batch(Gs) as B:
        zc, zv, ze = _buffers(B, d, dt)

        def run(sweeps, graph):
            zv.fill_(float("nan"))
            ze.fill_(float("nan"))
            n = _launches(H, lambda: B.vcycle(zc, zv, ze, 0.5, sweeps, use_cuda_graph=graph))
            for G in Gs:
                G.sync_status()
            return n, zv.clone(), ze.clone()
        with _StepLists(H):
            want = {k: run(k, False) for k in (3, 513)}
        own = None
        for k, graph in ((3, False), (3, True), (513, False), (3, False), (513, True), (3, True)):
            got = run(k, graph)
            assert torch.equal(got[1], want[k][1]) and torch.equal(got[2], want[k][2])
            assert (got[0] < want[k][0]) == (k == 3)
            if own is None:
                own = torch.cuda.CUDAGraph()
                s = torch.cuda.Stream()
                s.wait_stream(torch.cuda.current_stream())
                stream, B.stream = B.stream, s
                with torch.cuda.graph(own, stream=s, capture_error_mode="relaxed"):
                    B.vcycle(zc, zv, ze, 0.5, 3, use_cuda_graph=False)
                B.stream = stream
        zv.fill_(float("nan"))
        ze.fill_(float("nan"))
        own.replay()
        torch.cuda.synchronize()
        assert torch.equal(zv, want[3][1]) and torch.equal(ze, want[3][2])
    for G in Gs:
        G.close()


class _Allocator:
    """A device allocator hook that refuses once `left` requests were granted."""

    def __init__(self, H):
        import ctypes
        self.H, self.held, self.left = H, [], None
        AF = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
        FF = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
        self.fns = AF(self._alloc), FF(lambda p, s, ctx: None)
        self.ptrs = [ctypes.cast(f, ctypes.c_void_p) for f in self.fns]

    def _alloc(self, nbytes, s, ctx):
        import torch
        if self.left is not None:
            if self.left == 0:
                return None
            self.left -= 1
        self.held.append(torch.empty(nbytes, dtype=torch.uint8, device="cuda"))
        return self.held[-1].data_ptr()

    def __enter__(self):
        assert self.H.lib().hnv_set_allocator(self.ptrs[0], self.ptrs[1], None) == 0
        return self

    def __exit__(self, *exc):
        import torch
        torch.cuda.synchronize()
        assert self.H.lib().hnv_set_allocator(None, None, None) == 0


@needs_teams
@pytest.mark.parametrize("graph", [False, True])
def test_batch_survives_a_build_that_fails(H, graph):
    """Work lists for another dealing of the graphs (more sweeps than a team's
    launch takes), with the allocator refusing at every point of the build in
    turn: each call fails with HNV_ERR_OOM, the next tries again, and what was
    built before keeps working."""
    import torch
    d = 16
    with _Allocator(H) as hook:
        hgs, Gs = _graphs(H, 3, seed=21)
        with H.Batch(Gs) as B:
            zc, zv, ze = _buffers(B, d, torch.float32)
            B.vcycle(zc, zv, ze, 0.5, 4, use_cuda_graph=graph)
            few = zv.clone(), ze.clone()
            for granted in range(10_000):
                hook.left = granted
                try:
                    B.vcycle(zc, zv, ze, 0.5, 513, use_cuda_graph=graph)
                    break
                except H.HNVError as e:
                    assert e.code == -4
                hook.left = None
                if granted % 16 == 0:
                    B.vcycle(zc, zv, ze, 0.5, 4, use_cuda_graph=graph)
                    assert torch.equal(zv, few[0]) and torch.equal(ze, few[1])
            assert granted > 16
            hook.left = None
            co, vo, eo = B.offsets()
            for i, G in enumerate(Gs):
                G.sync_status()
                sv, se = _run_single(H, G, zc[co[i]:co[i + 1]].contiguous(), d, torch.float32, 513)
                assert torch.equal(sv, zv[vo[i]:vo[i + 1]]) and torch.equal(se, ze[eo[i]:eo[i + 1]])
            B.vcycle(zc, zv, ze, 0.5, 4, use_cuda_graph=graph)
            torch.cuda.synchronize()
            assert torch.equal(zv, few[0]) and torch.equal(ze, few[1])
        for G in Gs:
            G.close()


@needs_teams
def test_autotune_times_the_step_lists(H):
    """The row classes and lanes only matter to graphs in the step lists: they
    are timed there, also for a batch whose graphs the teams run, and what is
    found with the teams is not taken for a batch without them."""
    import torch
    d = 32
    hgs, Gs = _graphs(H, 7, seed=77)
    with H.Batch(Gs) as B:
        zc, zv, ze = _buffers(B, d, torch.float32)
        launches = []

        def one():
            launches.append(_launches(H, lambda: B.vcycle(zc, zv, ze, 0.5, 1)))
            return zv.clone(), ze.clone()
        want = one()
        one()
        tuned = {}
        n = _launches(H, lambda: tuned.update(B.autotune(H.F32, d)))
        assert tuned["from_cache"] == 0
        with _StepLists(H):
            B.kernel = H.BATCH_KERNEL_PER_CLASS
            one()                                        # (builds the lists)
            got = one()
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
            t = B.autotune(H.F32, d)
            assert t["from_cache"] == 0                  # no graph goes to the teams now
            assert B.autotune(H.F32, d)["from_cache"] == 1
        t = B.autotune(H.F32, d)
        assert t["from_cache"] == 1 and t["kernel"] == tuned["kernel"] == B.kernel
        # 4 timed V-cycles of each candidate (18 at this width)
        assert launches[1] == 1 and n > 4 * 18 * launches[3]
    for G in Gs:
        G.close()
