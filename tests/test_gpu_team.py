"""Small graphs run whole V-cycles in one cooperative launch (team.cu). Every
row is summed in the order of the per-launch kernels, so both paths give the
same bits. Phase timing needs a launch per half-sweep and so selects the
per-launch path; a graph that is too large for the one-launch path takes it as
well."""

import numpy as np
import pytest

import hypergen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    from paper_2103_09660_gb300 import build
    build.build()
    import paper_2103_09660_gb300 as mod
    import torch
    assert torch.cuda.is_available()
    return mod


def _hub_graph(hub, mids, seed=0):
    """Node 0 in `hub` hyperedges, nodes 1.. in `mids` each, and hyperedges of
    4, 5, 16, 17, 64, 65, 128, 129 and 300 members."""
    rng = np.random.default_rng(seed)
    n = 700
    edges = [[0, 20 + i % 600, 21 + i % 600] for i in range(hub)]
    for v, k in enumerate(mids):
        edges += [[v + 1, 20 + (7 * i) % 600, 640 + i % 50] for i in range(k)]
    edges += [rng.choice(n, k, replace=False).tolist() for k in (4, 5, 16, 17, 64, 65, 128, 129, 300)]
    ptr = np.concatenate([[0], np.cumsum([len(e) for e in edges])]).astype(np.int64)
    return hypergen.Hypergraph(n=n, m=len(edges), edge_ptr=ptr,
                               edge_nodes=np.concatenate(edges).astype(np.int32),
                               weights=rng.uniform(0.5, 2.0, len(edges)).astype(np.float32))


def _both(H, f):
    """f() on the one-launch path and on the per-launch path."""
    import torch
    before = H.kernel_launch_count()
    a = f()
    torch.cuda.synchronize()
    one = H.kernel_launch_count() - before
    H.timing_enable(True)
    try:
        before = H.kernel_launch_count()
        b = f()
        torch.cuda.synchronize()
        many = H.kernel_launch_count() - before
    finally:
        H.timing_enable(False)
        H.timing_reset()
    return a, b, one, many


# split rows: none; a few of 2-3 chunks (summed inside a block); many chunks
# (more than 32, a reduction step); and rows of both kinds
GRAPHS = [(40, []), (40, [129, 300]), (4200, []), (5000, [129, 300, 4096, 1000])]


@pytest.mark.parametrize("hub,mids", GRAPHS)
@pytest.mark.parametrize("dtname,d", [("f32", 4), ("f32", 36), ("f32", 100), ("f32", 256),
                                      ("bf16", 8), ("bf16", 72), ("bf16", 512)])
def test_one_launch_gives_the_same_bits(H, hub, mids, dtname, d):
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hg = _hub_graph(hub, mids)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    with H.Graph.from_hypergraph(hg) as G:
        L = G.coarsen(min_nodes=30, max_levels=3)
        top = G.level_info(L - 1)
        zc = torch.randn((top[0] + top[1], d), generator=g, device="cuda").to(dt)
        zv = torch.empty((hg.n, d), dtype=dt, device="cuda")
        ze = torch.empty((hg.m, d), dtype=dt, device="cuda")
        z0v = torch.randn((hg.n, d), generator=g, device="cuda").to(dt)
        z0e = torch.randn((hg.m, d), generator=g, device="cuda").to(dt)
        for omega in (0.3, 1.0):
            def vcycle():
                zv.fill_(float("nan"))
                ze.fill_(float("nan"))
                G.vcycle(zc, zv, ze, omega, 3)
                return zv.clone(), ze.clone()
            a, b, one, many = _both(H, vcycle)
            assert one == 1 and many > one
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
            for mode in (H.SWEEP_TWO_PHASE, H.SWEEP_JACOBI):
                def refine():
                    v, e = z0v.clone(), z0e.clone()
                    G.refine(0, v, e, omega, 3, mode)
                    return v, e
                a, b, one, many = _both(H, refine)
                assert one == 1 and many > one
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])

                def until():
                    v, e = z0v.clone(), z0e.clone()
                    return v, e, G.refine_until(0, v, e, omega, 12, 0.2, mode)
                a, b, one, many = _both(H, until)
                assert one == 1 and many > one
                assert a[2] == b[2]
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        G.sync_status()


def test_more_sweeps_than_one_launch_takes(H):
    """The stopping rule over several launches; a fixed number of sweeps above
    the limit takes the per-launch path."""
    import torch
    hg = _hub_graph(40, [129])
    with H.Graph.from_hypergraph(hg) as G:
        z = torch.randn((hg.n + hg.m, 8), device="cuda")

        def until():
            v, e = z[:hg.n].clone(), z[hg.n:].clone()
            return v, e, G.refine_until(0, v, e, 0.001, 1100, -1.0)
        a, b, one, many = _both(H, until)
        assert one == 3 and a[2] == b[2] and a[2][0] == 1100
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])

        def refine():
            v, e = z[:hg.n].clone(), z[hg.n:].clone()
            G.refine(0, v, e, 0.001, 513)
            return v, e
        a, b, one, many = _both(H, refine)
        assert one == many
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_saved_rows_gradients_and_capture(H):
    """The differentiable V-cycle saves every level's starting rows in the same
    launch; a captured V-cycle replays it."""
    import torch
    hg = _hub_graph(300, [129, 300])
    d = 32
    with H.Graph.from_hypergraph(hg) as G:
        L = G.coarsen(min_nodes=30, max_levels=3)
        top = G.level_info(L - 1)
        zc = torch.randn((top[0] + top[1], d), device="cuda")
        w = torch.rand(hg.m, device="cuda") + 0.5

        def grads():
            ww, zz = w.clone().requires_grad_(True), zc.clone().requires_grad_(True)
            v, e = H.vcycle_autograd(G, ww, zz, 0.5, 3)
            return (v.detach(), e.detach()) + torch.autograd.grad(v.square().sum() + e.sum(), [ww, zz])
        a, b, one, many = _both(H, grads)
        assert one < many
        assert all(torch.equal(x, y) for x, y in zip(a, b))

        zv, ze = torch.empty((hg.n, d), device="cuda"), torch.empty((hg.m, d), device="cuda")
        G.vcycle(zc, zv, ze, 0.5, 3)
        want = zv.clone(), ze.clone()
        graph = torch.cuda.CUDAGraph()
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(graph, stream=s):
            H.hnv_vcycle(G.handle, zc, zv, ze, 0.5, 3, H.SWEEP_TWO_PHASE, s)
        zv.zero_()
        ze.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(zv, want[0]) and torch.equal(ze, want[1])


def test_two_streams_on_one_graph(H):
    """Calls on two streams may run beside each other (no split rows, so they
    share no scratch): each launch has its own barrier words."""
    import torch
    hg = _hub_graph(40, [])
    keep = [e for e in range(hg.m) if hg.edge_ptr[e + 1] - hg.edge_ptr[e] <= 128]
    edges = [hg.edge_nodes[hg.edge_ptr[e]:hg.edge_ptr[e + 1]] for e in keep]
    ptr = np.concatenate([[0], np.cumsum([len(e) for e in edges])]).astype(np.int64)
    with H.Graph(hg.n, len(edges), ptr, np.concatenate(edges).astype(np.int32)) as G:
        z = torch.randn((2, hg.n + len(edges), 16), device="cuda")

        def run(k, stream):
            v, e = z[k, :hg.n].clone(), z[k, hg.n:].clone()
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                H.hnv_refine(G.handle, 0, v, e, 0.3, 400, H.SWEEP_TWO_PHASE, stream)
            return v, e
        s = [torch.cuda.Stream(), torch.cuda.Stream()]
        want = []
        for k in range(2):
            want.append(run(k, s[0]))
            torch.cuda.synchronize()
        pairs = [(z[k, :hg.n].clone(), z[k, hg.n:].clone()) for k in range(2)]
        torch.cuda.synchronize()
        for k in range(2):
            H.hnv_refine(G.handle, 0, pairs[k][0], pairs[k][1], 0.3, 400, H.SWEEP_TWO_PHASE, s[k])
        torch.cuda.synchronize()
        G.sync_status()
        for k in range(2):
            assert torch.equal(pairs[k][0], want[k][0]) and torch.equal(pairs[k][1], want[k][1])


@pytest.mark.parametrize("dtname,d", [("f32", 36), ("bf16", 72)])
def test_refused_launch_takes_the_per_launch_path(H, dtname, d):
    """Where the device refuses the cooperative launch, every entry point that
    would use it runs a launch per half-sweep instead and gives the same bits."""
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    hg = _hub_graph(4200, [129, 300])
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    with H.Graph.from_hypergraph(hg) as G:
        L = G.coarsen(min_nodes=30, max_levels=3)
        top = G.level_info(L - 1)
        zc = torch.randn((top[0] + top[1], d), generator=g, device="cuda").to(dt)
        zv, ze = torch.empty((hg.n, d), dtype=dt, device="cuda"), \
            torch.empty((hg.m, d), dtype=dt, device="cuda")
        z = torch.randn((hg.n + hg.m, d), generator=g, device="cuda").to(dt)

        def work():
            out, n = [], []

            def call(f):
                before = H.kernel_launch_count()
                out.extend(f())
                torch.cuda.synchronize()
                n.append(H.kernel_launch_count() - before)

            def vcycle():
                zv.fill_(float("nan"))
                ze.fill_(float("nan"))
                G.vcycle(zc, zv, ze, 0.3, 3)
                return zv.clone(), ze.clone()
            call(vcycle)
            for mode in (H.SWEEP_TWO_PHASE, H.SWEEP_JACOBI):
                def refine():
                    v, e = z[:hg.n].clone(), z[hg.n:].clone()
                    G.refine(0, v, e, 0.3, 3, mode)
                    return v, e

                def until():
                    v, e = z[:hg.n].clone(), z[hg.n:].clone()
                    return (v, e) + tuple(G.refine_until(0, v, e, 0.3, 12, 0.2, mode))
                call(refine)
                call(until)
            G.sync_status()
            return out, n

        def batch(graph):
            zv.fill_(float("nan"))
            ze.fill_(float("nan"))
            before = H.kernel_launch_count()
            B.vcycle(zc, zv, ze, 0.3, 3, use_cuda_graph=graph)
            torch.cuda.synchronize()
            return zv.clone(), ze.clone(), H.kernel_launch_count() - before
        want, one = work()
        assert one == [1] * 5
        assert H.lib().hnv_selftest_team_refuse(G.handle, 1) == 0
        got, many = work()
        assert all(k > 1 for k in many)
        same = lambda a, b: torch.equal(a, b) if torch.is_tensor(a) else a == b
        assert all(same(a, b) for a, b in zip(got, want))
        for graph in (False, True):
            if d % 8:
                break
            with H.Batch([G]) as B:
                first = batch(graph)
                again = batch(graph)
                assert first[2] > again[2] > 1           # the first call builds the lists
                for r in (first, again):
                    assert torch.equal(r[0], want[0]) and torch.equal(r[1], want[1])
            with H.Batch([G]) as B:                      # the tuner meets it first
                assert B.autotune(H.BF16, d)["lanes_a"] > 0
                r = batch(graph)
                assert torch.equal(r[0], want[0]) and torch.equal(r[1], want[1])
        assert H.lib().hnv_selftest_team_refuse(G.handle, 0) == 0
        got, back = work()
        assert back == one and all(same(a, b) for a, b in zip(got, want))
        assert H.lib().hnv_selftest_team_refuse(None, 1) == -1


class _Refuser:
    """A device allocator hook that grants nothing and counts the requests."""

    def __init__(self, H):
        import ctypes
        self.H, self.calls = H, []
        AF = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
        FF = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)
        self.fns = AF(lambda n, s, ctx: self.calls.append(n)), \
            FF(lambda p, s, ctx: self.calls.append(-1))
        self.ptrs = [ctypes.cast(f, ctypes.c_void_p) for f in self.fns]

    def __enter__(self):
        assert self.H.lib().hnv_set_allocator(self.ptrs[0], self.ptrs[1], None) == 0
        return self

    def __exit__(self, *exc):
        assert self.H.lib().hnv_set_allocator(None, None, None) == 0


def test_warmed_calls_allocate_nothing(H):
    """After the first call of its kind (which may allocate scratch), refining a
    small level asks the allocator for nothing, also under capture: a captured
    call then owns everything that its replays use."""
    import torch
    hg = _hub_graph(4200, [129, 300])
    with H.Graph.from_hypergraph(hg) as G:
        z = torch.randn((hg.n + hg.m, 36), device="cuda")

        def calls():
            out = []
            for mode in (H.SWEEP_TWO_PHASE, H.SWEEP_JACOBI):
                v, e = z[:hg.n].clone(), z[hg.n:].clone()
                G.refine(0, v, e, 0.3, 3, mode)
                out += [v, e]
                v, e = z[:hg.n].clone(), z[hg.n:].clone()
                G.refine_until(0, v, e, 0.3, 3, -1.0, mode)
                out += [v, e]
            return out
        want = calls()
        v, e = z[:hg.n].clone(), z[hg.n:].clone()
        graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with _Refuser(H) as hook:
            got = calls()
            with torch.cuda.graph(graph, stream=s):
                H.hnv_refine(G.handle, 0, v, e, 0.3, 3, H.SWEEP_TWO_PHASE, s)
            assert hook.calls == []
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        for _ in range(2):
            v.copy_(z[:hg.n])
            e.copy_(z[hg.n:])
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(v, want[0]) and torch.equal(e, want[1])


def _rows_up_to_128():
    """A hypergraph without split rows (calls on it share no scratch)."""
    hg = _hub_graph(40, [])
    edges = [hg.edge_nodes[hg.edge_ptr[e]:hg.edge_ptr[e + 1]] for e in range(hg.m)
             if hg.edge_ptr[e + 1] - hg.edge_ptr[e] <= 128]
    ptr = np.concatenate([[0], np.cumsum([len(e) for e in edges])]).astype(np.int64)
    return hg.n, len(edges), ptr, np.concatenate(edges).astype(np.int32)


def test_more_streams_than_sets_of_barrier_words(H):
    """Launches on 20 streams, three rounds of them: a set of words that goes to
    another stream is free by then."""
    import torch
    n, m, ptr, nodes = _rows_up_to_128()
    with H.Graph(n, m, ptr, nodes) as G:
        z = torch.randn((20, n + m, 16), device="cuda")

        def fresh():
            return [(z[k, :n].clone(), z[k, n:].clone()) for k in range(20)]
        want = fresh()
        for v, e in want:
            G.refine(0, v, e, 0.3, 60)
        got = fresh()
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(20)]
        for _ in range(3):
            for s, (v, e) in zip(streams, got):
                H.hnv_refine(G.handle, 0, v, e, 0.3, 20, H.SWEEP_TWO_PHASE, s)
        torch.cuda.synchronize()
        G.sync_status()
        for a, b in zip(got, want):
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_more_captures_than_sets_of_barrier_words(H):
    """Every captured branch has a set of its own; when none is left a capture
    takes the per-launch path. All replay beside each other."""
    import torch
    n, m, ptr, nodes = _rows_up_to_128()
    with H.Graph(n, m, ptr, nodes) as G:
        z = torch.randn((60, n + m, 16), device="cuda")
        want = [(z[k, :n].clone(), z[k, n:].clone()) for k in range(60)]
        for v, e in want:
            G.refine(0, v, e, 0.3, 20)
        got = [(z[k, :n].clone(), z[k, n:].clone()) for k in range(60)]
        torch.cuda.synchronize()
        graphs, launches = [], []
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        for k in range(0, 60, 2):
            graphs.append(torch.cuda.CUDAGraph())
            before = H.kernel_launch_count()
            with torch.cuda.graph(graphs[-1], stream=a):
                b.wait_stream(a)
                H.hnv_refine(G.handle, 0, *got[k], 0.3, 20, H.SWEEP_TWO_PHASE, a)
                H.hnv_refine(G.handle, 0, *got[k + 1], 0.3, 20, H.SWEEP_TWO_PHASE, b)
                a.wait_stream(b)
            launches.append(H.kernel_launch_count() - before)
        assert launches[0] == 2 and launches[-1] > 2
        streams = [torch.cuda.Stream() for _ in graphs]
        for s, g in zip(streams, graphs):
            with torch.cuda.stream(s):
                g.replay()
        torch.cuda.synchronize()
        G.sync_status()
        for x, y in zip(got, want):
            assert torch.equal(x[0], y[0]) and torch.equal(x[1], y[1])


def test_first_call_on_a_hierarchy_does_not_wait(H):
    """The first call on a new hierarchy is asynchronous like the others: it
    returns while the stream is still busy with earlier work."""
    import torch
    hg = _hub_graph(300, [])
    d = 32
    s = torch.cuda.Stream()

    def once(busy):
        with H.Graph.from_hypergraph(hg) as G:
            L = G.coarsen(min_nodes=30, max_levels=3)
            top = G.level_info(L - 1)
            g = torch.Generator(device="cuda")
            g.manual_seed(1)
            zc = torch.randn((top[0] + top[1], d), generator=g, device="cuda")
            zv, ze = torch.empty((hg.n, d), device="cuda"), torch.empty((hg.m, d), device="cuda")
            torch.cuda.synchronize()
            done = torch.cuda.Event()
            with torch.cuda.stream(s):
                if busy:
                    torch.cuda._sleep(600_000_000)       # about 0.3 s
                done.record()
            H.hnv_vcycle(G.handle, zc, zv, ze, 0.5, 3, H.SWEEP_TWO_PHASE, s)
            early = not done.query()
            torch.cuda.synchronize()
            return early, zv, ze
    want = once(False)                                   # (loads the kernels)
    got = once(True)
    assert got[0]
    assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])


@pytest.mark.parametrize("mode", ["two_phase", "jacobi"])
@pytest.mark.parametrize("warm", [False, True])
def test_captured_calls_keep_their_scratch(H, mode, warm):
    """A graph's scratch grows with the row size. A capture that has to grow it
    takes memory of its own (what it allocates is valid in its replays only),
    and scratch that a capture uses outlives later growth."""
    import torch
    mode = H.SWEEP_JACOBI if mode == "jacobi" else H.SWEEP_TWO_PHASE
    hg = _hub_graph(4200, [129, 300])

    def rows(d):
        g = torch.Generator(device="cuda")
        g.manual_seed(d)
        return torch.randn((hg.n + hg.m, d), generator=g, device="cuda")

    def plain(G, d):
        z = rows(d)
        G.refine(0, z[:hg.n], z[hg.n:], 0.3, 3, mode)
        return z
    with H.Graph.from_hypergraph(hg) as G:
        want = {d: plain(G, d) for d in (32, 64)}
    with H.Graph.from_hypergraph(hg) as G:
        if warm:
            assert torch.equal(plain(G, 32), want[32])
        z = rows(32)
        torch.cuda.synchronize()
        graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=s):
            H.hnv_refine(G.handle, 0, z[:hg.n], z[hg.n:], 0.3, 3, mode, s)
        for d in (32, 64):
            assert torch.equal(plain(G, d), want[d])
            z.copy_(rows(32))
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(z, want[32])
        G.sync_status()
        del graph
    # nothing of the capture was released outside it
    with H.Graph.from_hypergraph(hg) as G:
        assert torch.equal(plain(G, 32), want[32])


def _ring(n, m):
    """m hyperedges of three consecutive nodes: 3 m incidences."""
    nodes = (np.arange(m, dtype=np.int64)[:, None] + np.arange(3)[None, :]) % n
    return n, m, 3 * np.arange(m + 1, dtype=np.int64), nodes.astype(np.int32).ravel()


# incidences at which the launch per row class takes over, by row size
@pytest.mark.parametrize("dtname,d,most", [
    ("f32", 4, 1_800_000), ("bf16", 8, 2_000_000), ("f32", 8, 1_800_000), ("bf16", 16, 1_800_000),
    ("f32", 32, 192_000_000 // 128), ("bf16", 64, 192_000_000 // 128),
    ("f32", 36, 125_000_000 // 144), ("bf16", 128, 170_000_000 // 256),
    ("bf16", 136, 125_000_000 // 272), ("f32", 128, 125_000_000 // 512),
    ("f32", 132, 160_000_000 // 528), ("bf16", 512, 160_000_000 // 1024)])
def test_levels_at_the_limit(H, dtname, d, most):
    """Both sides of the line between the one-launch path and the launch per
    row class; the stopping rule's is at 192 MB of gathered rows throughout."""
    import torch
    dt = torch.float32 if dtname == "f32" else torch.bfloat16
    for m in (most // 3, most // 3 + 1):
        n = 30_000 if d > 500 else 60_000 if d > 100 else 100_000
        with H.Graph(*_ring(n, m)) as G:
            z = torch.randn((n + m, d), device="cuda").to(dt)

            def refine():
                v, e = z[:n].clone(), z[n:].clone()
                G.refine(0, v, e, 0.3, 2)
                return v, e
            a, b, one, many = _both(H, refine)
            assert (one == 1) == (3 * m <= most) and many > 1
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])

            def until():
                v, e = z[:n].clone(), z[n:].clone()
                return v, e, G.refine_until(0, v, e, 0.3, 2, -1.0)
            a, b, one, many = _both(H, until)
            assert (one == 1) == (3 * m * d * z.element_size() <= 192_000_000) and a[2] == b[2]
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("d,teams", [(8, False), (32, True)])
def test_batch_takes_the_path_estimated_faster(H, d, teams):
    """Eight graphs that fill the device: narrow rows go to the step lists."""
    import torch
    Gs = [H.Graph(*_ring(200_000, 400_000 + i)) for i in range(8)]
    with H.Batch(Gs) as B:
        co, vo, eo = (int(a[-1]) for a in B.offsets())
        zc = torch.randn((co, d), device="cuda")
        zv, ze = torch.empty((vo, d), device="cuda"), torch.empty((eo, d), device="cuda")

        def vcycle():
            zv.fill_(float("nan"))
            ze.fill_(float("nan"))
            B.vcycle(zc, zv, ze, 0.3, 2)
            return zv.clone(), ze.clone()
        vcycle()                                         # (builds the lists)
        H.timing_enable(True)
        vcycle()
        H.timing_enable(False)
        H.timing_reset()
        a, b, one, many = _both(H, vcycle)
        assert (one == 1) == teams and many > 1
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    for G in Gs:
        G.close()


def test_hierarchies_of_many_levels(H):
    """Coarsening one graph again and again, to fewer and to more levels than
    a graph has room to describe from the start (40)."""
    import torch
    # hyperedges along a path, taken in order of their weight: a step merges
    # three nodes of 300
    n = 300
    nodes = (np.arange(n - 2)[:, None] + np.arange(3)[None, :]).astype(np.int32).ravel()
    prio = np.tile(np.arange(n - 2, dtype=np.uint64), (70, 1))
    with H.Graph(n, n - 2, 3 * np.arange(n - 1, dtype=np.int64), nodes) as G:
        seen = set()
        for most in (3, 64, 64, 5, 70):
            L = G.coarsen(policy=H.ASSIGN_EXPLICIT, explicit_prio=prio, min_nodes=2,
                          max_levels=most)
            seen.add(L > 40)
            top = G.level_info(L - 1)
            zc = torch.randn((top[0] + top[1], 16), device="cuda")
            zv = torch.empty((n, 16), device="cuda")
            ze = torch.empty((n - 2, 16), device="cuda")

            def vcycle():
                G.vcycle(zc, zv, ze, 0.5, 2)
                return zv.clone(), ze.clone()
            a, b, one, many = _both(H, vcycle)
            assert one == 1 and many > one
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        assert seen == {False, True}
