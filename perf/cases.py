"""The measured work of this repository: what a user has the library do,
through the Python entry points of ``paper_2103_09660_gb300`` (and the C ABI
under them where the binding has no device-side reader).

Every input is a planted-community hypergraph of the same family as
``hypergen`` (sizes ``min(cap, 2 + Zipf(alpha))``, members from a home
community with probability ``p_in``), drawn on the GPU from the seed so that
making it is quick. Member lists may name a node twice (the library removes
repeats). A node that was drawn into no hyperedge joins a random one (the
paper's cleaning removes such nodes; joining them keeps the row counts those
of the case). Sizes are the distribution's quantiles in a seeded order, so
that every seed has the same number of incidences, up to those joined.

The sizes of coarse levels differ from seed to seed. What is read of them
goes into buffers that a caller can size beforehand, from level 0; the rest
of such a buffer holds -1 (indices) or 0.

Kinds of work, and what each stands for:

* ``hierarchy``: new data arrives; build the incidence, coarsen, and read the
  rep maps and the coarsest star expansion (the input of the initial
  embedding method).
* ``features``: the same with node features and the cosine rule.
* ``step``: the whole method on new data (build, coarsen, V-cycle).
* ``vcycle``: a V-cycle on a hierarchy that is kept (another initial
  embedding of the same hypergraph), float32 or bfloat16 rows.
* ``refine``: sweeps on one level, either sweep order.
* ``until``: sweeps on one level until two iterates differ by at most eps.
* ``train``: differentiable V-cycle: forward and backward.
* ``batch``: many hypergraphs refined together.
"""

import math

import numpy as np
import torch

import paper_2103_09660_gb300 as H

_GAMMA = 0x9E3779B97F4A7C15
_M64 = (1 << 64) - 1


def listed():
    g2k = dict(n=2000, m=1000, C=8, alpha=2.0, cap=50, p_in=0.8, weighted=False)
    g200k = dict(n=200_000, m=150_000, C=16, alpha=1.8, cap=5000, p_in=0.7, weighted=True)
    g1m = dict(n=1_000_000, m=1_000_000, C=64, alpha=1.8, cap=5000, p_in=0.7, weighted=True)
    return [
        # one small graph (the size of the paper's smallest citation data): latency and launches
        dict(name="hierarchy_2k", kind="hierarchy", min_nodes=0, max_levels=4, **g2k),
        # the 1M-node workload's build and coarsening: sorts and scans at full size
        dict(name="hierarchy_1m", kind="hierarchy", min_nodes=0, max_levels=4, **g1m),
        # feature-based coarsening of a mid-size graph, a few levels as in the paper
        dict(name="features_200k", kind="features", min_nodes=0, max_levels=3, k=32, **g200k),
        # the V-cycle of one small graph: latency and launches
        dict(name="vcycle_2k", kind="vcycle", min_nodes=200, max_levels=32, d=32, sweeps=10,
             omega=0.5, dtype="f32", **g2k),
        # an ordinary graph of the size of the paper's co-authorship data, ragged sizes
        dict(name="vcycle_40k", kind="vcycle", min_nodes=400, max_levels=32, d=100, sweeps=20,
             omega=0.5, dtype="f32", n=41_302, m=22_363, C=6, alpha=2.0, cap=500, p_in=0.8,
             weighted=False),
        # the whole method at the benchmark's size
        dict(name="step_1m", kind="step", min_nodes=10_000, max_levels=32, d=128, sweeps=20,
             omega=0.5, dtype="f32", **g1m),
        # bfloat16 rows at the benchmark's size
        dict(name="vcycle_1m_bf16", kind="vcycle", min_nodes=10_000, max_levels=32, d=128,
             sweeps=20, omega=0.5, dtype="bf16", **g1m),
        # refinement without coarsening, the Jacobi order, odd sizes
        dict(name="refine_jacobi_150k", kind="refine", mode="jacobi", d=100, sweeps=10, omega=0.4,
             dtype="f32", n=150_001, m=120_003, C=16, alpha=1.8, cap=3000, p_in=0.7,
             weighted=True),
        # the stopping rule on one level
        dict(name="until_200k", kind="until", mode="two_phase", d=64, sweeps=40, omega=0.5,
             eps=0.03, dtype="f32", **g200k),
        # learning hyperedge weights: forward and backward of the V-cycle
        dict(name="train_200k", kind="train", min_nodes=0, max_levels=3, d=64, sweeps=10,
             omega=0.5, dtype="f32", **g200k),
        # a collection of small and ordinary hypergraphs
        dict(name="batch_64", kind="batch", graphs=64, n=1000, n_max=100_000, d=64, sweeps=10,
             omega=0.5, dtype="f32", C=8, alpha=2.0, cap=500, p_in=0.8, weighted=False,
             m_ratio=0.8, max_levels=32),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["hierarchy", "features", "step", "vcycle", "vcycle", "refine", "until",
                       "train", "batch"])
    alpha, cap = rng.choice([(1.8, 5000), (1.8, 1000), (2.0, 500), (2.0, 50)])
    dtype = rng.choice(["f32", "f32", "bf16"]) if kind in ("step", "vcycle", "refine", "batch") \
        else "f32"
    c = dict(kind=kind, C=rng.choice([4, 8, 16, 64]), alpha=alpha, cap=cap,
             p_in=rng.choice([0.5, 0.7, 0.8, 0.9]), weighted=rng.random() < 0.6)
    if kind == "batch":
        c.update(graphs=rng.randint(4, 48), n=logint(300, 2000), n_max=logint(3000, 60_000),
                 m_ratio=round(rng.uniform(0.5, 1.1), 3), max_levels=rng.choice([4, 8, 32]))
    else:
        top = {"features": 200_000, "train": 200_000}.get(kind, 900_000)
        c["n"] = logint(1000, top)
        c["m"] = max(1, int(c["n"] * rng.uniform(0.5, 1.0)))
    if kind in ("hierarchy", "features", "step", "vcycle", "train"):
        fixed = kind in ("hierarchy", "features", "train")
        c["min_nodes"] = 0 if fixed else max(50, c["n"] // rng.choice([20, 100]))
        c["max_levels"] = rng.choice([2, 3]) if fixed else 12
    if kind == "features":
        c["k"] = rng.choice([5, 16, 32, 50])
    if kind in ("step", "vcycle", "refine", "until", "train", "batch"):
        # bfloat16 rows and batches take d % 8 == 0, float32 rows d % 4 == 0
        q = 8 if dtype == "bf16" or kind == "batch" else 4
        most = 64 if kind in ("train", "batch") else 128
        c.update(d=q * rng.randint(1, most // q), omega=round(rng.uniform(0.2, 0.9), 2),
                 sweeps=rng.randint(3, 10 if kind == "train" else 20), dtype=dtype)
    if kind in ("refine", "until"):
        c["mode"] = rng.choice(["two_phase", "two_phase", "jacobi"])
    if kind == "until":
        c["eps"] = rng.choice([0.1, 0.03])
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _size_probs(case):
    """P(size = 2 + z), z = 1..cap, for Zipf(alpha) clipped at cap."""
    cap = int(case["cap"]) - 2
    k = np.arange(1, cap + 1, dtype=np.float64)
    p = k ** -float(case["alpha"])
    # the mass above the cap, by the integral of the tail
    a = float(case["alpha"])
    tail = (cap + 0.5) ** (1 - a) / (a - 1)
    p[-1] += tail
    return p / p.sum()


def _sizes(case, n, m):
    """Hyperedge sizes: m quantiles of the size distribution, ascending."""
    q = (np.arange(m) + 0.5) / m
    z = np.searchsorted(np.cumsum(_size_probs(case)), q)
    return np.minimum(z + 3, min(int(case["cap"]), n))


def _graph(case, n, m, seed):
    """(n, m, edge_ptr int64, edge_nodes int32, weights float32) on the GPU."""
    dev = "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    C = min(int(case["C"]), n)
    sizes = torch.from_numpy(_sizes(case, n, m)).to(dev)
    sizes = sizes[torch.randperm(m, generator=g, device=dev)]
    home = torch.randint(0, C, (m,), generator=g, device=dev)
    order = torch.randperm(n, generator=g, device=dev)       # community c: order[c::C]
    edge = torch.repeat_interleave(torch.arange(m, device=dev), sizes)
    nnz = edge.numel()
    h = home[edge]
    inside = torch.rand(nnz, generator=g, device=dev) < case["p_in"]
    u = torch.rand(nnz, generator=g, device=dev, dtype=torch.float64)
    count = (n - h + C - 1) // C
    pos = torch.where(inside, (u * count).long() * C + h, (u * n).long())
    nodes = order[torch.clamp(pos, max=n - 1)]
    used = torch.zeros(n, dtype=torch.bool, device=dev)
    used[nodes] = True
    lone = torch.nonzero(~used)[:, 0]
    if lone.numel():
        edge = torch.cat([edge, torch.randint(0, m, (lone.numel(),), generator=g, device=dev)])
        edge, at = torch.sort(edge, stable=True)
        nodes = torch.cat([nodes, lone])[at]
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=dev)
    ptr[1:] = torch.cumsum(torch.bincount(edge, minlength=m), 0)
    w = (torch.rand(m, generator=g, device=dev) * 1.5 + 0.5) if case["weighted"] \
        else torch.ones(m, device=dev)
    return n, m, ptr, nodes.int().contiguous(), w.float()


def _rows(rows, d, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    z = torch.randn((rows, d), generator=g, device="cuda")
    return z.to(torch.bfloat16) if dtype == "bf16" else z


def _batch_sizes(case):
    """(n, m) of every graph: n spread over the logarithm of its range."""
    lo, hi = math.log(case["n"]), math.log(case["n_max"])
    k = case["graphs"]
    ns = [int(math.exp(lo + (hi - lo) * (i + 0.5) / k)) for i in range(k)]
    return [(n, max(1, int(case["m_ratio"] * n))) for n in ns]


def _coarsest_capacity(case):
    """Rows that hold the coarsest level of a differentiated hierarchy."""
    return case["n"] + case["m"]


def _torch_dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    s.seed = seed
    kind = case["kind"]
    if kind == "batch":
        s.graphs = []
        for i, (n, m) in enumerate(_batch_sizes(case)):
            G = H.Graph(*_graph(case, n, m, seed * 1009 + i))
            G.coarsen(seed=seed, min_nodes=max(200, n // 100), max_levels=case["max_levels"])
            s.graphs.append(G)
        s.batch = H.Batch(s.graphs)
        co, vo, eo = (int(a[-1]) for a in s.batch.offsets())
        s.zc = _rows(co, case["d"], case["dtype"], seed)
        s.zv = torch.empty((vo, case["d"]), dtype=_torch_dtype(case), device="cuda")
        s.ze = torch.empty((eo, case["d"]), dtype=_torch_dtype(case), device="cuda")
        return s
    s.data = _graph(case, case["n"], case["m"], seed)
    n, m = s.data[0], s.data[1]
    s.capacity = int(_sizes(case, n, m).sum()) + n       # incidences of level 0, at most
    if kind == "hierarchy":
        return s
    if kind == "features":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed * 31 + 5)
        mu = torch.randn((int(case["C"]), case["k"]), generator=g, device="cuda")
        lab = torch.randint(0, int(case["C"]), (n,), generator=g, device="cuda")
        s.x = mu[lab] + torch.randn((n, case["k"]), generator=g, device="cuda")
        return s
    G = H.Graph(*s.data)
    if kind in ("refine", "until"):
        s.z0v = _rows(n, case["d"], case["dtype"], seed)
        s.z0e = _rows(m, case["d"], case["dtype"], seed + 1)
        s.mode = H.SWEEP_JACOBI if case["mode"] == "jacobi" else H.SWEEP_TWO_PHASE
        s.graph = G
        return s
    L = G.coarsen(seed=seed, min_nodes=case["min_nodes"], max_levels=case["max_levels"])
    tn, tm, _ = G.level_info(L - 1)
    if kind == "train":
        s.graph = G
        s.rows = tn + tm
        s.w = s.data[4].clone().requires_grad_(True)
        # the learned table: the coarsest level takes its first rows
        s.zc = _rows(_coarsest_capacity(case), case["d"], "f32", seed).requires_grad_(True)
        s.gv = _rows(n, case["d"], "f32", seed + 2) / n
        s.ge = _rows(m, case["d"], "f32", seed + 3) / m
        return s
    s.zc = _rows(tn + tm, case["d"], case["dtype"], seed)
    s.zv = torch.empty((n, case["d"]), dtype=_torch_dtype(case), device="cuda")
    s.ze = torch.empty((m, case["d"]), dtype=_torch_dtype(case), device="cuda")
    if kind == "vcycle":
        s.graph = G
    else:
        G.close()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _level_tensor(G, level, which, capacity):
    """A level's array in a device tensor of `capacity` (hnv_copy_level_array)."""
    if which == H.ARR_W:
        t = torch.zeros(capacity, dtype=torch.float32, device="cuda")
    else:
        t = torch.full((capacity,), -1, dtype=torch.int32, device="cuda")
    rc = H.lib().hnv_copy_level_array(G.handle, level, which, t.data_ptr(), 4 * capacity, 1,
                                      torch.cuda.current_stream().cuda_stream)
    if rc != 0:
        raise RuntimeError("hnv_copy_level_array: %d" % rc)
    return t


def _hierarchy_out(G, L, n, m, capacity):
    """The rep maps of every level and the coarsest star expansion."""
    out = []
    for l in range(L - 1):
        out += [_level_tensor(G, l, H.ARR_REP_V, n), _level_tensor(G, l, H.ARR_REP_E, m)]
    out += [_level_tensor(G, L - 1, H.ARR_E_PTR, m + 1), _level_tensor(G, L - 1, H.ARR_W, m)]
    return out + [_level_tensor(G, L - 1, H.ARR_E_NODES, capacity)]


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "batch":
        s.batch.vcycle(s.zc, s.zv, s.ze, case["omega"], case["sweeps"])
        return s.zv, s.ze
    if kind == "vcycle":
        s.graph.vcycle(s.zc, s.zv, s.ze, case["omega"], case["sweeps"])
        return s.zv, s.ze
    if kind == "refine":
        zv, ze = s.z0v.clone(), s.z0e.clone()
        s.graph.refine(0, zv, ze, case["omega"], case["sweeps"], s.mode)
        return zv, ze
    if kind == "until":
        zv, ze = s.z0v.clone(), s.z0e.clone()
        done, delta = s.graph.refine_until(0, zv, ze, case["omega"], case["sweeps"], case["eps"],
                                           s.mode)
        return zv, ze, done, delta
    if kind == "train":
        zv, ze = H.vcycle_autograd(s.graph, s.w, s.zc[:s.rows], case["omega"], case["sweeps"])
        gw, gz = torch.autograd.grad([zv, ze], [s.w, s.zc], [s.gv, s.ge])
        return zv.detach(), ze.detach(), gw, gz
    G = H.Graph(*s.data)
    try:
        if kind == "features":
            G.set_node_features(s.x)
            L = G.coarsen(policy=H.ASSIGN_COSINE, seed=s.seed, min_nodes=case["min_nodes"],
                          max_levels=case["max_levels"])
            out = _hierarchy_out(G, L, s.data[0], s.data[1], s.capacity)
            for l in range(1, L):
                t = torch.zeros((s.data[0], case["k"]), device="cuda")
                rc = H.lib().hnv_copy_level_features(
                    G.handle, l, t.data_ptr(), t.numel() * 4, 1,
                    torch.cuda.current_stream().cuda_stream)
                if rc != 0:
                    raise RuntimeError("hnv_copy_level_features: %d" % rc)
                out.append(t)
            return out
        L = G.coarsen(seed=s.seed, min_nodes=case["min_nodes"], max_levels=case["max_levels"])
        if kind == "hierarchy":
            return _hierarchy_out(G, L, s.data[0], s.data[1], s.capacity)
        G.vcycle(s.zc, s.zv, s.ze, case["omega"], case["sweeps"])
        return s.zv, s.ze
    finally:
        G.close()


# ---------------------------------------------------------------------------
# Work and tolerance
# ---------------------------------------------------------------------------

# Rows and incidences of the levels of a hierarchy as shares of level 0
# (nodes, hyperedges, incidences): the planted 1M-node workload's.
_SHARES = [(1.0, 1.0, 1.0), (0.127, 0.984, 0.68), (0.034, 0.983, 0.52), (0.013, 0.976, 0.37),
           (0.0064, 0.889, 0.24)]


def _levels(case, n, m):
    """Estimated (n, m, nnz) of every level (the real counts depend on the draw)."""
    mean = float((_size_probs(case) * (np.arange(1, int(case["cap"]) - 1) + 2)).sum())
    nnz = m * min(mean, 0.9 * n)
    out = []
    for i, (a, b, c) in enumerate(_SHARES):
        if i and (out[-1][0] <= case.get("min_nodes", 0) or i > case.get("max_levels", 99)):
            break
        out.append((max(2.0, a * n), b * m, c * nnz))
    return out


def _sweep_work(case, n, m, nnz):
    """Bytes and flops of one two-sided sweep: both row tables read and
    written once, the incidence read once."""
    es = 2 if case["dtype"] == "bf16" else 4
    d = case["d"]
    return 2 * es * d * (n + m) + 4 * nnz + 8 * (n + m), 3 * nnz * d + 6 * (n + m) * d


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for n, m in _batch_sizes(case):
            for lv in _levels(dict(case, min_nodes=max(200, n // 100)), n, m):
                x, y = _sweep_work(case, *lv)
                b, f = b + x * case["sweeps"], f + y * case["sweeps"]
        return {"bytes": b, "flops": f}
    lv = _levels(case, case["n"], case["m"])
    n, m, nnz = lv[0]
    hier = 12 * m + 4 * nnz + sum(8 * (a + c) + 8 * q for a, c, q in lv[1:])
    if kind == "hierarchy":
        return {"bytes": hier, "flops": 0.0}
    if kind == "features":
        k = case["k"]
        b = f = 0.0
        for i, (a, c, q) in enumerate(lv):
            b += 4 * k * a + (4 * k * a + 12 * q if i + 1 < len(lv) else 0)
            f += 3 * q * k if i + 1 < len(lv) else 0
        return {"bytes": b + hier, "flops": f}
    if kind in ("refine", "until"):
        x, y = _sweep_work(case, n, m, nnz)
        # the stopping rule ends the sweeps early; about a third of the most
        k = case["sweeps"] if kind == "refine" else max(3, case["sweeps"] // 3)
        return {"bytes": x * k, "flops": y * k}
    b = f = 0.0
    for a in lv:
        x, y = _sweep_work(case, *a)
        b, f = b + x * case["sweeps"], f + y * case["sweeps"]
    if kind == "train":
        b, f = 3 * b, 3 * f          # forward, replay of the iterates, reverse
    if kind == "step":
        b += hier
    return {"bytes": b, "flops": f}


def tolerance(case):
    kind = case["kind"]
    if kind in ("hierarchy", "features"):
        return "exact"               # integers; features have a fixed order of rounded steps
    if case["dtype"] == "bf16":
        return {"rel": 4e-3, "max": 0.1}
    if kind == "train":
        return {"rel": 2e-5, "max": 2e-3}
    return {"rel": 8e-6, "max": 3e-4}


# ---------------------------------------------------------------------------
# The same in 64 bits, without the library
# ---------------------------------------------------------------------------

def _mix64(z):
    """SplitMix64 finaliser on int64 tensors (two's complement)."""
    def shr(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)

    def signed(c):
        return c - (1 << 64) if c >= 1 << 63 else c
    z = (z ^ shr(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _mix64_int(z):
    z &= _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


class _Level:
    """Incidence pairs (edge, node), distinct and in hyperedge order."""

    def __init__(self, n, m, edge, node, w):
        self.n, self.m, self.edge, self.node, self.w = n, m, edge, node, w

    def operators(self):
        dev = self.node.device
        cnt = torch.bincount(self.edge, minlength=self.m)
        ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), torch.cumsum(cnt, 0)])
        A = torch.sparse_csr_tensor(ptr, self.node, (1.0 / cnt.double())[self.edge],
                                    size=(self.m, self.n))
        order = torch.argsort(self.node, stable=True)
        deg = torch.zeros(self.n, dtype=torch.float64, device=dev).index_add_(
            0, self.node, self.w[self.edge])
        vc = torch.bincount(self.node, minlength=self.n)
        vp = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), torch.cumsum(vc, 0)])
        e = self.edge[order]
        B = torch.sparse_csr_tensor(vp, e, self.w[e] / deg[self.node[order]],
                                    size=(self.n, self.m))
        return A, B, (vc > 0).double()[:, None]


def _level0(data):
    n, m, ptr, nodes, w = data
    e = torch.repeat_interleave(torch.arange(m, device="cuda"), ptr[1:] - ptr[:-1])
    key = torch.unique(e * n + nodes.long())
    return _Level(n, m, key // n, key % n, w.double())


def _coarsen(lv, seed, min_nodes, max_levels):
    levels, reps = [lv], []
    while lv.n > min_nodes and len(levels) - 1 < max_levels and lv.m > 0:
        salt = _mix64_int(seed + (len(levels) - 1) * _GAMMA)
        salt = salt - (1 << 64) if salt >= 1 << 63 else salt
        prio = _mix64(torch.arange(lv.m, device="cuda") ^ salt) ^ (-(1 << 63))
        order = torch.argsort(prio)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(lv.m, device="cuda")
        best = torch.full((lv.n,), lv.m, dtype=torch.int64, device="cuda")
        best.scatter_reduce_(0, lv.node, rank[lv.edge], "amin")
        lone = best == lv.m
        c = order[torch.clamp(best, max=lv.m - 1)]
        key = torch.where(lone, lv.m + torch.arange(lv.n, device="cuda"), c)
        uniq, rep_v = torch.unique(key, return_inverse=True)
        n2 = uniq.numel()
        if n2 == lv.n:
            break
        img = torch.unique(lv.edge * n2 + rep_v[lv.node])
        ie, iv = img // n2, img % n2
        size = torch.bincount(ie, minlength=lv.m)
        keep = size >= 2
        new = torch.cumsum(keep, 0) - 1
        rep_e = new.clone()
        gone = ~keep[ie]
        rep_e[ie[gone]] = -1 - iv[gone]
        sel = keep[ie]
        lv = _Level(n2, int(keep.sum()), new[ie[sel]], iv[sel], lv.w[keep])
        levels.append(lv)
        reps.append((rep_v, rep_e))
    return levels, reps


def _sweep(A, B, has, zv, ze, omega, jacobi=False):
    e2 = (1 - omega) * ze + omega * (A @ zv)
    return (1 - omega * has) * zv + omega * (B @ (ze if jacobi else e2)), e2


def _project(rep, zv, ze):
    rep_v, rep_e = rep
    both = torch.cat([ze, zv])
    idx = torch.where(rep_e >= 0, rep_e, ze.shape[0] - 1 - rep_e)
    return zv[rep_v], both[idx]


def _omega(case):
    return float(np.float32(case["omega"]))


def _vcycle64(levels, reps, zc, omega, sweeps):
    zv, ze = zc[:levels[-1].n], zc[levels[-1].n:]
    for l in range(len(levels) - 1, -1, -1):
        if l < len(reps):
            zv, ze = _project(reps[l], zv, ze)
        if levels[l].m == 0:
            continue
        ops = levels[l].operators()
        for _ in range(sweeps):
            zv, ze = _sweep(*ops, zv, ze, omega)
    return zv, ze


def _train64(levels, reps, zc, omega, sweeps, gv, ge):
    """Gradients by torch.autograd over plain indexing, in float64."""
    w0 = levels[0].w.clone().requires_grad_(True)
    zc = zc.clone().requires_grad_(True)
    top = levels[-1]
    zv, ze = zc[:top.n], zc[top.n:top.n + top.m]
    ws = [w0]
    for l, (_, rep_e) in enumerate(reps):
        ws.append(ws[l][rep_e >= 0])
    for l in range(len(levels) - 1, -1, -1):
        if l < len(reps):
            zv, ze = _project(reps[l], zv, ze)
        lv, w = levels[l], ws[l]
        if lv.m == 0:
            continue
        inv = 1.0 / torch.bincount(lv.edge, minlength=lv.m).double()[:, None]
        deg = torch.zeros(lv.n, dtype=torch.float64, device="cuda").index_add(
            0, lv.node, w[lv.edge])
        has = (torch.bincount(lv.node, minlength=lv.n) > 0).double()[:, None]
        safe = torch.where(has[:, 0] > 0, deg, torch.ones_like(deg))[:, None]
        for _ in range(sweeps):
            ze = (1 - omega) * ze + omega * inv * torch.zeros_like(ze).index_add(
                0, lv.edge, zv[lv.node])
            s = torch.zeros_like(zv).index_add(0, lv.node, (w[:, None] * ze)[lv.edge])
            zv = (1 - omega * has) * zv + omega * s / safe
    gw, gz = torch.autograd.grad([zv, ze], [w0, zc], [gv, ge])
    return zv.detach(), ze.detach(), gw, gz


def exact(case, seed):
    kind = case["kind"]
    if kind in ("hierarchy", "features"):
        return None                  # integers, and features defined by their float32 steps
    omega = _omega(case)
    if kind == "batch":
        vs, es, at = [], [], 0
        hs = []
        for i, (n, m) in enumerate(_batch_sizes(case)):
            hs.append(_coarsen(_level0(_graph(case, n, m, seed * 1009 + i)), seed,
                               max(200, n // 100), case["max_levels"]))
        zc = _rows(sum(h[0][-1].n + h[0][-1].m for h in hs), case["d"], case["dtype"],
                   seed).double()
        for levels, reps in hs:
            rows = levels[-1].n + levels[-1].m
            v, e = _vcycle64(levels, reps, zc[at:at + rows], omega, case["sweeps"])
            at += rows
            vs.append(v)
            es.append(e)
        return torch.cat(vs), torch.cat(es)
    data = _graph(case, case["n"], case["m"], seed)
    lv = _level0(data)
    if kind in ("refine", "until"):
        zv = _rows(lv.n, case["d"], case["dtype"], seed).double()
        ze = _rows(lv.m, case["d"], case["dtype"], seed + 1).double()
        ops = lv.operators()
        done, delta = 0, 0.0
        for it in range(case["sweeps"]):
            v2, e2 = _sweep(*ops, zv, ze, omega, case["mode"] == "jacobi")
            if kind == "until":
                delta = max(float((v2 - zv).abs().max()), float((e2 - ze).abs().max()))
            zv, ze, done = v2, e2, it + 1
            if kind == "until" and delta <= case["eps"]:
                break
        return (zv, ze) if kind == "refine" else (zv, ze, done, delta)
    levels, reps = _coarsen(lv, seed, case["min_nodes"], case["max_levels"])
    if kind == "train":
        zc = _rows(_coarsest_capacity(case), case["d"], "f32", seed).double()
        gv = (_rows(lv.n, case["d"], "f32", seed + 2) / lv.n).double()
        ge = (_rows(lv.m, case["d"], "f32", seed + 3) / lv.m).double()
        return _train64(levels, reps, zc, omega, case["sweeps"], gv, ge)
    zc = _rows(levels[-1].n + levels[-1].m, case["d"], case["dtype"], seed).double()
    return _vcycle64(levels, reps, zc, omega, case["sweeps"])
