"""Measured cases: the calls a user of the library makes, over the sizes it is used at.

The paper's use is interactive: a graph is uploaded, a view of it (all nodes,
some nodes, or the supernodes of one hierarchy level) is turned into DPPR and
PDist, and the view is laid out. Every case is one such call, or the chain of
them, through the package's public entry points, on seeded synthetic graphs of
the kinds the tests and the benchmark use: Chung-Lu power-law graphs, stochastic
block models, dense weighted block models, directed graphs with dangling nodes.

FP32 layouts run few updates (a first picture, or one step of a progressive
display): an update amplifies the rounding of the one before, so after some
tens of updates two equally exact FP32 runs no longer agree in their digits.
The FP64 chain runs its full 300 updates.
"""
import math

import numpy as np
import torch

import paper_2112_14944_gb300 as pp

ALPHA = 0.15
EPS = 1e-6
DEV = "cuda:0"


def listed():
    return [
        # one click of an interactive session: a small cluster is uploaded, its DPPR and PDist
        # computed and drawn; launches and latency count, not bytes
        {"name": "view_150", "kind": "view", "n": 150, "blocks": 6, "iters": 20},
        # the benchmark's graph: ingest, then all-pairs DPPR and PDist of a 10,000-node view
        {"name": "dppr_10k", "kind": "dppr", "n": 10000, "degree": 20.0},
        # the paper's general setting: a directed graph, an odd number of nodes
        {"name": "dppr_directed_7k", "kind": "directed", "n": 7001, "degree": 20.0},
        # a dense weighted view (15 % of all pairs): the tensor-core sweeps
        {"name": "dppr_dense_6k", "kind": "dense", "n": 6000, "density": 0.15},
        # a view of some nodes of a large graph: the state of the sweeps does not fit in L2
        {"name": "dppr_view_of_2m", "kind": "subview", "n": 2000000, "k": 256},
        # the parity setting: everything in FP64, DPPR, PDist and 300 layout updates
        {"name": "fp64_1k", "kind": "fp64", "n": 1000, "degree": 10.0, "iters": 300},
        # a layout of the benchmark's size: L^w inverse and streaming passes over k x k matrices
        {"name": "layout_10k", "kind": "layout", "k": 10000, "iters": 30},
        # a layout of ordinary size, ragged against every tile; its matrices stay in L2
        {"name": "layout_2k", "kind": "layout", "k": 1999, "iters": 30},
        # one gradient step on the stress: energy forward, gradients of X and PDist backward
        {"name": "energy_8k", "kind": "energy", "k": 8192, "dtype": "float32"},
        # exact DPPR between the 25 children (25 leaves each) of a supernode of a large graph
        {"name": "level_2m", "kind": "level", "n": 2000000, "children": 25, "leaves": 25},
        # the same query answered approximately by Tau-Push from the DPR index
        {"name": "tau_push_2m", "kind": "tau", "n": 2000000, "children": 25, "leaves": 25},
        # many small views of a multi-level navigation in one call
        {"name": "views_32", "kind": "views", "count": 32, "n_min": 50, "n_max": 2000, "iters": 20},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["view", "dppr", "directed", "dense", "subview", "fp64", "layout", "layout", "energy", "level",
                       "tau", "views"])
    if kind == "view":
        return {"kind": kind, "n": _log(rng, 40, 800), "blocks": rng.randint(4, 8), "iters": rng.randint(10, 20)}
    if kind in ("dppr", "directed"):
        return {"kind": kind, "n": _log(rng, 1000, 9999 if kind == "dppr" else 7000),
                "degree": round(rng.uniform(8.0, 20.0), 1)}
    if kind == "dense":
        return {"kind": kind, "n": _log(rng, 1200, 6000), "density": round(rng.uniform(0.08, 0.15), 3)}
    if kind == "subview":
        return {"kind": kind, "n": _log(rng, 100000, 2000000), "k": _log(rng, 32, 255)}
    if kind == "fp64":
        return {"kind": kind, "n": _log(rng, 100, 999), "degree": round(rng.uniform(6.0, 10.0), 1),
                "iters": rng.randint(100, 300)}
    if kind == "layout":
        return {"kind": kind, "k": _log(rng, 100, 9999), "iters": rng.randint(10, 30)}
    if kind == "energy":
        double = rng.random() < 0.25
        return {"kind": kind, "k": _log(rng, 200, 3000 if double else 8191), "dtype": "float64" if double else "float32"}
    if kind in ("level", "tau"):
        return {"kind": kind, "n": _log(rng, 100000, 2000000), "children": rng.randint(8, 25),
                "leaves": rng.randint(1, 25)}
    return {"kind": kind, "count": rng.randint(8, 32), "n_min": 50, "n_max": _log(rng, 300, 1999),
            "iters": rng.randint(10, 20)}


# ---- inputs (on the GPU, from the seed alone) --------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 12345)
    return g


def _csr(n, u, v, w=None):
    """CSR (row_ptr int64, col int32, weights or None) of directed pairs, duplicates dropped, rows sorted."""
    key = u * n + v
    if w is None:
        key = torch.unique(key)
    else:
        key, order = torch.sort(key)
        w = w[order].contiguous()
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return rp, (key % n).to(torch.int32).contiguous(), w


def _chung_lu_pairs(n, degree, gen, exponent=2.5):
    """Undirected pairs u < v of a power-law graph, ids in descending expected degree: both ends of
    n degree / 2 edges drawn in proportion to (i + 1)^(-1 / (exponent - 1)), loops and repeats dropped."""
    w = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-1.0 / (exponent - 1.0))
    for _ in range(8):
        w = w * (degree * n / w.sum())
        w = torch.minimum(w, torch.sqrt(w.sum()))
    cum = torch.cumsum(w / w.sum(), 0)
    ends = torch.searchsorted(cum, torch.rand(2, int(n * degree / 2), generator=gen, device=DEV, dtype=torch.float64))
    ends = ends.clamp_(max=n - 1)
    u, v = torch.minimum(ends[0], ends[1]), torch.maximum(ends[0], ends[1])
    key = torch.unique((u * n + v)[u != v])
    return key // n, key % n


def _chung_lu(n, degree, gen):
    u, v = _chung_lu_pairs(n, degree, gen)
    return _csr(n, torch.cat([u, v]), torch.cat([v, u]))


def _directed(n, degree, gen):
    """30 % of the edges in both directions, the others in one; 2 % of the nodes without out-edges."""
    u, v = _chung_lu_pairs(n, degree, gen)
    both = torch.rand(u.shape[0], generator=gen, device=DEV) < 0.3
    fwd = torch.rand(u.shape[0], generator=gen, device=DEV) < 0.5
    s = torch.cat([u[both | fwd], v[both | ~fwd]])
    d = torch.cat([v[both | fwd], u[both | ~fwd]])
    keep = (torch.rand(n, generator=gen, device=DEV) >= 0.02)[s]
    return _csr(n, s[keep], d[keep])


def _blocks(n, blocks, p_in, p_out, gen, weighted=False):
    """Stochastic block model (symmetric lognormal weights if weighted); isolated nodes are kept."""
    b = torch.arange(n, device=DEV) * blocks // n
    p = torch.where(b[:, None] == b[None, :], p_in, p_out)
    hit = torch.triu(torch.rand(n, n, generator=gen, device=DEV) < p, 1)
    u, v = torch.nonzero(hit, as_tuple=True)
    if not weighted:
        return _csr(n, torch.cat([u, v]), torch.cat([v, u]))
    w = torch.exp(torch.randn(u.shape[0], generator=gen, device=DEV))
    return _csr(n, torch.cat([u, v]), torch.cat([v, u]), torch.cat([w, w]))


def _dense(n, density, gen):
    # 20 blocks, edges 8 times as likely inside a block as between blocks
    p_out = density / (8.0 / 20.0 + 1.0 - 1.0 / 20.0)
    return _blocks(n, 20, min(1.0, 8.0 * p_out), p_out, gen, weighted=True)


def _view_sizes(case):
    # spread evenly over the range, in a mixed order (the sizes are the case's, the graphs the seed's)
    at = np.arange(case["count"])
    sizes = case["n_min"] + (case["n_max"] - case["n_min"]) * (at * 7 % case["count"]) // max(1, case["count"] - 1)
    return sizes, 4 + at % 13


def _distances(k, gen, dtype):
    """A symmetric matrix with the values of a power-law view's PDist: Eq. (1) on the stationary share
    2 d_i d_j / m with a lognormal spread, and a larger share on the pairs that are edges."""
    d = torch.exp(torch.randn(k, generator=gen, device=DEV) * 0.9 + 2.5)
    m = d.sum()
    r = torch.randn(k, k, generator=gen, device=DEV)
    r = torch.triu(r, 1)
    r = r + r.T
    z = 2.0 * d[:, None] * d[None, :] / m
    z = z * torch.exp(0.35 * r) + torch.where(r > 2.8, 0.12, 0.0)
    delta = torch.clamp(1.0 - torch.log(z), 2.0, 2.0 * math.log(max(k, 8)))
    delta.fill_diagonal_(0.0)
    return delta.to(dtype).contiguous()


def _x0(rows, gen, dtype=torch.float32):
    return (2.0 * torch.rand(rows, 2, generator=gen, device=DEV) - 1.0).to(dtype)


def _leaves(n, children, leaves, gen):
    ids = torch.randperm(n, generator=gen, device=DEV)[: children * leaves].to(torch.int32)
    return torch.arange(children + 1, dtype=torch.int64, device=DEV) * leaves, ids


def _inputs(case, seed):
    """The arrays of a case; prepare() hands them to the library, exact() to plain torch."""
    gen, kind = _gen(seed), case["kind"]
    if kind == "view":
        return {"csr": _blocks(case["n"], case["blocks"], 0.3, 0.01, gen), "x0": _x0(case["n"], gen)}
    if kind == "dppr":
        return {"csr": _chung_lu(case["n"], case["degree"], gen)}
    if kind == "directed":
        return {"csr": _directed(case["n"], case["degree"], gen)}
    if kind == "dense":
        return {"csr": _dense(case["n"], case["density"], gen)}
    if kind == "subview":
        view = torch.randperm(case["n"], generator=gen, device=DEV)[: case["k"]].to(torch.int32)
        return {"csr": _chung_lu(case["n"], 10.0, gen), "view": view}
    if kind == "fp64":
        return {"csr": _chung_lu(case["n"], case["degree"], gen), "x0": _x0(case["n"], gen, torch.float64)}
    if kind == "layout":
        return {"delta": _distances(case["k"], gen, torch.float32), "x0": _x0(case["k"], gen)}
    if kind == "energy":
        dtype = getattr(torch, case["dtype"])
        return {"delta": _distances(case["k"], gen, dtype), "x": (5.0 * _x0(case["k"], gen)).to(dtype)}
    if kind in ("level", "tau"):
        ptr, idx = _leaves(case["n"], case["children"], case["leaves"], gen)
        return {"csr": _chung_lu(case["n"], 10.0, gen), "ptr": ptr, "idx": idx}
    sizes, blocks = _view_sizes(case)
    return {"csrs": [_blocks(int(n), int(b), 0.1, 0.002, gen) for n, b in zip(sizes, blocks)],
            "x0": _x0(int(sizes.sum()), gen)}


_ctx = None


def _context():
    """One library context for the process, as a program has it."""
    global _ctx
    if _ctx is None:
        _ctx = pp.Context(0, torch_stream=True)
    return _ctx


def _upload(csr, directed=False):
    rp, col, w = csr
    return _context().upload(rp.shape[0] - 1, rp, col, w, directed=directed)


def _square(k, dtype=torch.float32):
    return torch.empty(k, k, dtype=dtype, device=DEV)


def prepare(case, seed):
    """The inputs of the call on the GPU, the output buffers, and the graph handle a program keeps."""
    s, kind = _inputs(case, seed), case["kind"]
    s["case"] = case
    if kind in ("directed", "dense", "subview", "level", "tau"):
        s["graph"] = _upload(s["csr"], directed=kind == "directed")
    if kind in ("view", "dppr", "directed", "dense", "fp64"):
        n = case["n"]
        s["view"] = torch.arange(n, dtype=torch.int32, device=DEV)
        dtype = torch.float64 if kind == "fp64" else torch.float32
        s["dppr"], s["pdist"] = _square(n, dtype), _square(n, dtype)
    if kind == "subview":
        s["dppr"], s["pdist"] = _square(case["k"]), _square(case["k"])
    if "x0" in s:
        s["x"] = torch.empty_like(s["x0"])
    if kind == "energy":
        s["x"].requires_grad_(True)
        s["delta"].requires_grad_(True)
    if kind == "level":
        s["sets"] = list(s["idx"].cpu().numpy().reshape(case["children"], case["leaves"]))
    if kind == "tau":
        s["dpr"] = torch.empty(case["n"], dtype=torch.float64, device=DEV)
        _context().dpr(s["graph"], out=s["dpr"])
        s["dppr"], s["pdist"] = _square(case["children"], torch.float64), _square(case["children"], torch.float64)
    if kind == "views":
        s["graphs"] = [_upload(c) for c in s["csrs"]]
    for key in ("csr", "csrs"):
        if key in s and kind not in ("view", "dppr", "fp64"):
            del s[key]  # the library has its copy
    return s


def run(state):
    s, case, ctx = state, state["case"], _context()
    kind = case["kind"]
    if kind in ("view", "dppr", "fp64"):  # ingest included: a new graph each time
        fp64 = kind == "fp64"
        precision = pp.FP64 if fp64 else pp.FP32
        graph = _upload(s["csr"])
        ctx.dppr(graph, s["view"], alpha=ALPHA, eps=EPS, precision=precision, dppr_out=s["dppr"], pdist_out=s["pdist"],
                 out64=fp64)
        out = [s["dppr"], s["pdist"]]
        if kind != "dppr":
            x, stress = ctx.layout(s["pdist"], s["x0"], case["iters"], precision=precision, x_out=s["x"])
            out += [x, stress]
        graph.free()
        return out
    if kind in ("directed", "dense", "subview"):
        ctx.dppr(s["graph"], s["view"], alpha=ALPHA, eps=EPS, dppr_out=s["dppr"], pdist_out=s["pdist"])
        return [s["dppr"], s["pdist"]]
    if kind == "layout":
        x, stress = ctx.layout(s["delta"], s["x0"], case["iters"], x_out=s["x"])
        return [x, stress]
    if kind == "energy":
        energy = pp.StressEnergy.apply(s["x"], s["delta"], ctx)
        return [energy.detach(), *torch.autograd.grad(energy, (s["x"], s["delta"]))]
    if kind == "level":
        dppr, pdist, _, _ = ctx.level_dppr(s["graph"], s["sets"], alpha=ALPHA, eps=EPS)
        return [dppr, pdist]
    if kind == "tau":
        dppr, pdist, _ = ctx.tau_push(s["graph"], s["ptr"], s["idx"], s["dpr"], alpha=ALPHA, ldppr_out=s["dppr"],
                                      pdist_out=s["pdist"])
        return [dppr, pdist]
    x, pdist, stress, _ = ctx.views_batch(s["graphs"], s["x0"], alpha=ALPHA, eps=EPS, iters=case["iters"],
                                          want_pdist=True)
    # the stress of an FP32 layout is an FP32 quantity, whatever type it is summed in
    return [x, pdist, stress.astype(np.float32)]


# ---- what a pass cannot do without -------------------------------------------------------------------------------

SWEEPS = 10  # products with the walk matrix for DPPR to 1e-6 of a well-connected graph


def _dppr_work(n, nnz, k, elem=4, weighted=False):
    return {"bytes": 8.0 * n + (8.0 if weighted else 4.0) * nnz + 2.0 * elem * k * k, "flops": 2.0 * nnz * k * SWEEPS}


def _layout_work(k, iters, elem=4):
    # the symmetric matrices once, the inverse's k^3, and per update two products with a k x k matrix
    return {"bytes": elem * (1.0 * k * k + 4.0 * k), "flops": 1.0 * k ** 3 + iters * k * (k - 1.0) / 2.0 * 28.0}


def _sum(*parts):
    return {key: float(sum(p[key] for p in parts)) for key in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "view":
        n = case["n"]
        return _sum(_dppr_work(n, 0.06 * n * n, n), _layout_work(n, case["iters"]))
    if kind == "dppr":
        return _dppr_work(case["n"], case["n"] * case["degree"], case["n"])
    if kind == "directed":
        return _dppr_work(case["n"], 0.65 * case["n"] * case["degree"], case["n"])
    if kind == "dense":
        n = case["n"]
        return _dppr_work(n, case["density"] * n * n, n, weighted=True)
    if kind == "subview":
        return _dppr_work(case["n"], 10.0 * case["n"], case["k"])
    if kind == "fp64":
        n = case["n"]
        return _sum(_dppr_work(n, case["degree"] * n, n, 8), _layout_work(n, case["iters"], 8))
    if kind == "layout":
        return _layout_work(case["k"], case["iters"])
    if kind == "energy":
        k, elem = case["k"], 8 if case["dtype"] == "float64" else 4
        # forward reads PDist; backward reads it again (nothing is kept) and writes its gradient
        return {"bytes": elem * (3.0 * k * k + 6.0 * k), "flops": 12.0 * k * k + 22.0 * k * k}
    if kind == "level":
        return _dppr_work(case["n"], 10.0 * case["n"], case["children"])
    if kind == "tau":
        # the index and the graph are read where mass arrives: at most all of it
        return {"bytes": 16.0 * case["n"] + 40.0 * case["n"], "flops": 2.0 * 10.0 * case["n"] * case["children"]}
    mean2 = (case["n_min"] ** 2 + case["n_min"] * case["n_max"] + case["n_max"] ** 2) / 3.0
    k = math.sqrt(mean2)
    one = _sum(_dppr_work(k, 0.013 * mean2, k), _layout_work(k, case["iters"]))
    return {key: v * case["count"] for key, v in one.items()}


# ---- the same results in 64 bits, in plain torch -----------------------------------------------------------------


def _walk(csr):
    """Transposed walk matrix as sparse CSR (row t: the nodes that step to t), and d(v); dangling nodes keep their walk."""
    rp, col, w = csr
    n = rp.shape[0] - 1
    cnt = rp[1:] - rp[:-1]
    src = torch.repeat_interleave(torch.arange(n, device=DEV), cnt)
    val = torch.ones(col.shape[0], dtype=torch.float64, device=DEV) if w is None else w.double()
    deg = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, src, val)
    val = val / deg[src]
    loop = torch.nonzero(cnt == 0)[:, 0]
    src = torch.cat([src, loop])
    dst = torch.cat([col.long(), loop])
    val = torch.cat([val, torch.ones(loop.shape[0], dtype=torch.float64, device=DEV)])
    order = torch.argsort(dst * n + src)
    trp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    trp[1:] = torch.cumsum(torch.bincount(dst, minlength=n), 0)
    return torch.sparse_csr_tensor(trp, src[order], val[order], (n, n)), deg


def _ppr(csr, start, chunk=1024):
    """Columns of sum_t alpha (1 - alpha)^t (P^T)^t start, and d."""
    pt, deg = _walk(csr)
    n = deg.shape[0]
    if n <= 6000 and csr[1].shape[0] > 0.02 * n * n:  # dense enough: a direct solve
        a = torch.eye(n, dtype=torch.float64, device=DEV) - (1.0 - ALPHA) * pt.to_dense()
        return ALPHA * torch.linalg.solve(a, start), deg
    steps = int(math.ceil(math.log(1e-15) / math.log(1.0 - ALPHA)))
    out = torch.empty_like(start)
    for a in range(0, start.shape[1], chunk):
        b = ALPHA * start[:, a:a + chunk].contiguous()
        x = b
        for _ in range(steps):
            x = b + (1.0 - ALPHA) * (pt @ x)
        out[:, a:a + chunk] = x
    return out, deg


def _pdist(dppr, n_clamp):
    z = dppr + dppr.T
    p = torch.clamp(torch.clamp(1.0 - torch.log(z), min=2.0), max=2.0 * math.log(n_clamp))
    p.fill_diagonal_(0.0)
    return p


def _dppr(csr, view=None, chunk=1024):
    n = csr[0].shape[0] - 1
    view = torch.arange(n, device=DEV) if view is None else view.long()
    k = view.shape[0]
    start = torch.zeros(n, k, dtype=torch.float64, device=DEV)
    start[view, torch.arange(k, device=DEV)] = 1.0
    x, deg = _ppr(csr, start, chunk)
    dppr = deg[view][:, None] * x[view].T
    return dppr, _pdist(dppr, n)


def _stress(delta, x):
    k = x.shape[0]
    d = torch.sqrt((x[:, None, 0] - x[None, :, 0]) ** 2 + (x[:, None, 1] - x[None, :, 1]) ** 2)
    off = ~torch.eye(k, dtype=torch.bool, device=DEV)
    e = torch.where(off, 1.0 - d / torch.where(off, delta, 1.0), 0.0)
    return 0.5 * (e * e).sum()


def _layout(delta, x0, iters):
    """Stress majorization X <- (L^w)^+ L^Y(X) X in 64 bits, centred, and the stress."""
    delta, x = delta.double(), x0.double()
    k = x.shape[0]
    w = 1.0 / ((delta + delta.T) / 2.0)
    w.fill_diagonal_(0.0)
    a = 1.0 / k - w * w
    a.diagonal().copy_((w * w).sum(1) + 1.0 / k)
    inv = torch.linalg.inv(a)
    del a
    for _ in range(iters):
        dx, dy = x[:, None, 0] - x[None, :, 0], x[:, None, 1] - x[None, :, 1]
        d = torch.sqrt(dx * dx + dy * dy)
        c = torch.where(d > 0, w / torch.where(d > 0, d, 1.0), 0.0)
        x = inv @ torch.stack([(c * dx).sum(1), (c * dy).sum(1)], 1)
    x = x - x.mean(0)
    return x, float(_stress(delta, x))


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    if kind in ("dppr", "directed", "dense"):
        return list(_dppr(s["csr"]))
    if kind == "subview":
        return list(_dppr(s["csr"], s["view"], chunk=64))
    if kind in ("view", "fp64"):
        # (the FP64 power iteration stops at eps, so its DPPR is off by up to that)
        dppr, pdist = _dppr(s["csr"])
        return [dppr, pdist, *_layout(pdist, s["x0"], case["iters"])]
    if kind == "layout":
        return list(_layout(s["delta"], s["x0"], case["iters"]))
    if kind == "energy":
        x, delta = s["x"].double(), s["delta"].double()
        k = x.shape[0]
        dx, dy = x[:, None, 0] - x[None, :, 0], x[:, None, 1] - x[None, :, 1]
        d = torch.sqrt(dx * dx + dy * dy)
        off = ~torch.eye(k, dtype=torch.bool, device=DEV)
        u = torch.where(off, 1.0 / torch.where(off, delta, 1.0), 0.0)
        e = torch.where(off, 1.0 - d * u, 0.0)
        c = torch.where(d > 0, -2.0 * e * u / torch.where(d > 0, d, 1.0), 0.0)
        return [0.5 * (e * e).sum(), torch.stack([(c * dx).sum(1), (c * dy).sum(1)], 1), e * d * u * u]
    if kind == "level":
        n, k, size = case["n"], case["children"], case["leaves"]
        rp = s["csr"][0]
        deg = (rp[1:] - rp[:-1]).double()
        ids, child = s["idx"].long(), torch.arange(k, device=DEV).repeat_interleave(size)
        start = torch.zeros(n, k, dtype=torch.float64, device=DEV)
        start[ids, child] = deg[ids] / size
        x, _ = _ppr(s["csr"], start)
        dppr = (x[ids].reshape(k, size, k).sum(1) / size).T.contiguous()
        return [dppr, _pdist(dppr, n)]
    if kind == "tau":
        return None  # an approximation within (eps, delta): no value is the exact one
    dists, xs, stresses, at = [], [], [], 0
    for csr in s["csrs"]:
        n = csr[0].shape[0] - 1
        pdist = _dppr(csr)[1]
        x, stress = _layout(pdist, s["x0"][at:at + n], case["iters"])
        dists.append(pdist.reshape(-1))
        xs.append(x)
        stresses.append(stress)
        at += n
    return [torch.cat(xs), torch.cat(dists), np.array(stresses)]
