"""The work a user of the t-SGNE library has it do, as timed cases.

Five kinds of case, each through the package's public calls:

  run      iterations of a layout whose P is built: initial layout (or a saved
           state) in, layout out; exact or tree-code repulsion
  grad     gradient of Eq. 5 and Z at a given layout (monitoring, parity,
           an optimiser of the user's own); FP32 or BF16 storage
  build    the joint affinities P of a new graph and its embedding:
           perplexity bisection or random walks, from device or host arrays
  embed    the ShortestPath embedding of a graph for d target nodes
  batch    a batch of mixed graphs advanced together, every layout read back

Sizes are those of the repository's benchmark, tests and serving trace: block
models of 500 to 3,000,000 nodes with mean degree 3 to 20 and R-MAT graphs up
to 2^21 nodes.  Graphs, embeddings and layouts are drawn on the GPU.
"""

import ctypes
import math

import numpy as np
import torch

import paper_2310_11186_gb300 as tsgne

DEV = "cuda"


def listed():
    return [
        # a few steps of a small graph's layout, as an interactive view runs them: the benchmark's 2,000-node block model
        {"name": "run_sbm2k", "kind": "run", "graph": "sbm", "n": 2000, "deg": 10.0, "blocks": 10, "d": 128,
         "perp": 30.0, "tree": False, "iters": 15, "resume": True},
        # a medium graph of the serving trace, exact repulsion, an odd size
        {"name": "run_sbm20k", "kind": "run", "graph": "sbm", "n": 20011, "deg": 6.0, "blocks": 25, "d": 64,
         "perp": 30.0, "tree": False, "iters": 8, "resume": True},
        # the benchmark's headline graph, exact repulsion
        {"name": "run_zipf300k", "kind": "run", "graph": "zipf", "n": 300000, "deg": 6.67, "blocks": 50, "d": 128,
         "perp": 30.0, "tree": False, "iters": 2, "resume": False},
        # the same graph with the tree code, resumed from a spread-out layout (where most iterations are spent)
        {"name": "run_tree300k", "kind": "run", "graph": "zipf", "n": 300000, "deg": 6.67, "blocks": 50, "d": 128,
         "perp": 30.0, "tree": True, "iters": 5, "resume": True},
        # the largest: a power-law graph of 2^21 nodes and 2^24 edges, tree code
        {"name": "run_rmat21", "kind": "run", "graph": "rmat", "n": 1 << 21, "deg": 16.0, "blocks": 64, "d": 64,
         "perp": 30.0, "tree": True, "iters": 4, "resume": True},
        # one gradient of the smallest size that the server hands to the tree code
        {"name": "grad_tree20k", "kind": "grad", "graph": "sbm", "n": 20011, "deg": 6.0, "blocks": 25, "d": 32,
         "perp": 30.0, "tree": True, "bf16": False},
        # one exact gradient on a power-law graph (hub rows of thousands of entries) with BF16 storage
        {"name": "grad_rmat16_bf16", "kind": "grad", "graph": "rmat", "n": 1 << 16, "deg": 16.0, "blocks": 64, "d": 32,
         "perp": 30.0, "tree": False, "bf16": True},
        # P of the headline graph from device arrays (an embedding computed on the GPU)
        {"name": "build_zipf300k", "kind": "build", "graph": "zipf", "n": 300000, "deg": 6.67, "blocks": 50, "d": 128,
         "perp": 30.0, "walks": 0, "length": 3, "host": False},
        # P from host arrays with a perplexity below the degrees, so that every row is searched; d not a multiple of 4
        {"name": "build_perp5_host", "kind": "build", "graph": "sbm", "n": 50021, "deg": 17.3, "blocks": 40, "d": 50,
         "perp": 5.0, "walks": 0, "length": 3, "host": True},
        # P by the paper's random walks (Eq. 6) and the first gradient on it
        {"name": "build_walks300k", "kind": "build", "graph": "zipf", "n": 300000, "deg": 6.67, "blocks": 50, "d": 64,
         "perp": 30.0, "walks": 64, "length": 3, "host": False},
        # the paper's own embedding (Eq. 8) of the headline graph
        {"name": "embed_zipf300k", "kind": "embed", "graph": "zipf", "n": 300000, "deg": 6.67, "blocks": 50, "d": 128},
        # a batch of small and medium graphs advanced together
        {"name": "batch32", "kind": "batch", "count": 32, "lo": 500, "hi": 20000, "deg": 6.0, "d": 64, "perp": 30.0,
         "iters": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "grad", "build", "build", "embed", "batch"])
    if kind == "batch":
        hi = _log_int(rng, 2000, 20000)
        return {"kind": "batch", "count": rng.randint(6, 40), "lo": 500, "hi": hi, "deg": round(rng.uniform(4, 12), 2),
                "d": rng.randint(16, 64), "perp": rng.choice([5.0, 30.0]), "iters": rng.randint(2, 6)}
    tree = kind in ("run", "grad") and rng.random() < 0.5
    lo, hi = (20000, 3000000) if tree else (500, 300000)
    if rng.random() < 0.25:
        scale = rng.randint(14, 21) if tree else rng.randint(10, 18)
        c = {"kind": kind, "graph": "rmat", "n": 1 << scale, "deg": float(rng.randint(6, 16)), "blocks": 64}
    else:
        c = {"kind": kind, "graph": rng.choice(["sbm", "zipf"]), "n": _log_int(rng, lo, hi),
             "deg": round(rng.uniform(3.3, 17.3), 2), "blocks": rng.randint(10, 50)}
    if kind == "run":
        # few iterations: rounding grows from one to the next (a layout's path is chaotic), and the exact passes'
        # work stays below the headline case's
        resume = not tree or rng.random() < 0.5
        most = (5 if resume else 10) if tree else max(2, min(10, int(1.8e11 / c["n"] ** 2)))
        c.update(d=rng.choice([32, 64, 128]), perp=rng.choice([5.0, 30.0]), tree=tree,
                 iters=max(2, min(most, int(5e6 / c["n"]) if tree else most)), resume=resume)
    elif kind == "grad":
        c.update(d=rng.choice([32, 64]), perp=rng.choice([5.0, 30.0]), tree=tree, bf16=rng.random() < 0.5)
    elif kind == "build":
        c.update(d=rng.randint(16, 128), perp=rng.choice([2.0, 5.0, 30.0]),
                 walks=rng.choice([0, 0, rng.randint(8, 96)]), length=rng.randint(1, 5), host=rng.random() < 0.5)
    else:
        c.update(d=rng.randint(1, 256))
    return c


# ------------------------------------------------------------------ inputs

def _block_sizes(case):
    n, b = case["n"], max(1, min(case["blocks"], case["n"] // 64))
    if case["graph"] == "zipf":
        w = np.arange(1, b + 1, dtype=np.float64) ** -1.2
    else:
        w = np.ones(b)
    s = np.maximum(8, np.floor(n * w / w.sum())).astype(np.int64)
    s[0] += n - s.sum()
    return s


def _draw_edges(case, m, gen, blocks):
    n = case["n"]
    if case["graph"] == "rmat":
        u = torch.zeros(m, dtype=torch.int64, device=DEV)
        v = torch.zeros(m, dtype=torch.int64, device=DEV)
        for _ in range(n.bit_length() - 1):  # quadrants with probabilities 0.57, 0.19, 0.19, 0.05
            r = torch.rand(m, device=DEV, generator=gen)
            u = 2 * u + (r >= 0.76)
            v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    else:
        labels, start, sizes = blocks
        u = torch.randint(n, (m,), device=DEV, generator=gen)
        b = labels[u]
        v = start[b] + (torch.rand(m, device=DEV, dtype=torch.float64, generator=gen) * sizes[b]).long()
        far = torch.rand(m, device=DEV, generator=gen) < 0.10  # a tenth of the edges leave their block
        v = torch.where(far, torch.randint(n, (m,), device=DEV, generator=gen), v)
    return (torch.minimum(u, v) * n + torch.maximum(u, v))[u != v]


def _graph(case, gen):
    """(row_ptr, col, labels): a symmetric CSR of exactly n deg / 2 edges
    without loops or repeats, on the GPU."""
    n = case["n"]
    m = int(round(n * case["deg"] / 2))
    if case["graph"] == "rmat":
        blocks = None
        labels = torch.arange(n, device=DEV) >> max(0, n.bit_length() - 7)
    else:
        s = _block_sizes(case)
        sizes = torch.from_numpy(s).to(DEV)
        start = torch.from_numpy(np.concatenate([[0], np.cumsum(s)[:-1]])).to(DEV)
        labels = torch.repeat_interleave(torch.arange(len(s), device=DEV), sizes)
        blocks = (labels, start, sizes)
    key = torch.empty(0, dtype=torch.int64, device=DEV)
    while key.numel() < m:
        key = torch.unique(torch.cat([key, _draw_edges(case, m + m // 8 + 64, gen, blocks)]))
    drop = torch.rand(key.numel(), device=DEV, generator=gen).argsort()[m:]
    keep = torch.ones(key.numel(), dtype=torch.bool, device=DEV)
    keep[drop] = False
    key = key[keep]
    u, v = key // n, key % n
    key = torch.cat([key, v * n + u]).sort().values
    rp = torch.searchsorted(key, torch.arange(n + 1, device=DEV) * n)
    return rp, (key % n).to(torch.int32), labels


def _spread(labels, k, std, gen):
    """Points around their block's centre: centres N(0, std^2), points N(0, 1) around them."""
    c = std * torch.randn(int(labels.max()) + 1, k, device=DEV, generator=gen)
    return c[labels] + torch.randn(labels.numel(), k, device=DEV, generator=gen)


def _members(case, seed):
    for k in range(case["count"]):  # sizes log-uniform in [lo, hi]
        n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** ((k + 0.5) / case["count"])))
        yield {"kind": "run", "graph": "sbm", "n": n, "deg": case["deg"], "blocks": 5 + 7 * k % 36,
               "d": case["d"], "resume": True}, seed * 1000 + k


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rp, col, labels = _graph(case, gen)
    x = {"rp": rp, "col": col}
    if case["kind"] == "embed":
        x["targets"] = torch.randint(case["n"], (case["d"],), device=DEV, generator=gen).to(torch.int32)
        return x
    x["X"] = _spread(labels, case["d"], 2.0, gen)
    if case["kind"] == "grad" or case.get("resume") or case.get("walks"):
        x["Y"] = _spread(labels, 2, 30.0, gen)
    elif case["kind"] == "run":
        x["Y"] = 1e-4 * torch.randn(case["n"], 2, device=DEV, generator=gen)
    return x


def prepare(case, seed):
    if case["kind"] == "batch":
        b = tsgne.Batch(perplexity=case["perp"])
        st = {"case": case, "batch": b, "ids": [], "out": []}
        for c, s in _members(case, seed):
            x = _inputs(c, s)
            torch.cuda.synchronize()
            st["ids"].append(b.add(x["rp"], x["col"], x["X"], x["Y"]))
            st["out"].append(torch.empty(c["n"], 2, device=DEV))
        return st
    x = _inputs(case, seed)
    st = {"case": case, "x": x}
    if case["kind"] in ("run", "grad"):
        lay = tsgne.Layout(perplexity=case["perp"], repulsion=int(case["tree"]), precision=int(case.get("bf16", False)))
        lay.build_P(x["rp"], x["col"], x.pop("X"))
        if case["kind"] == "grad":
            lay.init_Y(x["Y"])
        st.update(lay=lay, out=torch.empty(case["n"], 2, device=DEV))
    elif case["kind"] == "build":
        st["out"] = torch.empty(case["n"], 2, device=DEV)
        if case["host"]:
            st["x"] = {k: v.cpu().numpy() for k, v in x.items()}
            st["out"] = st["out"].cpu().numpy()
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "batch":
        b = st["batch"]
        b.reset()
        b.run(case["iters"])
        return [b.get_Y(i, out=o)[0] for i, o in zip(st["ids"], st["out"])]
    x = st["x"]
    if case["kind"] == "run":
        lay = st["lay"]
        if case["resume"]:
            lay.set_state(x["Y"], iteration=300)
        else:
            lay.init_Y(x["Y"])
        lay.run(case["iters"])
        return lay.get_Y(out=st["out"])
    if case["kind"] == "grad":
        return st["lay"].gradient(1.0, out=st["out"])
    if case["kind"] == "embed":
        return tsgne.tsgne_shortest_path_embedding(x["rp"], x["col"], x["targets"])
    with tsgne.Layout(perplexity=case["perp"], p_walks=case["walks"], p_walk_length=case["length"],
                      repulsion=int(case["walks"] > 0)) as lay:
        lay.build_P(x["rp"], x["col"], x["X"])
        if case["walks"]:  # the structure is the walks' own: the first gradient on it
            lay.init_Y(x["Y"])
            return lay.gradient(1.0, out=st["out"])
        if case["host"]:
            return lay.get_P()
        n, nnz = lay.sizes()  # device arrays through the C call
        rp = torch.empty(n + 1, dtype=torch.int64, device=DEV)
        col = torch.empty(nnz, dtype=torch.int32, device=DEV)
        val = torch.empty(nnz, device=DEV)
        p = [ctypes.c_void_p(t.data_ptr()) for t in (rp, col, val)]
        st_ = tsgne.lib().tsgne_get_P(lay.ctx, *p, tsgne.PTR_DEVICE)
        if st_ != 0:
            raise tsgne.TsgneError(st_, tsgne.tsgne_last_error(lay.ctx))
        return rp, col, val


# ----------------------------------------------------------- cost of a pass

def _layout_work(case):
    """One iteration: 16 flops per unordered pair (or, tree code, per
    interaction: about 18 log2 n of them a point), 10 per entry, 30 per point."""
    n, nnz = case["n"], case["n"] * case["deg"]
    pairs = 18.0 * math.log2(n) * n if case.get("tree") else 0.5 * n * (n - 1.0)
    return 8.0 * nnz + 56.0 * n, 16.0 * pairs + 10.0 * nnz + 30.0 * n


def work(case):
    if case["kind"] == "batch":
        lo, hi = case["lo"], case["hi"]
        b = f = 0.0
        for q in range(16):
            n = lo * (hi / lo) ** ((q + 0.5) / 16)
            w = _layout_work({"n": n, "deg": case["deg"]})
            b += w[0] / 16
            f += w[1] / 16
        k = case["count"] * case["iters"]
        return {"bytes": k * b, "flops": k * f}
    n, nnz = case["n"], case["n"] * case["deg"]
    if case["kind"] in ("run", "grad"):
        b, f = _layout_work(case)
        it = case.get("iters", 1)
        return {"bytes": it * b, "flops": it * f}
    if case["kind"] == "embed":
        return {"bytes": 8.0 * n + 4.0 * nnz + 4.0 * n * case["d"], "flops": 0.0}
    # graph and X in; structure and P out
    b = 16.0 * n + 12.0 * nnz + 4.0 * n * case["d"]
    return {"bytes": b, "flops": 3.0 * nnz * case["d"]}


# ------------------------------------------------------------- exact values

def _exact_P(rp, col, X, perp):
    """Eqs. 2-3 in FP64: bisection on beta per row (uniform rows where the
    degree does not exceed the perplexity), then the symmetrised joint P."""
    n = rp.numel() - 1
    deg = rp[1:] - rp[:-1]
    row = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    c = col.long()
    d2 = torch.empty(c.numel(), dtype=torch.float64, device=DEV)
    for a in range(0, c.numel(), 1 << 20):
        s = slice(a, a + (1 << 20))
        d2[s] = (X[row[s]].double() - X[c[s]].double()).square().sum(1)

    def seg(v):
        return torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, v)

    big = torch.full((n,), math.inf, dtype=torch.float64, device=DEV)
    delta = d2 - big.scatter_reduce(0, row, d2, "amin")[row]
    target = math.log(perp)
    beta = torch.ones(n, dtype=torch.float64, device=DEV)
    lo, hi = torch.full_like(beta, -math.inf), torch.full_like(beta, math.inf)
    done = deg.double() <= perp
    for _ in range(99):
        w = torch.exp(-beta[row] * delta)
        S = seg(w)
        H = torch.log(S) + beta * seg(delta * w) / S
        done = done | ((H - target).abs() <= float(np.float32(1e-5)))
        if bool(done.all()):
            break
        up = H > target
        lo = torch.where(up & ~done, beta, lo)
        hi = torch.where(~up & ~done, beta, hi)
        nb = torch.where(up, torch.where(torch.isinf(hi), 2 * beta, 0.5 * (beta + hi)),
                         torch.where(torch.isinf(lo), 0.5 * beta, 0.5 * (beta + lo)))
        beta = torch.where(done, beta, nb)
    w = torch.exp(-beta[row] * delta)
    p = w / seg(w)[row]
    p = torch.where((deg.double() <= perp)[row], 1.0 / deg.double()[row], p)
    t = torch.searchsorted(row * n + c, c * n + row)  # position of (j, i)
    v = p + p[t]
    return row, c, v / v.sum()


def _exact_force(row, c, P, Y, alpha):
    """(gradient of Eq. 5 with P scaled by alpha, Z), every pair summed."""
    n = Y.shape[0]
    x, y = Y[:, 0].contiguous(), Y[:, 1].contiguous()
    F = torch.empty_like(Y)
    Z = 0.0
    step = max(1, int(1.5e8 // n))
    for a in range(0, n, step):
        dx = x[a:a + step, None] - x[None, :]
        dy = y[a:a + step, None] - y[None, :]
        w = (dx * dx).addcmul_(dy, dy).add_(1.0).reciprocal_()
        Z += float(w.sum())
        w.mul_(w)
        F[a:a + step, 0] = dx.mul_(w).sum(1)
        F[a:a + step, 1] = dy.mul_(w).sum(1)
    Z -= n
    e = Y[row] - Y[c]
    pw = (P / (1.0 + e.square().sum(1)))[:, None] * e
    A = torch.zeros_like(Y).index_add_(0, row, pw)
    return 4.0 * (alpha * A - F / Z), Z


def _exact_run(row, c, P, Y, iters, first):
    n = Y.shape[0]
    eta = float(max(np.float32(n) / np.float32(12.0) / np.float32(4.0), np.float32(50.0)))
    u, gain = torch.zeros_like(Y), torch.ones_like(Y)
    for t in range(first, first + iters):
        g, _ = _exact_force(row, c, P, Y, 12.0 if t < 250 else 1.0)
        gain = torch.where(g * u < 0, gain + 0.2, gain * 0.8).clamp_min(float(np.float32(0.01)))
        u = (0.5 if t < 250 else 0.8) * u - eta * gain * g
        Y = Y + u
    return Y


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for c, s in _members(case, seed):
            x = _inputs(c, s)
            out.append(_exact_run(*_exact_P(x["rp"], x["col"], x["X"], case["perp"]), x["Y"].double(), case["iters"], 0))
        return out
    if case["kind"] in ("run", "grad") and case["n"] ** 2 * case.get("iters", 1) > 2e11:
        return None  # minutes in FP64
    if case.get("walks"):
        return None  # a sampled estimate: its values are the counts of the library's own draws
    x = _inputs(case, seed)
    rp, col = x["rp"], x["col"]
    n = case["n"]
    if case["kind"] == "embed":
        l0 = int(math.sqrt(col.numel() // 2))
        A = torch.sparse_csr_tensor(rp, col.long(), torch.ones(col.numel(), device=DEV), size=(n, n))
        D = torch.full((n, case["d"]), float(l0 + 1), dtype=torch.float64, device=DEV)
        k = torch.arange(case["d"], device=DEV)
        new = torch.zeros(n, case["d"], device=DEV)
        new[x["targets"].long(), k] = 1.0
        D[x["targets"].long(), k] = 0.0
        seen = new > 0
        for level in range(1, l0 + 1):
            fresh = ((A @ new) > 0) & ~seen
            if not bool(fresh.any()):
                break
            D[fresh] = float(level)
            seen |= fresh
            new = fresh.float()
        return D
    row, c, P = _exact_P(rp, col, x["X"], case["perp"])
    if case["kind"] == "build":
        return None, None, P
    if case["kind"] == "grad":
        return _exact_force(row, c, P, x["Y"].double(), 1.0)
    return _exact_run(row, c, P, x["Y"].double(), case["iters"], 300 if case["resume"] else 0)
