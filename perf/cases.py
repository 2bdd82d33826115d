"""The work that users of this package have it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``prepare`` makes its inputs on the GPU from a seed (graph,
weights, scores) and the handle a program keeps, ``run`` makes one pass through the public entry
points, ``work`` counts the bytes and operations of a pass, and ``exact`` gives the computed
numbers in FP64 by plain torch.

Ranges (what ``listed`` samples and ``draw`` draws from):
  distance   Alg. 1 on one graph: 4-neighbour grids of 32^2 .. 1024^2 vertices, R-MAT of 2^12 .. 2^20
             vertices with 12 to 15 edges per vertex, Barabasi-Albert of 3K .. 1M vertices with about 8;
             R = 4 .. 48 test vectors, k = 5 .. 40 sweeps, FP32, FP16, BF16 or Q16 storage, unit or
             lognormal weights, plain or normalised scores
  batch      the same on a batch of 4 .. 128 Watts-Strogatz graphs of 1K .. 200K vertices in one handle
  select     ranking and sampling on scores the program has: per node (Alg. 2, local or global), whole
             graph, the binned mixture (Alg. 3) and Local Degree, 10% .. 70% kept, on the graphs above
  grad       forward and backward of the distances in the edge weights, R-MAT of 2^12 .. 2^22 vertices
  multilevel Alg. 6 in one call, Barabasi-Albert of 20K .. 2M vertices
  host       graph from host arrays, distances, both per-node selections, results on the host
"""
import math

import numpy as np
import torch

from paper_1601_05527_gb300 import Graph, _lib as L
from paper_1601_05527_gb300.autograd import algebraic_distance

OMEGA = 0.5


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # one small mesh: the call's latency and its launches are what count
        {"name": "grid64_distance", "kind": "distance", "graph": "grid", "n": 4096, "m": 8064, "R": 8, "k": 20,
         "storage": "fp32", "weighted": False, "normalize": False},
        # a social network of a million vertices, the headline size, full precision
        {"name": "rmat20_distance_fp32", "kind": "distance", "graph": "rmat", "n": 1 << 20, "m": 15_700_000, "R": 32,
         "k": 20, "storage": "fp32", "weighted": False, "normalize": False},
        # the same network with the 16-bit storage that is recommended where distances feed a selection
        {"name": "rmat20_distance_fp16", "kind": "distance", "graph": "rmat", "n": 1 << 20, "m": 15_700_000, "R": 32,
         "k": 20, "storage": "fp16", "weighted": False, "normalize": False},
        # the paper's own parameters (R = 10, k = 40) and its normalised score on a weighted network: a
        # number of vectors that fills no power of two, an odd number of vertices
        {"name": "ba200k_distance_paper", "kind": "distance", "graph": "ba", "n": 200_003, "m": 1_590_001, "R": 10,
         "k": 40, "storage": "fp32", "weighted": True, "normalize": True},
        # many small-world networks analysed together in one handle, 16-bit storage
        {"name": "ws128_batch_bf16", "kind": "batch", "graph": "ws", "graphs": 128, "n": 12_800_000, "m": 63_600_000,
         "R": 16, "k": 15, "storage": "bf16", "weighted": False, "normalize": False},
        # each network of such a batch reduced to a quarter of its edges, long-range edges first
        {"name": "ws128_select_global", "kind": "select", "method": "per_node", "mode": "global", "fraction": 0.25,
         "graph": "ws", "graphs": 128, "n": 12_800_000, "m": 63_600_000},
        # Alg. 2 on a social network: every node keeps its closest neighbours
        {"name": "rmat20_select_local", "kind": "select", "method": "per_node", "mode": "local", "fraction": 0.3,
         "graph": "rmat", "n": 1 << 20, "m": 15_700_000},
        # one threshold for the whole network
        {"name": "rmat20_select_whole", "kind": "select", "method": "whole_graph", "mode": "global", "fraction": 0.5,
         "graph": "rmat", "n": 1 << 20, "m": 15_700_000},
        # the binned mixture of Alg. 3
        {"name": "rmat19_select_binned", "kind": "select", "method": "binned", "mode": "local", "fraction": 0.3,
         "graph": "rmat", "n": 1 << 19, "m": 7_800_000},
        # learning edge weights through the distances: forward and backward at the largest size
        {"name": "rmat22_grad", "kind": "grad", "graph": "rmat", "n": 1 << 22, "m": 64_000_000, "R": 32, "k": 30,
         "weighted": True},
        # the multilevel method end to end on a weighted network of two million vertices
        {"name": "ba2m_multilevel", "kind": "multilevel", "graph": "ba", "n": 2_000_000, "m": 15_960_000, "R": 16,
         "k": 20, "weighted": True, "fraction": 0.4, "coarsest_n": 1000},
        # a program that starts from host arrays and wants the sparsified graph back on the host
        {"name": "rmat20_from_host", "kind": "host", "graph": "rmat", "n": 1 << 20, "m": 15_700_000, "R": 32, "k": 20,
         "weighted": False, "fraction": 0.3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, families, biggest):
    f = rng.choice(families)
    if f == "rmat":
        n = 1 << rng.randint(12, int(math.log2(biggest)))
        return {"graph": f, "n": n, "m": int(n * rng.uniform(12.0, 15.0)) - rng.randint(0, 63)}
    if f == "grid":
        a, b = _log(rng, 32, 1024), _log(rng, 32, 1024)
        return {"graph": f, "n": a * b, "rows": a, "m": a * (b - 1) + b * (a - 1)}
    if f == "ws":
        graphs = _log(rng, 4, 128)
        n = graphs * _log(rng, 2000, 100_000) + rng.randint(0, 99)
        return {"graph": f, "graphs": graphs, "n": n, "m": int(4.95 * n)}
    n = _log(rng, 3001, biggest) | 1
    return {"graph": f, "n": n, "m": int(7.9 * n) - 40}


def draw(rng):
    kind = rng.choice(["distance", "distance", "batch", "select", "select", "select", "grad", "multilevel", "host"])
    if kind == "distance":
        c = _draw_graph(rng, ["rmat", "ba", "grid"], 1 << 20)
        weighted = rng.random() < 0.5
        return {"kind": kind, **c, "R": _log(rng, 4, 48), "k": rng.randint(5, 40),
                "storage": rng.choice(["fp32", "fp32", "fp16", "bf16", "q16"]), "weighted": weighted,
                "normalize": rng.random() < 0.25}
    if kind == "batch":
        c = _draw_graph(rng, ["ws"], 0)
        return {"kind": kind, **c, "R": _log(rng, 4, 32), "k": rng.randint(5, 20),
                "storage": rng.choice(["fp32", "bf16", "bf16", "fp16"]), "weighted": rng.random() < 0.3,
                "normalize": False}
    if kind == "select":
        method = rng.choice(["per_node", "per_node", "whole_graph", "binned", "local_degree"])
        c = _draw_graph(rng, ["rmat", "ba", "ws"], 1 << 20)
        return {"kind": kind, "method": method, "mode": rng.choice(["local", "global"]),
                "fraction": round(rng.uniform(0.1, 0.7), 3), **c}
    if kind == "grad":
        return {"kind": kind, **_draw_graph(rng, ["rmat", "ba"], 1 << 20), "R": _log(rng, 4, 32),
                "k": rng.randint(5, 30), "weighted": True}
    if kind == "multilevel":
        n = _log(rng, 20_000, 1_000_000) | 1
        return {"kind": kind, "graph": "ba", "n": n, "m": int(7.9 * n), "R": _log(rng, 8, 32), "k": rng.randint(5, 20),
                "weighted": rng.random() < 0.5, "fraction": round(rng.uniform(0.2, 0.6), 3), "coarsest_n": 1000}
    return {"kind": kind, **_draw_graph(rng, ["rmat", "ba"], 1 << 20), "R": _log(rng, 4, 32), "k": rng.randint(5, 20),
            "weighted": rng.random() < 0.5, "fraction": round(rng.uniform(0.1, 0.6), 3)}


# --------------------------------------------------------------------------- inputs
_stream = None


def _context():
    """One stream of our own for everything, and the package's memory from torch's allocator."""
    global _stream
    if _stream is None:
        L.use_torch_allocator()
        _stream = torch.cuda.Stream()
    return torch.cuda.stream(_stream)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & (2**62 - 1))


def _rmat_pairs(n, count, g):
    scale = n.bit_length() - 1
    src = torch.zeros(count, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        r = torch.rand(count, device="cuda", generator=g)
        src = src * 2 + (r >= 0.76)
        dst = dst * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return src, dst


def _ba_pairs(n, g, per=8):
    """Preferential attachment by uniform picks from the list of earlier edges' ends."""
    m0 = per + 1
    clique = torch.triu_indices(m0, m0, 1, device="cuda")
    nc, new = clique.shape[1], (n - m0) * per
    src = torch.cat([clique[0], torch.arange(m0, n, device="cuda").repeat_interleave(per)])
    first = nc + (src[nc:] - m0) * per
    pos = (torch.rand(new, device="cuda", dtype=torch.float64, generator=g) * (2 * first)).long()
    even, old = pos % 2 == 0, pos // 2
    dst = torch.cat([clique[1], torch.where(even, src[old], torch.full_like(old, -1))])
    ptr = torch.cat([torch.arange(nc, device="cuda"), old])       # the edge whose far end is copied
    while True:
        left = dst < 0
        if not bool(left.any()):
            return src, dst
        dst = torch.where(left, dst[ptr], dst)
        ptr = torch.where(left, ptr[ptr], ptr)


def _ws_offsets(case):
    """Sizes of the batch's graphs: uneven, the same for every seed, n vertices in all."""
    G = case["graphs"]
    share = np.random.RandomState(G).uniform(0.01, 2.0, G)
    cut = np.floor(np.cumsum(share) / share.sum() * case["n"]).astype(np.int64)
    cut[-1] = case["n"]
    return np.concatenate([[0], cut])


def _ws_pairs(voff, n, g, per=5, p=0.1):
    off = torch.from_numpy(voff).cuda()
    size = (off[1:] - off[:-1]).repeat_interleave(off[1:] - off[:-1]).repeat_interleave(per)
    base = off[:-1].repeat_interleave(off[1:] - off[:-1]).repeat_interleave(per)
    u = torch.arange(n, device="cuda").repeat_interleave(per)
    step = torch.arange(1, per + 1, device="cuda").repeat(n)
    far = torch.where(torch.rand(n * per, device="cuda", generator=g) < p,
                      (torch.rand(n * per, device="cuda", dtype=torch.float64, generator=g) * size).long(),
                      (u - base + step) % size)
    return u, base + far


def _graph(case, seed):
    """The undirected simple graph of a case as a symmetric CSR with exactly m edges, and the edge id
    of every entry; columns ascend in each row, edge ids ascend in (smaller end, larger end)."""
    n, m, g = case["n"], case["m"], _generator(seed)
    voff = _ws_offsets(case) if case["graph"] == "ws" else None
    if case["graph"] == "grid":
        a = case.get("rows", math.isqrt(n))
        i = torch.arange(n, device="cuda").view(a, n // a)
        u, v = torch.cat([i[:, :-1].reshape(-1), i[:-1].reshape(-1)]), torch.cat([i[:, 1:].reshape(-1), i[1:].reshape(-1)])
    elif case["graph"] == "ba":
        u, v = _ba_pairs(n, g)
    elif case["graph"] == "ws":
        u, v = _ws_pairs(voff, n, g)
    else:
        u, v = _rmat_pairs(n, m + m // 6, g)
    keys = None
    while True:
        k = (torch.minimum(u, v) * n + torch.maximum(u, v))[u != v]
        keys = torch.unique(k if keys is None else torch.cat([keys, k]))
        if len(keys) >= m or case["graph"] != "rmat":
            break
        u, v = _rmat_pairs(n, m // 3, g)
    if len(keys) < m:
        raise ValueError("the graph has %d edges, %d are wanted" % (len(keys), m))
    if len(keys) > m:   # a random surplus goes, so that every seed has the same size
        keys = keys[torch.rand(len(keys), device="cuda", generator=g).argsort()[:m]].sort().values
    lo, hi = keys // n, keys % n
    both, order = torch.cat([lo * n + hi, hi * n + lo]).sort()
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(both // n, minlength=n).cumsum(0)
    eid = order % m
    weight = None
    if case.get("weighted"):   # heavy-tailed interaction strengths; 0.5 .. 2 where weights are learned
        weight = (torch.rand(m, device="cuda", generator=g) * 1.5 + 0.5 if case["kind"] == "grad"
                  else torch.randn(m, device="cuda", generator=g).exp())
    return {"row_ptr": row_ptr, "col": (both % n).int(), "eid": eid, "lo": lo, "hi": hi, "weight": weight, "voff": voff}


def _scores(m, seed):
    """Scores like distances: positive, skewed, FP32."""
    g = _generator(seed + 1)
    return (torch.randn(m, device="cuda", generator=g) * 0.8 - 4.0).exp()


def _loss_edges(m, seed):
    return (torch.rand(m, device="cuda", generator=_generator(seed + 2)) < 0.01).nonzero().flatten()


def _vectors_seed(seed):
    return (0x1601055270000000 + int(seed)) & (2**64 - 1)


def prepare(case, seed):
    with _context():
        s = {"case": case, "seed": _vectors_seed(seed)}
        c = _graph(case, seed)
        m, kind = case["m"], case["kind"]
        if kind == "host":
            for key in ("row_ptr", "col", "weight"):
                x = c[key]
                if key == "weight" and x is not None:
                    x = x[c["eid"]]
                s[key] = None if x is None else x.cpu().pin_memory()
            s["rho"] = torch.empty(m, dtype=torch.float32).pin_memory()
            s["keep"] = [torch.empty(m, dtype=torch.uint8).pin_memory() for _ in range(2)]
            return s
        w = c["weight"]
        s["graph"] = Graph(c["row_ptr"], c["col"], None if w is None else w[c["eid"]], n=case["n"],
                           vertex_offset=c["voff"], stream=_stream)
        if kind in ("distance", "batch"):
            s["rho"] = torch.empty(m, dtype=torch.float32, device="cuda")
        elif kind == "select":
            s["keep"] = torch.empty(m, dtype=torch.uint8, device="cuda")
            s["scores"] = None if case["method"] == "local_degree" else _scores(m, seed)
        elif kind == "grad":
            s["w"] = w.requires_grad_(True)
            s["loss_edges"] = _loss_edges(m, seed)
        elif kind == "multilevel":
            s["keep"] = torch.empty(m, dtype=torch.uint8, device="cuda")
        return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    with torch.cuda.stream(_stream):
        if kind in ("distance", "batch"):
            s["graph"].algebraic_distance(case["R"], case["k"], OMEGA, s["seed"], storage=case["storage"],
                                          normalize=case["normalize"], out=s["rho"])
            return {"rho": s["rho"]}
        if kind == "select":
            if case["method"] == "binned":
                kept, e = L.ad_sparsify_binned(s["graph"].handle, s["scores"], case["fraction"], s["seed"], s["keep"])
            elif case["method"] == "local_degree":
                kept, e = L.ad_sparsify_local_degree(s["graph"].handle, case["fraction"], s["keep"])
            else:
                _, kept, e = s["graph"].sparsify(case["fraction"], case["mode"], case["method"], s["keep"], s["scores"])
            return {"keep": s["keep"], "kept": kept, "e": e}
        if kind == "grad":
            s["w"].grad = None
            rho = algebraic_distance(s["w"], s["graph"], case["R"], case["k"], OMEGA, s["seed"])
            rho[s["loss_edges"]].square().sum().backward()
            return {"rho": rho.detach(), "w_grad": s["w"].grad}
        if kind == "multilevel":
            levels = L.ad_multilevel(s["graph"].handle, [1.0, 1.0], case["fraction"], s["keep"], R=case["R"], k=case["k"],
                                     omega=OMEGA, seed=s["seed"], Q=0.5, coarsest_n=case["coarsest_n"], mode="local")
            return {"keep": s["keep"], "levels": levels}
        with Graph(s["row_ptr"], s["col"], s["weight"], n=case["n"], stream=_stream) as g:
            g.algebraic_distance(case["R"], case["k"], OMEGA, s["seed"], out=s["rho"])
            kept, e = L.ad_sparsify_local_global(g.handle, case["fraction"], *s["keep"])
        return {"rho": s["rho"], "keep_local": s["keep"][0], "keep_global": s["keep"][1], "kept": kept, "e": e}


def work(case):
    n, m = case["n"], case["m"]
    nnz = 2 * m
    csr = 8 * (n + 1) + 4 * nnz
    weights = 4 * nnz if case.get("weighted") else 0
    kind = case["kind"]
    if kind == "select":   # scores in, one byte per edge out
        return {"bytes": csr + (0 if case["method"] == "local_degree" else 4 * m) + m, "flops": 0}
    R, k = case["R"], case["k"]
    sweep = 2 * nnz * R + 3 * n * R
    relax = k * sweep + 3 * m * R
    if kind == "grad":     # weights in once per edge, distances and gradient out; the adjoint gathers twice
        return {"bytes": csr + 4 * m + 8 * m, "flops": relax + k * (2 * sweep) + 6 * m * R}
    if kind == "multilevel":
        return {"bytes": csr + weights + m, "flops": relax}
    out = 4 * m + (2 * m if kind == "host" else 0)
    return {"bytes": csr + weights + out, "flops": relax}


# --------------------------------------------------------------------------- FP64 values
def _philox(c0, c2, c3, key):
    """Word 0..3 of Philox4x32-10 for int64 tensors of counter words 0 and 2 (word 1 is zero)."""
    M = 0xFFFFFFFF

    def mul(a, b):
        t = (a >> 16) * b + (((a & 0xFFFF) * b) >> 16)
        return t >> 16, (a * b) & M
    c = [c0, torch.zeros_like(c0), c2, torch.full_like(c0, c3)]
    k0, k1 = key & M, key >> 32
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c


def _start_vectors(n, R, key, voff):
    i = torch.arange(n, device="cuda")
    if voff is not None:
        off = torch.from_numpy(voff).cuda()
        i = i - off[:-1].repeat_interleave(off[1:] - off[:-1])
    x = torch.empty(n, R, dtype=torch.float64, device="cuda")
    for q in range((R + 3) // 4):
        for j, word in enumerate(_philox(i, torch.full_like(i, q), 0, key)):
            if 4 * q + j < R:
                x[:, 4 * q + j] = (word >> 8).double() * 2.0**-24 - 0.5
    return x


class _Exact:
    """FP64 sweeps of Alg. 1 with a rescale after each."""

    def __init__(self, case, seed):
        c = _graph(case, seed)
        self.n, self.m, self.R, self.k = case["n"], case["m"], case["R"], case["k"]
        self.lo, self.hi, self.eid = c["lo"], c["hi"], c["eid"]
        self.row_ptr, self.col = c["row_ptr"], c["col"]
        w = torch.ones(2 * self.m, dtype=torch.float64, device="cuda") if c["weight"] is None else c["weight"].double()[c["eid"]]
        self.W = self.matrix(w)
        self.D = self.W @ torch.ones(self.n, 1, dtype=torch.float64, device="cuda")
        self.active = self.D[:, 0] > 0
        self.Dinv = torch.where(self.D > 0, 1 / self.D, torch.zeros_like(self.D))
        self.voff = [0, self.n] if c["voff"] is None else c["voff"].tolist()
        self.x0 = _start_vectors(self.n, self.R, _vectors_seed(seed), c["voff"])

    def matrix(self, values):
        return torch.sparse_csr_tensor(self.row_ptr.int(), self.col, values, (self.n, self.n), dtype=torch.float64,
                                       check_invariants=False)

    def rescale(self, y):
        """(y mapped onto [-1/2, 1/2] per vector and graph, minimum and maximum per graph)"""
        x, ends = torch.empty_like(y), []
        inf = math.inf
        for a, b in zip(self.voff[:-1], self.voff[1:]):
            on = self.active[a:b, None]
            lo = torch.where(on, y[a:b], inf).amin(0)
            hi = torch.where(on, y[a:b], -inf).amax(0)
            x[a:b] = torch.where(hi > lo, (y[a:b] - lo) / (hi - lo) - 0.5, torch.zeros_like(lo))
            ends.append((lo, hi))
        return x, ends

    def sweep(self, x):
        return torch.where(self.active[:, None], (1 - OMEGA) * x + OMEGA * (self.W @ x) * self.Dinv, x)

    def per_edge(self, f, chunk=1 << 21):
        return torch.cat([f(self.lo[t:t + chunk], self.hi[t:t + chunk]) for t in range(0, self.m, chunk)])

    def distances(self, x, normalize=False):
        rho = self.per_edge(lambda i, j: (x[i] - x[j]).square().sum(1).sqrt())
        return rho * (self.D[self.lo, 0] * self.D[self.hi, 0]).sqrt() if normalize else rho

    def gradient(self, loss_edges):
        xs, scale = [self.x0], []
        for _ in range(self.k):
            y = self.sweep(xs[-1])
            x, ends = self.rescale(y)
            lo, hi = ends[0]
            far = torch.full((), self.n, device="cuda")
            at = torch.arange(self.n, device="cuda")[:, None]
            on = self.active[:, None]
            scale.append((torch.where(hi > lo, 1 / (hi - lo), torch.zeros_like(lo)),
                          torch.where(on & (y == lo), at, far).amin(0), torch.where(on & (y == hi), at, far).amin(0)))
            xs.append(x)
            del y
        x = xs[-1]
        rho = self.distances(x)
        c = torch.zeros(self.m, dtype=torch.float64, device="cuda")
        c[loss_edges] = 2.0 * (rho[loss_edges] > 0).double()   # (d loss / d rho) / rho, loss = sum of rho^2
        C = self.matrix(c[self.eid])
        bar = x * (C @ torch.ones(self.n, 1, dtype=torch.float64, device="cuda")) - C @ x
        r = torch.arange(self.R, device="cuda")
        grad = torch.zeros(self.m, dtype=torch.float64, device="cuda")
        const = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        for t in range(self.k, 0, -1):
            a, imin, imax = scale[t - 1]
            A, B = (bar * (xs[t] - 0.5)).sum(0), (bar * (xs[t] + 0.5)).sum(0)
            y = a * bar
            y[imin, r] += a * A
            y[imax, r] -= a * B
            U, prev = y * self.Dinv, xs[t - 1]
            const += (U * (self.W @ prev) * self.Dinv).sum(1)
            grad += self.per_edge(lambda i, j: (U[i] * prev[j]).sum(1) + (U[j] * prev[i]).sum(1))
            bar = (1 - OMEGA) * y + OMEGA * (self.W @ U)
            xs.pop()
        return rho, OMEGA * (grad - const[self.lo] - const[self.hi])


def exact(case, seed):
    if case["kind"] in ("select", "multilevel"):   # whole numbers and bytes: nothing is rounded
        return None
    e = _Exact(case, seed)
    if case["kind"] == "grad":
        rho, grad = e.gradient(_loss_edges(case["m"], seed))
        return {"rho": rho, "w_grad": grad}
    x = e.x0
    for _ in range(e.k):
        x, _ = e.rescale(e.sweep(x))
    rho = e.distances(x, case.get("normalize", False))
    if case["kind"] == "host":
        return {"rho": rho, "keep_local": None, "keep_global": None, "kept": [None, None], "e": [None, None]}
    return {"rho": rho}
