"""The calls this library is measured by: the work its users bring, over the range of sizes it is used for.

A case is one call (or one batch, or one burst of requests) through the package's public functions.  Its kind says
which:

  apsp    all-pairs shortest paths of one weighted digraph (`apsp`)
  gemm    one tropical product (`gemm`)
  paths   distances and next hops of one digraph (`apsp_paths`)
  sssp    distances from one vertex (`sssp`)
  batch   many graphs and many products of uneven sizes in one launch (`Batch`)
  serve   a burst of mixed requests with host buffers (`Server`)

Graphs are G(n, p) digraphs with weights uniform in [1, w], no edge = INF_I32 and a zero diagonal; p = 1 gives the
random matrices (complete graphs) of the library's source paper.
"""
import math

import torch

import paper_1701_04733_gb300 as btas

INF = btas.INF_I32


# ------------------------------------------------------------------ cases
def listed():
    return [
        # The largest of the paper's own sizes: a complete graph small enough that launches and the read-back of the
        # outcome are most of the call.
        {"name": "apsp_complete_n128", "kind": "apsp", "n": 128, "p": 1.0, "w": 100},
        # The benchmark's single small graph.
        {"name": "apsp_n256", "kind": "apsp", "n": 256, "p": 0.1, "w": 100},
        # A dense graph of an odd size with weights too large for 16 bits: no sparsity and no short type to lean on.
        {"name": "apsp_dense_n2999", "kind": "apsp", "n": 2999, "p": 0.5, "w": 1000000},
        # The benchmark's graph for the exact 16-bit path: many equal weights, so most edges lie on shortest paths.
        {"name": "apsp_n4096_w7", "kind": "apsp", "n": 4096, "p": 0.05, "w": 7},
        # The benchmark's large graph, the largest solve a user brings.
        {"name": "apsp_n8192", "kind": "apsp", "n": 8192, "p": 0.01, "w": 1000},
        # One product of the size that the serving mix has most of.
        {"name": "gemm_i32_n200", "kind": "gemm", "dtype": "i32", "semiring": "min", "m": 200, "n": 200, "k": 200,
         "trans_b": False, "packed": False},
        # An ordinary product with ragged sides, the other semiring, real values.
        {"name": "gemm_f32_max_ragged", "kind": "gemm", "dtype": "f32", "semiring": "max", "m": 1000, "n": 1531,
         "k": 777, "trans_b": False, "packed": False},
        # The benchmark's large product, the library's headline call.
        {"name": "gemm_i32_n8192", "kind": "gemm", "dtype": "i32", "semiring": "min", "m": 8192, "n": 8192, "k": 8192,
         "trans_b": True, "packed": False},
        # Routing: next hops as well as distances.
        {"name": "paths_n2048", "kind": "paths", "n": 2048, "p": 0.05, "w": 1000},
        # Distances from one vertex of the large graph.
        {"name": "sssp_n8192", "kind": "sssp", "n": 8192, "p": 0.01, "w": 1000},
        # The benchmark's batch: 512 graphs and 512 products of the same uneven sizes.
        {"name": "batch_512", "kind": "batch", "graphs": 512, "lo": 32, "hi": 1024, "p": 0.1, "w": 100},
        # A burst of the benchmark's request mix, host buffers to host buffers.
        {"name": "serve_burst_48", "kind": "serve", "requests": 48, "lo": 64, "hi": 2048, "p": 0.1, "w": 100},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["apsp", "apsp", "apsp", "gemm", "gemm", "paths", "sssp", "batch", "serve"])
    p = round(math.exp(rng.uniform(math.log(0.01), 0.0)), 4)
    w = rng.choice([7, 100, 1000, 1000000])
    if kind == "apsp":
        return {"kind": kind, "n": _log(rng, 8, 8192), "p": p, "w": w}
    if kind == "gemm":
        dtype = rng.choice(["i32", "f32"])
        return {"kind": kind, "dtype": dtype, "semiring": rng.choice(["min", "max"]), "m": _log(rng, 32, 8192),
                "n": _log(rng, 32, 8192), "k": _log(rng, 32, 8192), "trans_b": rng.random() < 0.3,
                "packed": dtype == "i32" and rng.random() < 0.3}
    if kind == "paths":
        return {"kind": kind, "n": _log(rng, 32, 3000), "p": p, "w": w}
    if kind == "sssp":
        return {"kind": kind, "n": _log(rng, 256, 8192), "p": p, "w": w}
    if kind == "batch":
        hi = rng.randint(100, 1024)
        return {"kind": kind, "graphs": _log(rng, 8, 256), "lo": 16, "hi": hi, "p": max(p, 0.02), "w": w}
    return {"kind": kind, "requests": _log(rng, 6, 64), "lo": 64, "hi": rng.randint(300, 2048), "p": max(p, 0.02),
            "w": w}


# ----------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _graph_values(g, count, p, w):
    """`count` entries: a weight in [1, w] with probability p, else INF."""
    v = torch.randint(1, w + 1, (count,), dtype=torch.int32, device="cuda", generator=g)
    if p < 1.0:
        v.masked_fill_(torch.rand(count, device="cuda", generator=g) >= p, INF)
    return v


def _graph(g, n, p, w):
    W = _graph_values(g, n * n, p, w).view(n, n)
    W.fill_diagonal_(0)
    return W


def _matrix(g, rows, cols, dtype, packed):
    if dtype == "f32":
        return torch.rand(rows, cols, device="cuda", generator=g)
    # the packed path takes operands of small range; the others the benchmark's [0, 10^6]
    lo, hi = (-4000, 4001) if packed else (0, 1000001)
    return torch.randint(lo, hi, (rows, cols), dtype=torch.int32, device="cuda", generator=g)


def _sizes(count, lo, hi, log):
    """`count` sizes of [lo, hi] at even steps (of the logarithm with `log`), in a fixed shuffled order: two states
    of one case have the same sizes."""
    out = []
    for i in range(count):
        t = ((i * 0.6180339887498949) + 0.5) % 1.0
        out.append(int(round(lo * (hi / lo) ** t if log else lo + (hi - lo) * t)))
    return out


def _views(flat, sizes):
    out, at = [], 0
    for n in sizes:
        out.append(flat[at:at + n * n].view(n, n))
        at += n * n
    return out


def _batch_inputs(case, seed):
    g = _generator(seed)
    sizes = _sizes(case["graphs"], case["lo"], case["hi"], False)
    total = sum(n * n for n in sizes)
    W = _graph_values(g, total, case["p"], case["w"])
    A = torch.rand(total, device="cuda", generator=g)
    B = torch.rand(total, device="cuda", generator=g)
    for v in _views(W, sizes):
        v.fill_diagonal_(0)
    return sizes, W, A, B


def _serve_requests(case):
    """(kind, semiring, dtype, n) per request: half APSP, half products; semirings and types half and half."""
    reqs = []
    for i, n in enumerate(_sizes(case["requests"], case["lo"], case["hi"], True)):
        if i % 2 == 0:
            reqs.append(("apsp", "min", "i32", n))
        else:
            reqs.append(("gemm", "max" if i % 4 == 1 else "min", "f32" if i % 8 < 4 else "i32", n))
    return reqs


def _serve_inputs(case, seed):
    g = _generator(seed)
    ins = []
    for kind, _, dtype, n in _serve_requests(case):
        if kind == "apsp":
            ins.append((_graph(g, n, case["p"], case["w"]),))
        else:
            ins.append((_matrix(g, n, n, dtype, False), _matrix(g, n, n, dtype, False)))
    return ins


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("apsp", "paths", "sssp"):
        return {"case": case, "W": _graph(_generator(seed), case["n"], case["p"], case["w"]),
                "src": seed % case["n"]}
    if kind == "gemm":
        g = _generator(seed)
        A = _matrix(g, case["m"], case["k"], case["dtype"], case["packed"])
        B = _matrix(g, case["n"] if case["trans_b"] else case["k"], case["k"] if case["trans_b"] else case["n"],
                    case["dtype"], case["packed"])
        return {"case": case, "A": A, "B": B}
    if kind == "batch":
        sizes, W, A, B = _batch_inputs(case, seed)
        D, C = torch.empty_like(W), torch.empty_like(A)
        b = btas.Batch()
        for w, d in zip(_views(W, sizes), _views(D, sizes)):
            b.add_apsp(w, d)
        for x, y, z in zip(_views(A, sizes), _views(B, sizes), _views(C, sizes)):
            b.add_gemm(x, y, z, "max")
        return {"case": case, "batch": b, "D": D, "C": C, "keep": (W, A, B)}
    # serve: pinned host buffers, one flat output buffer per type
    reqs = _serve_requests(case)
    ins = [tuple(x.cpu().pin_memory() for x in xs) for xs in _serve_inputs(case, seed)]
    outs, work = {}, []
    for dtype, t in (("i32", torch.int32), ("f32", torch.float32)):
        flat = torch.empty(sum(n * n for _, _, d, n in reqs if d == dtype), dtype=t).pin_memory()
        outs[dtype] = (flat, iter(_views(flat, [n for _, _, d, n in reqs if d == dtype])))
    for (kind, semiring, dtype, n), xs in zip(reqs, ins):
        work.append((kind, semiring, xs, next(outs[dtype][1])))
    return {"case": case, "server": btas.Server(40 << 30), "work": work, "i32": outs["i32"][0], "f32": outs["f32"][0]}


# -------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apsp":
        return btas.apsp(state["W"])
    if kind == "paths":
        return btas.apsp_paths(state["W"])
    if kind == "sssp":
        return btas.sssp(state["W"], state["src"])
    if kind == "gemm":
        return btas.gemm(state["A"], state["B"], case["semiring"], trans_b=case["trans_b"], packed=case["packed"])
    if kind == "batch":
        state["batch"].launch()
        state["batch"].wait()  # its status word says whether the results are complete
        return state["D"], state["C"]
    server = state["server"]
    for what, semiring, xs, out in state["work"]:
        if what == "apsp":
            server.submit_apsp(xs[0], out)
        else:
            server.submit_gemm(xs[0], xs[1], out, semiring)
    server.wait_all()
    return state["i32"], state["f32"]


# ------------------------------------------------------------------- work
def work(case):
    """Each input read and each output written once.  Operations: an add and a minimum per term of a product; for
    shortest paths one relaxation (an add and a minimum) of each edge from each source, which no method that looks
    at the weights avoids in general."""
    def apsp(n):
        return 8 * n * n, 2 * n * int(case["p"] * n * n)

    def gemm(m, n, k):
        return 4 * (m * k + k * n + m * n), 2 * m * n * k

    kind = case["kind"]
    if kind == "apsp":
        parts = [apsp(case["n"])]
    elif kind == "paths":
        b, f = apsp(case["n"])
        parts = [(b + 4 * case["n"] ** 2, f)]
    elif kind == "sssp":
        n = case["n"]
        parts = [(4 * n * n + 4 * n, 2 * int(case["p"] * n * n))]
    elif kind == "gemm":
        parts = [gemm(case["m"], case["n"], case["k"])]
    elif kind == "batch":
        sizes = _sizes(case["graphs"], case["lo"], case["hi"], False)
        parts = [apsp(n) for n in sizes] + [gemm(n, n, n) for n in sizes]
    else:
        parts = [apsp(n) if k == "apsp" else gemm(n, n, n) for k, _, _, n in _serve_requests(case)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ------------------------------------------------------------------ exact
_BIG = 1 << 40  # no edge, in 64 bits


def _exact_apsp(W):
    """Floyd-Warshall in 64-bit integers."""
    D = W.long()
    D[W == INF] = _BIG
    T = torch.empty_like(D)
    for k in range(W.shape[0]):
        torch.add(D[:, k:k + 1], D[k:k + 1, :], out=T)
        torch.minimum(D, T, out=D)
    D[D >= _BIG] = INF
    return D


def _exact_paths(W):
    """Squarings of D in 64 bits with the smallest minimising k, which gives the next hop; stops once nothing changes."""
    n = W.shape[0]
    D = W.long()
    D[W == INF] = _BIG
    cols = torch.arange(n, device=W.device).expand(n, n)
    rows = cols.t()
    N = torch.where(W == INF, -1, cols).contiguous()
    for _ in range(max(0, math.ceil(math.log2(n - 1))) if n > 2 else 0):
        best, arg = torch.full_like(D, 2 * _BIG + 1), torch.zeros_like(D)
        for k in range(n):
            T = D[:, k:k + 1] + D[k:k + 1, :]
            less = T < best
            torch.minimum(best, T, out=best)
            arg.masked_fill_(less, k)
        best.clamp_(max=_BIG)
        nxt = torch.where(arg == rows, N, torch.gather(N, 1, arg))
        nxt = torch.where(best >= _BIG, -1, nxt)
        if torch.equal(best, D) and torch.equal(nxt, N):
            break
        D, N = best, nxt
    D[D >= _BIG] = INF
    return D, N


def _exact_gemm(A, B, semiring):
    """The product in 64 bits: term by term, the sums exact."""
    t = torch.float64 if A.dtype == torch.float32 else torch.int64
    A, B = A.to(t), B.to(t)
    C = A[:, :1] + B[:1, :]
    T = torch.empty_like(C)
    pick = torch.minimum if semiring == "min" else torch.maximum
    for k in range(1, A.shape[1]):
        torch.add(A[:, k:k + 1], B[k:k + 1, :], out=T)
        pick(C, T, out=C)
    return C


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apsp", "paths", "sssp"):
        W = _graph(_generator(seed), case["n"], case["p"], case["w"])
        if kind == "apsp":
            return _exact_apsp(W)
        if kind == "paths":
            return _exact_paths(W)
        d = torch.full((case["n"],), _BIG, dtype=torch.int64, device="cuda")
        d[seed % case["n"]] = 0
        L = W.long()
        L[W == INF] = _BIG
        while True:
            new = (d[:, None] + L).amin(0).clamp_(max=_BIG)
            if torch.equal(new, d):
                break
            d = new
        d[d >= _BIG] = INF
        return d
    if kind == "gemm":
        s = prepare(case, seed)
        return _exact_gemm(s["A"], s["B"].t() if case["trans_b"] else s["B"], case["semiring"])
    if kind == "batch":
        # the distances are whole numbers and have to be equal anyway; the products are the rounded values
        sizes, _, A, B = _batch_inputs(case, seed)
        C = torch.empty(A.numel(), dtype=torch.float64, device="cuda")
        for x, y, z in zip(_views(A, sizes), _views(B, sizes), _views(C, sizes)):
            z.copy_(_exact_gemm(x, y, "max"))
        return None, C
    i32, f32 = [], []
    for (what, semiring, dtype, n), xs in zip(_serve_requests(case), _serve_inputs(case, seed)):
        C = _exact_apsp(xs[0]) if what == "apsp" else _exact_gemm(xs[0], xs[1], semiring)
        (i32 if dtype == "i32" else f32).append(C.reshape(-1).cpu())
    return (torch.cat(i32) if i32 else None), (torch.cat(f32) if f32 else None)
