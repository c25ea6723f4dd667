"""Performance cases: what a user of the library has it do, end to end through
the binding, from ten 500-node graphs to 1e9 edges.

A case is one of
  scores      eq. 5 on a ready handle, then the top-k
  sweep       one run of an identification sweep: generate the backgrounds on
              the device, score them, take the top-k, drop the handle
  upload      the same from CSR arrays in pinned host memory, top-k read back
  grad        scores, top-k and the edge gradient of the top-k score
  restart     eq. 5 by restarted Lanczos (bounded basis), then the top-k
  centrality  sub-graph centrality of candidate nodes of one graph

Graphs are Erdos-Renyi (`deg`: mean degree), Watts-Strogatz (`deg`: ring
degree, rewiring 0.1) or Barabasi-Albert (`deg`: links per new node), with a
planted target of `k` nodes: a clique in a single background, a random tree
plus k/2 edges where several realisations share it.
"""
import math
import random

import numpy as np
import torch

from paper_1409_5000_gb300 import binding as B

REWIRE = 0.1
L2_BYTES = 100e6  # what stays on the chip between two Lanczos steps


def _case(name, kind, model, N, n_lo, n_hi, deg, m, k, prec="f32", **more):
    return dict(name=name, kind=kind, model=model, N=N, n_lo=n_lo, n_hi=n_hi, deg=deg, m=m, k=k,
                prec=prec, **more)


def listed():
    return [
        # the smallest call: ten 500-node realisations, as in the smoke run
        _case("small-ensemble", "scores", "er", 10, 500, 500, 8.0, 20, 15),
        # one run of a Table 1 sweep column: 40 fresh backgrounds per call
        _case("sweep-run", "sweep", "er", 40, 4000, 4000, 4.9, 30, 20),
        # one 1e5-node background with a planted clique, single precision
        _case("er-100k", "scores", "er", 1, 100_000, 100_000, 10.0, 30, 12),
        # the same with hubs, in double precision
        _case("ba-100k-f64", "scores", "ba", 1, 100_000, 100_000, 5, 30, 12, prec="f64"),
        # double precision with full reorthogonalisation: the reference-grade mode
        _case("ws-100k-reorth", "scores", "ws", 1, 100_003, 100_003, 10, 30, 12, prec="f64",
              reorth=True),
        # a background of a million nodes
        _case("er-1m", "scores", "er", 1, 1_000_003, 1_000_003, 16.0, 40, 20),
        # the headline workload: 256 uneven realisations, 1e9 entries
        _case("ensemble-256", "scores", "er", 256, 20_000, 400_000, 20.0, 25, 30),
        # the largest single graph: 1e7 nodes, 1.6e8 entries
        _case("ba-10m", "scores", "ba", 1, 10_000_000, 10_000_000, 8, 40, 20),
        # 40 realisations from pinned host memory to the recovered target
        _case("upload-40", "upload", "er", 40, 20_000, 400_000, 20.0, 25, 30),
        # forward and backward: the edge sensitivities of the recovered target
        _case("grad-64", "grad", "er", 64, 100_000, 100_000, 16.0, 30, 25),
        # a bounded basis: five restarted cycles of five steps
        _case("restart-40", "restart", "er", 40, 20_000, 400_000, 20.0, 5, 30, cycles=5),
        # eq. 3 for the candidates of one background
        _case("centrality-30", "centrality", "er", 1, 100_000, 100_000, 10.0, 20, 30),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _deg(rng, model, lo=4.0, hi=24.0):
    d = rng.uniform(lo, hi)
    return round(d, 1) if model == "er" else 2 * max(2, int(d / 2)) if model == "ws" else max(2, int(d / 2))


def draw(rng):
    kind = rng.choice(["scores"] * 5 + ["sweep", "upload", "grad", "restart", "centrality"])
    model = rng.choice(["er", "er", "ba", "ws"])
    prec = rng.choice(["f32", "f32", "f64"])
    c = dict(kind=kind, model=model, N=1, prec=prec, m=rng.randint(10, 40), k=rng.randint(8, 40))
    shape = rng.choice(["small", "single", "single", "large", "ensemble"]) if kind == "scores" else kind
    if shape in ("small", "sweep"):
        c.update(N=_log(rng, 2, 64), deg=_deg(rng, model))
        n = _log(rng, 300, 9000)
        c.update(n_lo=n, n_hi=n if shape == "sweep" else n + rng.randint(0, n))
    elif shape in ("single", "centrality"):
        n = _log(rng, 10_000, 500_000 if shape == "single" else 150_000)
        c.update(n_lo=n, n_hi=n, deg=_deg(rng, model))
        if model == "ba" and (kind == "centrality" or n > 150_000):
            c.update(prec="f64")  # hubs: the largest eigenvalue nears a hundred
        c.update(reorth=shape == "single" and rng.random() < 0.2)
    elif shape == "large":
        n = _log(rng, 530_000, 9_000_000)
        model = "er" if model == "ba" else model
        c.update(model=model, n_lo=n, n_hi=n, deg=_deg(rng, model, 8.0, 16.0), prec="f32")
    else:  # ensembles of uneven realisations
        lo = _log(rng, 10_000, 100_000)
        c.update(N=_log(rng, 8, 160 if shape == "ensemble" else 48), n_lo=lo,
                 n_hi=lo + rng.randint(0, 3 * lo), deg=_deg(rng, model, 8.0, 24.0))
        c.update(m=rng.randint(10, 30))
        # no drawn case costs more than the largest listed one
        most = {"scores": 6e8, "grad": 1e8}.get(kind, 2e8) * (0.15 if prec == "f64" else 1.0)
        mean = (c["n_lo"] + c["n_hi"]) / 2 * c["deg"] * (2 if model == "ba" else 1)
        c.update(N=max(2, min(c["N"], int(most / mean))))
    if kind == "restart":
        c.update(m=rng.randint(4, 10), cycles=rng.randint(2, 6))
    return c


# ---- inputs ---------------------------------------------------------------

class Graph:
    def __init__(self, n, row_ptr, col):
        self.n, self.row_ptr, self.col = n, row_ptr, col


def _sizes(case):
    r = random.Random("%(N)d %(n_lo)d %(n_hi)d" % case)
    return [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case["N"])]


def _target(case, seed):
    """The planted target's edges, an (E, 2) array: a clique in one background,
    a random tree plus k/2 edges where several realisations share it."""
    r, k = random.Random(seed), case["k"]
    nodes = r.sample(range(min(_sizes(case))), k)
    if case["N"] == 1:
        e = {(a, b) for a in range(k) for b in range(a)}
    else:
        e = {(a, r.randrange(a)) for a in range(1, k)}
        while len(e) < min(k - 1 + k // 2, k * (k - 1) // 2):
            a, b = sorted(r.sample(range(k), 2), reverse=True)
            e.add((a, b))
    return np.array([(nodes[a], nodes[b]) for a, b in sorted(e)], dtype=np.int64)


def _pairs(model, n, deg, gen):
    dev = "cuda"
    if model == "er":
        M = int(deg * n / 2)
        return (torch.randint(n, (M,), generator=gen, device=dev),
                torch.randint(n, (M,), generator=gen, device=dev))
    if model == "ws":
        h = deg // 2
        t = torch.arange(n * h, device=dev)
        u, v = t // h, (t // h + t % h + 1) % n
        far = torch.rand(n * h, generator=gen, device=dev) < REWIRE
        return u, torch.where(far, torch.randint(n, (n * h,), generator=gen, device=dev), v)
    # ba: edge t of new node deg + t // deg takes a uniform place of the list of
    # all earlier edges' ends; a place that holds a target is followed back
    E = deg * (n - deg)
    t = torch.arange(E, device=dev)
    pos = (torch.rand(E, generator=gen, device=dev, dtype=torch.float64) * (2 * deg * (t // deg))).long()
    v = torch.where(t < deg, t, torch.where(pos % 2 == 0, deg + pos // 2 // deg, -1))
    todo = (v < 0).nonzero()[:, 0]
    at = pos[todo] // 2
    while todo.numel():
        got = v[at]
        v[todo] = got
        left = (got < 0).nonzero()[:, 0]
        todo, at = todo[left], pos[at[left]] // 2
    return deg + t // deg, v


def _graphs(case, seed):
    tgt = torch.from_numpy(_target(case, seed)).cuda()
    gen = torch.Generator("cuda").manual_seed(seed)
    out = []
    for n in _sizes(case):
        u, v = _pairs(case["model"], n, case["deg"], gen)
        M = u.numel()
        key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
        t = torch.unique(tgt.min(1)[0] * n + tgt.max(1)[0])
        key = key[(key // n != key % n) & ~torch.isin(key, t)]
        if case["kind"] == "grad":  # as many edges for every seed: the gradient's length
            key = key[torch.randperm(key.numel(), generator=gen, device="cuda")[: int(0.98 * M)]]
        key = torch.cat([key, t])
        key = torch.sort(torch.cat([key, key % n * n + key // n]))[0]
        rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).int()
        out.append(Graph(n, rp, (key % n).int()))
    return out


def _prec(case):
    p = B.CB_FP64 if case["prec"] == "f64" else B.CB_FP32
    return p | B.CB_REORTH if case.get("reorth") else p


def _nodes(case, seed):
    """Candidate nodes: half of them in the target, the others anywhere."""
    r, k = random.Random(seed + 1), case["k"]
    some = sorted(set(_target(case, seed).reshape(-1).tolist()))[: (k + 1) // 2]
    rest = [i for i in r.sample(range(case["n_lo"]), 2 * k) if i not in some]
    return (some + rest)[:k]


class Result:
    """Buffers a program keeps: scores, log scale and top values in one block."""

    def __init__(self, n, k):
        self.block = torch.empty(n + 1 + k, dtype=torch.float64, device="cuda")
        self.S, self.ls, self.val = self.block[:n], self.block[n:n + 1], self.block[n + 1:]
        self.idx = torch.empty(k, dtype=torch.int32, device="cuda")

    def out(self, case):
        # single precision's results go on as float32, in one conversion
        n, b = self.S.numel(), self.block if case["prec"] == "f64" else self.block.float()
        return {"scores": b[:n], "log_scale": b[n:n + 1], "top": self.idx, "top_scores": b[n + 1:]}


def prepare(case, seed):
    st = {"case": case, "seed": seed, "prec": _prec(case), "res": Result(max(_sizes(case)), case["k"])}
    kind = case["kind"]
    if kind == "sweep":
        st["target"] = _target(case, seed)
        return st
    graphs = _graphs(case, seed)
    if kind == "upload":
        st["graphs"] = [Graph(g.n, g.row_ptr.cpu().pin_memory(), g.col.cpu().pin_memory()) for g in graphs]
        return st
    st["gs"] = B.GraphSet(graphs)
    if kind == "centrality":
        st["nodes"] = _nodes(case, seed)
    return st


def run(st):
    case, prec, res, kind = st["case"], st["prec"], st["res"], st["case"]["kind"]
    m, k = case["m"], case["k"]
    if kind == "centrality":
        ls, sc = B.subgraph_centrality(st["gs"], 0, m, st["nodes"], prec)
        return {"log_scale": ls, "sc": sc} if case["prec"] == "f64" else {"log_scale": ls.float(), "sc": sc.float()}
    if kind == "sweep":
        model, sizes = case["model"], _sizes(case)
        if model == "er":
            gs = B.GraphSet.generate_er(sizes, case["deg"], st["seed"], st["target"])
        elif model == "ws":
            gs = B.GraphSet.generate_ws(sizes, case["deg"], REWIRE, st["seed"], st["target"])
        else:
            gs = B.GraphSet.generate_ba(sizes, case["deg"], st["seed"], st["target"])
    else:
        gs = B.GraphSet(st["graphs"]) if kind == "upload" else st["gs"]
    if kind == "restart":
        B.ensemble_scores_restarted(gs, m, case["cycles"], prec, out=(res.S, res.ls))
    else:
        B.ensemble_scores(gs, m, prec, out=(res.S, res.ls))
    B.topk(res.S, k, out=(res.idx, res.val))
    out = res.out(case)
    if kind == "grad":
        ls, g = B.scores_backward(gs, m, res.idx, prec)
        out.update(grad=g, grad_log_scale=ls if case["prec"] == "f64" else ls.float())
    elif kind == "upload":
        out.update(top=res.idx.cpu(), top_scores=out["top_scores"].cpu())
    if kind in ("sweep", "upload"):
        gs.close()
    return out


# ---- work -----------------------------------------------------------------

def work(case):
    """Bytes: the CSR arrays and three vectors once per Lanczos step where they
    are larger than what stays on the chip, else once; the results once."""
    esz = 8 if case["prec"] == "f64" else 4
    per_node = case["deg"] * (2 if case["model"] == "ba" else 1)
    n = sum(_sizes(case))
    nnz = per_node * n
    cols = case["k"] if case["kind"] == "centrality" else 1
    steps = case["m"] * case.get("cycles", 1) * (2 if case["kind"] == "grad" else 1)
    one = 4 * nnz + 4 * n + 3 * esz * n * cols
    b = one * (steps if one > L2_BYTES else 1) + 8 * max(_sizes(case))
    f = steps * cols * (2 * nnz + 8 * n)
    if case.get("reorth"):  # two Gram-Schmidt passes over the basis so far
        b += 2 * esz * n * steps * steps / 2 if esz * n * steps > L2_BYTES else 0
        f += 4 * n * steps * steps
    if case["kind"] == "grad":  # both bases once, two m-vectors per edge, the gradient
        b += 2 * esz * n * case["m"] + 4 * nnz
        f += 2 * nnz * case["m"]
    if case["kind"] == "upload":
        b += 4 * nnz + 4 * n
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, by torch's sparse products and dense exponentials ----

def _matrix(g):
    return torch.sparse_csr_tensor(g.row_ptr, g.col, torch.ones(g.col.numel(), dtype=torch.float64, device="cuda"),
                                   size=(g.n, g.n))


def _lanczos(A, b, m):
    """V (steps + 1, n), T, ||b|| and the norm after the last step."""
    b0 = float(b.norm())
    V = torch.zeros(m + 1, b.numel(), dtype=torch.float64, device="cuda")
    V[0] = b / b0
    al, be = [], []
    for j in range(m):
        w = A @ V[j]
        if j:
            w -= be[-1] * V[j - 1]
        al.append(float(V[j] @ w))
        w -= al[-1] * V[j]
        for _ in range(2):
            w -= V[:j + 1].T @ (V[:j + 1] @ w)
        be.append(float(w.norm()))
        if be[-1] <= 1e-12 * (abs(al[-1]) + (be[-2] if j else 0.0)):
            be[-1] = 0.0
            break
        V[j + 1] = w / be[-1]
    return V, np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1), b0, be[-1]


def _exp_e1(T):
    lam, Q = np.linalg.eigh(T)
    return lam[-1], Q @ (np.exp(lam - lam[-1]) * Q[0])


def _scores64(g, case):
    A, one = _matrix(g), torch.ones(g.n, dtype=torch.float64, device="cuda")
    if case["kind"] != "restart":
        V, T, b0, _ = _lanczos(A, one, case["m"])
        th, c = _exp_e1(T)
        return th, b0 * (V[:len(c)].T @ torch.from_numpy(c).cuda())
    blocks, couple, Vs, b, norm = [], [], [], one, None
    for _ in range(case["cycles"]):
        V, T, b0, last = _lanczos(A, b, case["m"])
        norm = norm or b0
        blocks.append(T)
        couple.append(last)
        Vs.append(V[:len(T)])
        if last == 0.0:
            break
        b = V[-1]
    H = np.zeros((sum(map(len, blocks)),) * 2)
    at = 0
    for q, T in enumerate(blocks):
        H[at:at + len(T), at:at + len(T)] = T
        if q:
            H[at, at - 1] = couple[q - 1]
        at += len(T)
    th = max(np.linalg.eigvalsh(T)[-1] for T in blocks)
    c = torch.linalg.matrix_exp(torch.from_numpy(H - th * np.eye(at)))[:, 0].cuda()
    return th, norm * (torch.cat(Vs).T @ c)


def _grad64(g, case, top):
    A, m = _matrix(g), case["m"]
    w = torch.zeros(g.n, dtype=torch.float64, device="cuda")
    w[top[top < g.n]] = 1.0
    V1, T1, b1, _ = _lanczos(A, torch.ones_like(w), m)
    rows = torch.repeat_interleave(torch.arange(g.n, device="cuda"), g.row_ptr.diff())
    if not w.any():
        return -math.inf, torch.zeros(g.col.numel(), dtype=torch.float64, device="cuda")
    Vw, Tw, bw, _ = _lanczos(A, w, m)
    p, q = len(Tw), len(T1)
    th = max(np.linalg.eigvalsh(Tw)[-1], np.linalg.eigvalsh(T1)[-1])
    H = np.zeros((p + q, p + q))
    H[:p, :p], H[p:, p:], H[0, p] = Tw - th * np.eye(p), T1 - th * np.eye(q), 1.0
    M = torch.linalg.matrix_exp(torch.from_numpy(H))[:p, p:].cuda() * (bw * b1)
    P, U = Vw[:p].T @ M, V1[:q].T.contiguous()
    out, col = torch.empty(rows.numel(), dtype=torch.float64, device="cuda"), g.col.long()
    for e in range(0, rows.numel(), 1 << 20):
        i, j = rows[e:e + (1 << 20)], col[e:e + (1 << 20)]
        out[e:e + (1 << 20)] = (P[i] * U[j]).sum(1) + (P[j] * U[i]).sum(1)
    return th, out


def _centrality64(g, case, nodes):
    A, k = _matrix(g), len(nodes)
    V = [torch.zeros(g.n, k, dtype=torch.float64, device="cuda")]
    V[0][torch.tensor(nodes, device="cuda"), torch.arange(k, device="cuda")] = 1.0
    al, be, live = [], [], torch.ones(k, dtype=torch.float64, device="cuda")
    for j in range(case["m"]):
        w = A @ V[j]
        if j:
            w -= be[-1] * V[j - 1]
        al.append((V[j] * w).sum(0))
        w -= al[-1] * V[j]
        for _ in range(2):
            for v in V:
                w -= v * (v * w).sum(0)
        b = w.norm(dim=0) * live
        b[b <= 1e-12 * (al[-1].abs() + (be[-1] if j else 0.0))] = 0.0
        live = (b > 0).double()
        be.append(b)
        V.append(w * (live / torch.where(b > 0, b, torch.ones_like(b))))
    al, be = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()
    th, c0 = np.empty(k), np.empty(k)
    for q in range(k):
        s = next((j + 1 for j in range(len(be)) if be[j, q] == 0.0), len(be))
        th[q], c = _exp_e1(np.diag(al[:s, q]) + np.diag(be[:s - 1, q], 1) + np.diag(be[:s - 1, q], -1))
        c0[q] = c[0]
    return th.max(), np.exp(th - th.max()) * c0


def exact(case, seed):
    kind, k = case["kind"], case["k"]
    if kind == "sweep":  # its graphs are the library's own
        return None
    graphs = _graphs(case, seed)
    if kind == "centrality":
        th, sc = _centrality64(graphs[0], case, _nodes(case, seed))
        return {"log_scale": np.array([th]), "sc": sc}
    th, ys = zip(*(_scores64(g, case) for g in graphs))
    top_th = max(th)
    S = torch.zeros(max(g.n for g in graphs), dtype=torch.float64, device="cuda")
    for t, y in zip(th, ys):
        S[:y.numel()] += math.exp(t - top_th) * y
    val, idx = torch.topk(S, k)
    out = {"scores": S, "log_scale": np.array([top_th]), "top": None, "top_scores": val}
    if kind == "grad":
        th, gr = zip(*(_grad64(g, case, idx) for g in graphs))
        top_th = max(th)
        out["grad"] = torch.cat([math.exp(t - top_th) * x for t, x in zip(th, gr)])
        out["grad_log_scale"] = np.array([top_th])
    return out
