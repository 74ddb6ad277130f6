"""Performance cases: the work that users of this library have it do, through
its Python entry points.

Inputs are seeded synthetic graphs built on the GPU, of the families that the
tests and the benchmark use: R-MAT (edge factor 16, .57/.19/.19/.05), planted
stochastic block models (half of every vertex's expected degree leaves its
block) and rewired 3-D lattices; modularity or the constant Potts model.

A case is a dict of plain values; ``listed()`` names the fixed ones, ``draw``
gives others of the same ranges, ``prepare`` makes the inputs a program has in
hand, ``run`` makes one pass, ``work`` counts the bytes one pass cannot do
without and ``exact`` states the computed numbers independently.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_01503_gb300 as lc

# ----------------------------------------------------------------- the cases

# Ranges of the drawn cases; the listed ones lie at their ends and between.
_SCALE = (10, 22)              # R-MAT: 2^scale vertices
_SBM_N = (1_000, 1_000_000)    # vertices of a block model
_SIDE = (16, 256)              # lattice: side^3 vertices
_BATCH = (16, 512)             # graphs of a batch, each of 100 .. 100,000 vertices
_SERVED = (4, 24)              # requests handed to the service at once


def listed() -> list[dict]:
    return [
        # The smallest ordinary request: one block model of 10,000 vertices and
        # about 50,000 edges on device tensors; launches and host steps count.
        {"name": "cluster_sbm_10k", "call": "cluster", "graph": "sbm", "n": 10_000, "k": 100, "d": 9.9,
         "wmax": 1, "cpm": False, "replay": False},
        # A skewed graph of middle size (2 M stored edges), weighted, the
        # constant Potts model with lambda = 1/50, as service requests have it.
        {"name": "cluster_rmat_16", "call": "cluster", "graph": "rmat", "scale": 16, "wmax": 8, "cpm": True,
         "replay": False},
        # The benchmark's own graph: R-MAT 22, 128 M stored edges, hubs of
        # degree above 100,000 beside 43 % isolated vertices.
        {"name": "cluster_rmat_22", "call": "cluster", "graph": "rmat", "scale": 22, "wmax": 8, "cpm": False,
         "replay": False},
        # The largest vertex count: a 256^3 lattice (100 M stored edges, degree
        # 6), CPM 1/100, a deep hierarchy; repeated passes replayed as graphs.
        {"name": "cluster_grid_256", "call": "cluster", "graph": "grid", "side": 256, "wmax": 16, "cpm": True,
         "replay": True},
        # Many independent graphs in one call: 512 block models of 100 to
        # 100,000 vertices and mean degree 4 to 32, packed in one CSR.
        {"name": "batch_512", "call": "batch", "count": 512, "n_lo": 100, "n_hi": 100_000, "wmax": 1,
         "replay": True},
        # pLeiden+ on a skewed graph: refinement beside the local moves, many
        # levels.
        {"name": "leiden_rmat_18", "call": "leiden", "graph": "rmat", "scale": 18, "wmax": 8, "cpm": False,
         "plus": True},
        # Iterated Louvain+ on a lattice of odd side: constrained coarsening.
        {"name": "iterated_grid_97", "call": "iterated", "graph": "grid", "side": 97, "wmax": 16, "cpm": True,
         "iterations": 3},
        # One local-move call that improves a clustering at hand (a known
        # partition of which a tenth of the vertices has gone stale).
        {"name": "local_move_sbm_1m", "call": "local_move", "graph": "sbm", "n": 1_000_000, "k": 500, "d": 16.0,
         "wmax": 8, "cpm": False, "stale": 0.1},
        # One level of a program's own multilevel driver: contract a graph by
        # the clustering of its local-move pass, then move on the coarse graph.
        {"name": "level_rmat_20", "call": "level", "graph": "rmat", "scale": 20, "wmax": 8, "cpm": False},
        # The exact objective of a given clustering of a large graph.
        {"name": "objective_rmat_21", "call": "objective", "graph": "rmat", "scale": 21, "wmax": 8, "cpm": False},
        # Host buffers in, labels out: a weighted block model in pinned memory.
        {"name": "host_sbm_100k", "call": "host", "graph": "sbm", "n": 100_003, "k": 60, "d": 20.0, "wmax": 8,
         "cpm": True},
        # The service: 24 host requests of mixed families and sizes (block
        # models and R-MAT, modularity and CPM) submitted at once, all awaited.
        {"name": "served_24", "call": "served", "requests": 24, "n_lo": 1_000, "n_hi": 200_000},
    ]


def _log_uniform(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, most: int) -> dict:
    """A graph of at most about `most` stored edges (and of the ranges above)."""
    kind = rng.choice(("sbm", "rmat", "grid"))
    out = {"graph": kind, "wmax": rng.choice((1, 8, 16)), "cpm": rng.random() < 0.5}
    if kind == "rmat":
        out["scale"] = rng.randint(_SCALE[0], min(_SCALE[1], int(math.log2(most / 32))))
    elif kind == "sbm":
        out["d"] = round(rng.uniform(4.0, 32.0), 2)
        out["n"] = _log_uniform(rng, _SBM_N[0], min(_SBM_N[1], int(most / out["d"])))
        out["k"] = _log_uniform(rng, 2, min(500, out["n"] // 8))
    else:
        out["cpm"] = True
        out["side"] = _log_uniform(rng, _SIDE[0], min(_SIDE[1], int((most / 6) ** (1 / 3))))
    return out


def draw(rng) -> dict:
    call = rng.choice(("cluster", "cluster", "cluster", "batch", "leiden", "iterated", "local_move", "level",
                       "objective", "host", "served"))
    if call == "batch":
        return {"call": call, "count": _log_uniform(rng, *_BATCH), "n_lo": 100,
                "n_hi": _log_uniform(rng, 1_000, 100_000), "wmax": rng.choice((1, 8)), "replay": rng.random() < 0.5}
    if call == "served":
        return {"call": call, "requests": rng.randint(*_SERVED), "n_lo": 1_000,
                "n_hi": _log_uniform(rng, 10_000, 200_000)}
    most = {"cluster": 100_000_000, "leiden": 8_000_000, "iterated": 6_000_000, "local_move": 64_000_000,
            "level": 32_000_000, "objective": 64_000_000, "host": 4_000_000}[call]
    case = {"call": call, **_draw_graph(rng, most)}
    if call == "cluster":
        case["replay"] = rng.random() < 0.5
    elif call == "leiden":
        case["plus"] = rng.random() < 0.5
    elif call == "iterated":
        case["iterations"] = rng.randint(2, 4)
    elif call == "local_move":
        case["stale"] = round(rng.uniform(0.02, 0.3), 3)
    return case


# ---------------------------------------------------------------- the graphs


def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(count: int, gen) -> torch.Tensor:
    return torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)


def _csr(n: int, u, v, wmax: int, gen):
    """Undirected CSR of the pairs (u, v): loops and duplicates removed, rows
    sorted, integer weights in [1, wmax] equal in both directions."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    lo, hi = key // n, key % n
    w = torch.randint(1, wmax + 1, (key.numel(),), generator=gen, device="cuda", dtype=torch.int32)
    both, order = torch.sort(torch.cat((key, hi * n + lo)))
    ew = torch.cat((w, w))[order]
    src = both // n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return row_ptr, (both - src * n).to(torch.int32), ew, src


def _rmat_pairs(scale: int, gen):
    m = 16 << scale
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(m, generator=gen, device="cuda")
        u.mul_(2).add_(r >= 0.76)
        v.mul_(2).add_(((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    return u, v


def _sbm_pairs(n, k, d, gen):
    """Pairs of a disjoint union of block models with n[g] vertices in k[g]
    contiguous blocks and mean degree d[g] (sequences), and each vertex's
    block, numbered over the union.  Half of the pairs fall inside a block."""
    n = torch.tensor(n, dtype=torch.int64, device="cuda")
    k = torch.tensor(k, dtype=torch.int64, device="cuda")
    d = torch.tensor(d, dtype=torch.float64, device="cuda")
    base = torch.cumsum(n, 0) - n
    m = (n * d / 4).ceil().to(torch.int64)
    g = torch.repeat_interleave(torch.arange(n.numel(), device="cuda"), m)
    ng, kg, bg = n[g], k[g], base[g]
    pairs = []
    for inside in (True, False):
        x = torch.minimum((_uniform(g.numel(), gen) * ng).to(torch.int64), ng - 1)
        if inside:
            b = x * kg // ng
            start = (b * ng + kg - 1) // kg
            size = ((b + 1) * ng + kg - 1) // kg - start
            y = start + torch.minimum((_uniform(g.numel(), gen) * size).to(torch.int64), size - 1)
        else:
            y = torch.minimum((_uniform(g.numel(), gen) * ng).to(torch.int64), ng - 1)
        pairs.append((bg + x, bg + y))
    gv = torch.repeat_interleave(torch.arange(n.numel(), device="cuda"), n)
    local = torch.arange(gv.numel(), device="cuda") - base[gv]
    block = local * k[gv] // n[gv] + (torch.cumsum(k, 0) - k)[gv]
    return torch.cat((pairs[0][0], pairs[1][0])), torch.cat((pairs[0][1], pairs[1][1])), block, gv


def _grid_pairs(side: int, gen):
    v = torch.arange(side ** 3, device="cuda").view(side, side, side)
    u = torch.cat((v[1:].reshape(-1), v[:, 1:].reshape(-1), v[:, :, 1:].reshape(-1)))
    w = torch.cat((v[:-1].reshape(-1), v[:, :-1].reshape(-1), v[:, :, :-1].reshape(-1)))
    far = (_uniform(u.numel(), gen) * side ** 3).to(torch.int64)
    return torch.where(_uniform(u.numel(), gen) < 0.01, far, u), w


def _graph(case: dict, seed: int) -> dict:
    """row_ptr, col, ew, vw, lambda of a case's graph (CUDA tensors)."""
    gen = _generator(seed)
    block = None
    if case["graph"] == "rmat":
        n = 1 << case["scale"]
        u, v = _rmat_pairs(case["scale"], gen)
    elif case["graph"] == "grid":
        n = case["side"] ** 3
        u, v = _grid_pairs(case["side"], gen)
    else:
        n = case["n"]
        u, v, block, _ = _sbm_pairs([n], [case["k"]], [case["d"]], gen)
    row_ptr, col, ew, src = _csr(n, u, v, case["wmax"], gen)
    if case["cpm"]:
        vw = torch.ones(n, dtype=torch.int64, device="cuda")
        num, den = 1, 100 if case["graph"] == "grid" else 50
    else:
        vw = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, src, ew.to(torch.int64))
        num, den = 1, max(1, int(ew.sum(dtype=torch.int64)))
    return {"row_ptr": row_ptr, "col": col, "ew": ew, "vw": vw, "num": num, "den": den, "block": block}


def _batch(case: dict, seed: int) -> dict:
    rng = np.random.default_rng(seed)
    count = case["count"]
    # sizes at even quantiles of the log-uniform law, so every seed does the same work
    q = (np.arange(count) + 0.5) / count
    n = np.exp(np.log(case["n_lo"]) + q * np.log(case["n_hi"] / case["n_lo"])).round().astype(np.int64)
    rng.shuffle(n)
    k = np.maximum(1, np.exp(rng.uniform(np.log(2), np.log(np.minimum(500, n // 2)))).astype(np.int64))
    d = 4.0 + 28.0 * rng.permutation(q)
    gen = _generator(seed)
    u, v, _, gv = _sbm_pairs(n.tolist(), k.tolist(), d.tolist(), gen)
    row_ptr, col, ew, src = _csr(int(n.sum()), u, v, case["wmax"], gen)
    vw = torch.zeros(int(n.sum()), dtype=torch.int64, device="cuda").index_add_(0, src, ew.to(torch.int64))
    total = torch.zeros(count, dtype=torch.int64, device="cuda").index_add_(0, gv, vw)
    return {"row_ptr": row_ptr, "col": col, "ew": ew, "vw": vw,
            "graph_ptr": np.concatenate(([0], np.cumsum(n))), "num": np.ones(count, np.int64),
            "den": total.clamp_(min=1).cpu().numpy()}


def _on_host(g: dict) -> dict:
    """The graph's arrays in pinned host memory (numpy views of them)."""
    out = {"num": g["num"], "den": g["den"], "pinned": []}
    for key in ("row_ptr", "col", "ew", "vw"):
        t = torch.empty(g[key].shape, dtype=g[key].dtype, pin_memory=True)
        t.copy_(g[key])
        out["pinned"].append(t)  # the numpy view does not own the memory
        out[key] = t.numpy()
    return out


def _served_graphs(case: dict, seed: int) -> list[dict]:
    """Requests of mixed families: sizes at even quantiles, three in ten
    R-MAT, every second one the constant Potts model."""
    rng = np.random.default_rng(seed)
    count, out = case["requests"], []
    for i in range(count):
        n = int(round(math.exp(math.log(case["n_lo"]) + (i + 0.5) / count * math.log(case["n_hi"] / case["n_lo"]))))
        one = {"wmax": 8, "cpm": i % 2 == 0}
        if i % 10 in (2, 5, 8):
            one.update(graph="rmat", scale=max(10, int(math.log2(n))))
        else:
            one.update(graph="sbm", n=n, k=max(2, int(rng.integers(2, max(3, min(500, n // 8))))),
                       d=float(rng.uniform(4.0, 32.0)))
        out.append(_on_host(_graph(one, seed * 1_000 + i)))
    return [out[i] for i in np.random.default_rng(count).permutation(count)]


_service = None


def _the_server():
    """The service a program keeps running; its requests come and go."""
    global _service
    if _service is None:
        _service = lc.Server(slots=4, max_batch=8)
    return _service


def prepare(case: dict, seed: int) -> dict:
    call = case["call"]
    if call == "batch":
        state = _batch(case, seed)
    elif call == "served":
        state = {"server": _the_server(), "graphs": _served_graphs(case, seed)}
    else:
        state = _graph(case, seed)
    if call == "host":
        state = _on_host(state)
    if call == "local_move":  # a known partition, a share of it stale
        n = state["row_ptr"].numel() - 1
        gen = _generator(seed + 1)
        labels = state["block"]
        if labels is None:
            labels = torch.arange(n, device="cuda") // 64
        wrong = _uniform(n, gen) < case["stale"]
        other = torch.minimum((_uniform(n, gen) * n).to(torch.int64), torch.tensor(n - 1, device="cuda"))
        state["labels"] = torch.where(wrong, labels[other], labels).to(torch.int32)
    if call == "objective":  # blocks, or runs of ids where there are none
        n = state["row_ptr"].numel() - 1
        labels = state["block"] if state["block"] is not None else torch.arange(n, device="cuda") // 37
        state["labels"] = labels.to(torch.int32)
    if call == "level":
        n = state["row_ptr"].numel() - 1
        labels = torch.arange(n, dtype=torch.int32, device="cuda")
        lc.lc_local_move(state["row_ptr"], state["col"], state["ew"], state["vw"], state["num"], state["den"], labels,
                         singleton_start=True)
        used, dense = torch.unique(labels, return_inverse=True)
        state["labels"], state["n_c"] = dense.to(torch.int32), used.numel()
        # the driver's buffers for the coarse level, sized once for the fine one
        state["buffers"] = {"row_ptr": torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
                            "vw": torch.zeros(n, dtype=torch.int64, device="cuda"),
                            "labels": torch.zeros(n, dtype=torch.int32, device="cuda")}
    state.pop("block", None)
    state["call"], state["case"] = call, case
    if call in ("cluster", "batch"):
        state["opts"] = lc.Options(graphs=case["replay"])
    elif call == "leiden":
        state["opts"] = lc.Options(uncoarsen=case["plus"])
    elif call == "level":
        state["opts"] = lc.Options(validate=False)  # coarse rows are not sorted
    return state


# ------------------------------------------------------------------- a pass


def _numbers(res: dict) -> dict:
    return {k: res[k] for k in ("n_clusters", "levels", "passes_total", "phi", "objective", "modularity")}


def run(state: dict) -> dict:
    call = state["call"]
    if call == "served":
        s = state["server"]
        ids = [s.submit(g["row_ptr"], g["col"], g["ew"], g["vw"], g["num"], g["den"]) for g in state["graphs"]]
        done = [s.wait(i) for i in ids]
        return {"labels": [d[0] for d in done], "phi": np.array([d[1]["phi"] for d in done])}
    g = (state["row_ptr"], state["col"], state["ew"], state["vw"])
    if call == "batch":
        labels, res = lc.lc_cluster_batch(*g, state["graph_ptr"], state["num"], state["den"], opts=state["opts"])
        return {"labels": labels, "phi": np.array([r["phi"] for r in res]),
                "n_clusters": np.array([r["n_clusters"] for r in res]),
                "modularity": np.array([r["modularity"] for r in res])}
    lam = (state["num"], state["den"])
    if call == "cluster":
        labels, res = lc.lc_cluster(*g, *lam, opts=state["opts"])
    elif call == "leiden":
        labels, res = lc.lc_cluster_leiden(*g, *lam, opts=state["opts"])
    elif call == "iterated":
        labels, res = lc.lc_cluster_iterated(*g, *lam, state["case"]["iterations"])
    elif call == "host":
        labels, res = lc.lc_cluster_host(*g, *lam)
    elif call == "local_move":
        labels, res = lc.lc_local_move(*g, *lam, state["labels"].clone())
    elif call == "objective":
        res = lc.lc_objective(*g, *lam, state["labels"])
        return _numbers(res)
    else:  # one level of a multilevel driver
        row_ptr, col, ew, vw = lc.lc_contract(*g, state["labels"], state["n_c"])
        coarse = torch.arange(state["n_c"], dtype=torch.int32, device="cuda")
        labels, res = lc.lc_local_move(row_ptr, col, ew, vw, *lam, coarse, singleton_start=True, opts=state["opts"])
        buffers = state["buffers"]
        for key, t in (("row_ptr", row_ptr), ("vw", vw), ("labels", labels)):
            buffers[key][:t.numel()].copy_(t)
        return {**buffers, **_numbers(res)}
    return {"labels": labels, **_numbers(res)}


# --------------------------------------------------------------- accounting


def _size(case: dict) -> tuple[float, float]:
    """(vertices, stored edges) of a case's graph, as expected."""
    if case["graph"] == "rmat":
        return float(1 << case["scale"]), 30.0 * (1 << case["scale"])
    if case["graph"] == "grid":
        return float(case["side"] ** 3), 6.0 * case["side"] ** 2 * (case["side"] - 1)
    return float(case["n"]), case["n"] * case["d"]


def work(case: dict) -> dict:
    """The graph read once (16 bytes a vertex, 8 a stored edge) and 4 bytes of
    label a vertex written; one gain (a multiply and an add) a stored edge."""
    if case["call"] == "batch":
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        nnz = 18.0 * n
    elif case["call"] == "served":
        n = case["requests"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        nnz = 20.0 * n
    else:
        n, nnz = _size(case)
    return {"bytes": 20.0 * n + 8.0 * nnz, "flops": 2.0 * nnz}


def exact(case: dict, seed: int):
    """The objective of a given clustering from its definition, in 64-bit
    integers; the other calls return a method's own choices (labels and what
    follows from them), for which there is no plain counterpart."""
    if case["call"] != "objective":
        return None
    s = prepare(case, seed)
    n = s["row_ptr"].numel() - 1
    deg = s["row_ptr"][1:] - s["row_ptr"][:-1]
    lab = s["labels"].to(torch.int64)
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    ew = s["ew"].to(torch.int64)
    inside = int(ew[lab[src] == lab[s["col"].to(torch.int64)]].sum())
    sizes = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, lab, s["vw"])
    squares = int((s["vw"] * s["vw"]).sum())
    phi = s["den"] * inside - s["num"] * (int((sizes * sizes).sum()) - squares)
    return {"n_clusters": None, "levels": None, "passes_total": None, "phi": phi, "objective": phi / s["den"],
            "modularity": (phi - s["num"] * squares) / (s["den"] * int(ew.sum()))}
