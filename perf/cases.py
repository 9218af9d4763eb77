"""The workloads whose speed this library is judged by, through its public calls.

Each case is a dict of plain values.  `kind` names the call a user's program makes:

  solve    a whole pDECO solve (deco_solve): starts, phases, rounding, cuts, best start
  phase    T steps of projected gradient ascent on a caller's block (deco_run_phase)
  batch    a population search over many graphs (deco_solve_batch)
  train    Adam steps of the learned initial mean on a batch of graphs (Mpnn.train)
  infer    the learned mean of one graph (Mpnn.infer)
  greedy   the greedy comparator (deco_greedy)
  search   the 1-flip local search of rounded vectors (deco_local_search)
  round    rounding, cuts and argmax of a block (deco_round_cut)

Graphs are drawn from the case's seed with the generators below (Erdos-Renyi
by number of edges, Barabasi-Albert, the +-1 torus), so another seed is another
graph.  `tuned` stands for a program that has the library time its launch
shapes once per graph (deco_autotune) and then keeps the handle.
"""
import math

import numpy as np
import torch

import paper_2509_18612_gb300 as deco

FP32, BF16 = deco.DECO_PREC_FP32, deco.DECO_PREC_BF16
MULTILINEAR, LAPLACIAN = deco.DECO_OBJ_MULTILINEAR01, deco.DECO_OBJ_LAPLACIAN
PREC = {"fp32": FP32, "bf16": BF16}
OBJ = {"multilinear": MULTILINEAR, "laplacian": LAPLACIAN}
INIT = {"uniform": deco.DECO_INIT_UNIFORM, "idi": deco.DECO_INIT_IDI, "dui": deco.DECO_INIT_DUI,
        "idi_half_uniform": deco.DECO_INIT_IDI_HALF_UNIFORM, "explicit": deco.DECO_INIT_EXPLICIT}


def listed():
    return [
        # the smallest call: one hundred nodes, a few dozen starts, one phase (latency)
        {"name": "solve_er100", "kind": "solve", "family": "er", "n": 100, "degree": 9.9, "weights": "unit",
         "starts": 64, "precision": "fp32", "objective": "multilinear", "init": "explicit", "steps": 500,
         "alpha": 0.01, "momentum": 0.0, "lift": 1, "lift_steps": 0, "repeats": 1, "polish": 0, "tuned": False},
        # the solver's ordinary job: a graph of 800 nodes, 1024 starts, the lifted / unlifted alternation
        {"name": "solve_er800_pdeco", "kind": "solve", "family": "er", "n": 800, "degree": 48.0, "weights": "unit",
         "starts": 1024, "precision": "fp32", "objective": "multilinear", "init": "idi_half_uniform", "steps": 800,
         "alpha": 0.01, "momentum": 0.9, "lift": 2, "lift_steps": 200, "repeats": 2, "polish": 0, "tuned": True},
        # the +-1 torus family in 16 bits, a phase on the caller's own block
        {"name": "phase_torus800_bf16", "kind": "phase", "family": "torus", "n": 800, "degree": 4.0,
         "weights": "sign", "columns": 1024, "precision": "bf16", "objective": "multilinear", "steps": 400,
         "alpha": 0.01, "momentum": 0.9, "tuned": False},
        # the large sparse graph the benchmark solves: 10^6 nodes, 128 starts in 16 bits, shapes tuned once
        {"name": "phase_er1m_bf16", "kind": "phase", "family": "er", "n": 1000000, "degree": 10.0, "weights": "unit",
         "columns": 128, "precision": "bf16", "objective": "multilinear", "steps": 30, "alpha": 0.01,
         "momentum": 0.0, "tuned": True},
        # a sparse graph with integral weights, the paper's own objective, momentum, an odd size and a ragged
        # block, 32 bits, no tuning
        {"name": "phase_er200k_weighted", "kind": "phase", "family": "er", "n": 200003, "degree": 12.0,
         "weights": "general", "columns": 100, "precision": "fp32", "objective": "laplacian", "steps": 30,
         "alpha": 0.0005, "momentum": 0.9, "tuned": False},
        # the dense graph (half of all pairs), 16 bits, shapes tuned once
        {"name": "phase_dense4096_bf16", "kind": "phase", "family": "er", "n": 4096, "degree": 2047.5,
         "weights": "unit", "columns": 128, "precision": "bf16", "objective": "multilinear", "steps": 300,
         "alpha": 0.0001, "momentum": 0.0, "tuned": True},
        # a data set of scale-free graphs with one shared hyper-parameter population
        {"name": "batch_ba48", "kind": "batch", "graphs": 48, "n_lo": 200, "n_hi": 1200, "starts": 256,
         "candidates": 32, "rounds": 2, "t_lo": 100, "t_hi": 400, "precision": "fp32"},
        # training the learned mean on a batch of small graphs (forward, backward, Adam)
        {"name": "train_48graphs", "kind": "train", "graphs": 48, "n_lo": 100, "n_hi": 800, "hidden": 64,
         "layers": 3, "steps": 10},
        # the learned mean of one larger graph, 16-bit activations
        {"name": "infer_er50k_bf16", "kind": "infer", "family": "er", "n": 50000, "degree": 10.0, "weights": "unit",
         "hidden": 64, "layers": 3, "precision": "bf16"},
        # the greedy comparator, many random orderings at once
        {"name": "greedy_er5000", "kind": "greedy", "family": "er", "n": 5000, "degree": 10.0, "weights": "unit",
         "starts": 256},
        # polishing a solver's rounded vectors to 1-flip optima
        {"name": "search_er5000", "kind": "search", "family": "er", "n": 5000, "degree": 10.0, "weights": "unit",
         "starts": 256, "max_rounds": 50, "pga_steps": 40},
        # rounding and integer cuts of the large graph's block
        {"name": "round_er1m", "kind": "round", "family": "er", "n": 1000000, "degree": 10.0, "weights": "unit",
         "starts": 128, "lift": 1, "precision": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "phase", "phase", "phase", "batch", "train", "infer", "greedy", "search",
                       "round"])
    prec = rng.choice(["fp32", "bf16"])
    weights = rng.choice(["unit", "unit", "sign", "general"])
    momentum = rng.choice([0.0, 0.9])
    if kind == "solve":
        n = _log(rng, 40, 1100)
        degree = min(rng.uniform(3.0, 48.0), 0.2 * n)
        starts = _log(rng, 8, 1024)
        lift = rng.choice([1, 2, 2, 3])
        return {"kind": kind, "family": "er", "n": n, "degree": degree, "weights": rng.choice(["unit", "sign"]),
                "starts": starts, "precision": prec, "objective": rng.choice(["multilinear", "laplacian"]),
                "init": rng.choice(["uniform", "idi", "dui", "idi_half_uniform"]), "steps": _log(rng, 50, 500),
                "alpha": 0.2 / max(degree, 4.0), "momentum": momentum, "lift": lift,
                "lift_steps": 0 if lift == 1 else _log(rng, 20, 120), "repeats": rng.choice([1, 2]),
                "polish": rng.choice([0, 20]) if prec == "bf16" else 0, "tuned": False}
    if kind == "phase":
        where = rng.choice(["small", "large", "large", "dense"])
        if where == "dense":
            n = _log(rng, 500, 4096)
            return {"kind": kind, "family": "er", "n": n, "degree": rng.uniform(0.2, 0.5) * n, "weights": "unit",
                    "columns": _log(rng, 16, 128), "precision": "bf16", "objective": "multilinear",
                    "steps": _log(rng, 20, 300), "alpha": 0.4 / (0.5 * n), "momentum": momentum, "tuned": True}
        n = _log(rng, 300, 1500) if where == "small" else _log(rng, 5000, 1000000)
        degree = rng.uniform(3.0, 24.0) if n < 100000 else rng.uniform(4.0, 10.0)
        columns = _log(rng, 8, 128) if where == "large" else _log(rng, 16, 1024)
        if prec == "fp32" and n > 500000:
            columns = min(columns, 64)
        return {"kind": kind, "family": "er", "n": n, "degree": degree, "weights": weights, "columns": columns,
                "precision": prec, "objective": rng.choice(["multilinear", "laplacian"]),
                "steps": _log(rng, 8, 30) if where == "large" else _log(rng, 30, 300),
                "alpha": (0.2 if weights != "general" else 0.06) / max(degree, 4.0), "momentum": momentum,
                "tuned": rng.random() < 0.5}
    if kind == "batch":
        candidates = rng.choice([4, 8, 16, 32])
        hi = _log(rng, 200, 1200)
        return {"kind": kind, "graphs": _log(rng, 3, 40), "n_lo": max(20, hi // 5), "n_hi": hi,
                "starts": candidates * rng.choice([2, 4, 7, 8]), "candidates": candidates, "rounds": 2, "t_lo": 40,
                "t_hi": _log(rng, 60, 400), "precision": prec}
    if kind == "train":
        hi = _log(rng, 100, 800)
        return {"kind": kind, "graphs": _log(rng, 2, 48), "n_lo": max(20, hi // 4), "n_hi": hi,
                "hidden": rng.choice([16, 32, 64, 64, 96]), "layers": rng.choice([1, 2, 3, 4]),
                "steps": rng.choice([1, 3, 10])}
    family = {"family": "er", "degree": rng.uniform(3.0, 24.0), "weights": weights}
    if kind == "infer":
        return {"kind": kind, "n": _log(rng, 300, 100000), **family, "hidden": rng.choice([16, 32, 64, 64, 100]),
                "layers": rng.choice([1, 2, 3, 4]), "precision": prec}
    if kind == "greedy":
        return {"kind": kind, "n": _log(rng, 100, 5000), **family, "starts": _log(rng, 8, 512)}
    if kind == "search":
        return {"kind": kind, "n": _log(rng, 200, 20000), **family, "starts": _log(rng, 8, 256),
                "max_rounds": rng.choice([5, 20, 50]), "pga_steps": rng.choice([0, 40])}
    n = _log(rng, 300, 1000000)
    family["degree"] = min(family["degree"], 10.0) if n > 200000 else family["degree"]
    lift = rng.choice([1, 1, 2, 3])
    return {"kind": kind, "n": n, **family, "starts": _log(rng, 8, 128) if n > 100000 else _log(rng, 8, 1024),
            "lift": lift if n <= 100000 else 1, "precision": prec}


# ---------------------------------------------------------------- graphs (host CSR, both orientations)

def _gen(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _csr(n, a, b, w):
    """Symmetric CSR of the distinct pairs (a, b), a < b, with weights w or None; sorted on the GPU."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    a, b = torch.as_tensor(a, device=dev), torch.as_tensor(b, device=dev)
    key, perm = torch.sort(torch.cat([a * n + b, b * n + a]))
    rows = torch.div(key, n, rounding_mode="floor")
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    weights = None
    if w is not None:
        w = torch.as_tensor(w, device=dev)
        weights = torch.cat([w, w])[perm].to(torch.float32).cpu().numpy()
    return (n, row_ptr.to(torch.int32).cpu().numpy(), (key - rows * n).to(torch.int32).cpu().numpy(), weights)


def _edge_weights(rng, kind, m):
    if kind == "unit":
        return None
    if kind == "sign":
        return rng.choice(np.array([-1.0, 1.0]), size=m)
    w = rng.integers(1, 8, size=m)
    return np.where(rng.random(m) < 0.3, -w, w).astype(np.float64)


def _er(n, degree, weights, rng):
    """About n * degree / 2 distinct uniform pairs."""
    total = n * (n - 1) // 2
    m = min(int(n * degree / 2), total)
    if m > total // 8:   # dense: choose among all pairs
        r, c = np.nonzero(np.tril(rng.random((n, n)) < m / total, -1))
        a, b = c.astype(np.int64), r.astype(np.int64)
    else:
        u, v = rng.integers(0, n, size=m), rng.integers(0, n, size=m)
        keep = u != v
        lo, hi = np.minimum(u, v)[keep], np.maximum(u, v)[keep]
        key = torch.unique(torch.as_tensor(lo * n + hi)).numpy()
        a, b = key // n, key % n
    return _csr(n, a, b, _edge_weights(rng, weights, a.size))


def _torus(n, weights, rng):
    ny = 20 if n % 20 == 0 else 5
    idx = np.arange(n).reshape(n // ny, ny)
    u = np.concatenate([idx.ravel(), idx.ravel()])
    v = np.concatenate([np.roll(idx, -1, 0).ravel(), np.roll(idx, -1, 1).ravel()])
    return _csr(n, np.minimum(u, v), np.maximum(u, v), _edge_weights(rng, weights, u.size))


def _ba(n, m, rng):
    """Preferential attachment: every new node links to m distinct earlier nodes by degree."""
    a, b = [], []
    pool = []
    for v in range(1, m + 1):
        for u in range(v):
            a.append(u), b.append(v)
            pool += [u, v]
    picks = rng.random((n, 4 * m))
    for v in range(m + 1, n):
        chosen = []
        for x in picks[v]:
            t = pool[int(x * len(pool))]
            if t not in chosen:
                chosen.append(t)
                if len(chosen) == m:
                    break
        for t in chosen:
            a.append(t), b.append(v)
            pool += [t, v]
    return _csr(n, np.array(a), np.array(b), None)


def _graph(case, seed):
    rng = _gen(seed, 1)
    if case["family"] == "torus":
        return _torus(case["n"], case["weights"], rng)
    return _er(case["n"], case["degree"], case["weights"], rng)


def _graph_set(case, seed):
    """Scale-free graphs (batch), or scale-free and Erdos-Renyi graphs in turn (train); sizes belong to the case."""
    rng = _gen(seed, 2)
    sizes = _gen(case["graphs"], case["n_hi"]).integers(case["n_lo"], case["n_hi"] + 1, size=case["graphs"])
    out = []
    for i, n in enumerate(int(x) for x in sizes):
        if case["kind"] == "train" and i % 2 == 0:
            out.append(_er(n, max(2.0, rng.uniform(0.01, 0.1) * n), "unit", rng))
        else:
            out.append(_ba(n, 4, rng))
    return out


def _handle(csr):
    n, rp, ci, w = csr
    return deco.deco_create_graph(n, rp, ci, w)


def _adjacency(csr, dtype=torch.float64):
    n, rp, ci, w = csr
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    val = torch.ones(ci.size, dtype=dtype) if w is None else torch.as_tensor(w).to(dtype)
    return torch.sparse_csr_tensor(torch.as_tensor(rp, dtype=torch.int64), torch.as_tensor(ci, dtype=torch.int64),
                                   val, (n, n)).to(dev)


def _cuda_rng(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + salt)


def _starts(n, columns, seed, scale):
    """Gaussian starts around a +-1 mean, scaled down: what the solver steps from."""
    g = _cuda_rng(seed, 3)
    mean = torch.randint(0, 2, (n, 1), generator=g, device="cuda").float() * 2 - 1
    return scale * (mean + math.sqrt(0.8) * torch.randn(n, columns, generator=g, device="cuda"))


# ---------------------------------------------------------------- preparation

def _schedule(case):
    unlifted = (1, case["steps"], case["alpha"], case["momentum"])
    if not case["lift_steps"]:
        return [unlifted] * case["repeats"]
    return [unlifted, (case["lift"], case["lift_steps"], 0.1 * case["alpha"], case["momentum"])] * case["repeats"]


def _x0(case, seed):
    return torch.rand(case["n"], case["starts"], generator=_cuda_rng(seed, 4), device="cuda")


def _theta(hidden, layers, seed):
    """Xavier-uniform weights and small biases, in the order the library keeps them."""
    rng = _gen(seed, 5)
    parts = [rng.uniform(-1, 1, 8 * hidden) * math.sqrt(6 / (8 + hidden)), rng.uniform(-0.1, 0.1, hidden)]
    for _ in range(layers):
        for _ in range(2):
            parts.append(rng.uniform(-1, 1, hidden * hidden) * math.sqrt(3 / hidden))
        parts.append(rng.uniform(-0.1, 0.1, hidden))
    parts.append(rng.uniform(-1, 1, hidden) * math.sqrt(6 / (hidden + 1)))
    parts.append(np.zeros(1))
    return np.concatenate(parts).astype(np.float32)


def _labels(case, seed, n):
    return torch.randint(0, 2, (n,), generator=_cuda_rng(seed, 6), device="cuda").to(torch.uint8)


def _vectors(case, csr, seed):
    """Binary columns: random, or rounded after some gradient steps from random starts."""
    n, B = case["n"], case["starts"]
    y = torch.rand(n, B, generator=_cuda_rng(seed, 7), device="cuda") * 2 - 1
    if case["pga_steps"]:
        A = _adjacency(csr, torch.float32)
        for _ in range(case["pga_steps"]):
            y = torch.clamp(y - 0.05 * (A @ y), -1, 1)
    return (y > 0).to(torch.uint8).contiguous()


def _ld(columns):
    return (columns + 63) // 64 * 64


def _block(case, columns, seed, scale):
    ld = _ld(columns)
    y = torch.zeros(case["n"], ld, device="cuda", dtype=torch.bfloat16 if case["precision"] == "bf16" else torch.float32)
    y[:, :columns] = _starts(case["n"], columns, seed, scale)
    return y


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "seed": int(seed)}
    if kind in ("batch", "train"):
        graphs = [_handle(c) for c in _graph_set(case, seed)]
        state["batch"] = deco.deco_create_batch(graphs)
        if kind == "train":
            state["model"] = deco.Mpnn(case["hidden"], case["layers"], seed)
            state["theta"] = _theta(case["hidden"], case["layers"], seed)
            state["z"] = _labels(case, seed, state["batch"].n)
            state["grad"] = torch.zeros(state["model"].n_params, device="cuda")
        return state
    csr = _graph(case, seed)
    G = state["G"] = _handle(csr)
    n = case["n"]
    if kind == "solve":
        if case["tuned"]:
            for lift in sorted({ph[0] for ph in _schedule(case)}):
                deco.deco_autotune(G, case["starts"] * lift, PREC[case["precision"]], OBJ[case["objective"]],
                                   case["momentum"], 20)
        state["params"] = deco.params(objective=OBJ[case["objective"]], precision=PREC[case["precision"]],
                                      init=INIT[case["init"]], polish_steps=case["polish"])
        state["x0"] = _x0(case, seed) if case["init"] == "explicit" else None
    elif kind == "phase":
        if case["tuned"]:
            deco.deco_autotune(G, case["columns"], PREC[case["precision"]], OBJ[case["objective"]], case["momentum"],
                               20)
        # two thirds of the way into a solve's rise: values between the tiny starts and the box's faces
        state["y0"] = _block(case, case["columns"], seed, 0.05)
        state["y"] = torch.empty_like(state["y0"])
        state["v"] = torch.empty(n, _ld(case["columns"]), device="cuda") if case["momentum"] else None
        state["args"] = deco.step_args(OBJ[case["objective"]], PREC[case["precision"]], case["alpha"],
                                       case["momentum"])
    elif kind == "infer":
        state["model"] = deco.Mpnn(case["hidden"], case["layers"], seed)
        state["model"].set_params(_theta(case["hidden"], case["layers"], seed))
        state["h"] = torch.empty(n, device="cuda")
    elif kind == "greedy":
        state["z"] = torch.empty(n, case["starts"], device="cuda", dtype=torch.uint8)
        state["cuts"] = torch.empty(case["starts"], device="cuda", dtype=torch.int64)
    elif kind == "search":
        state["z0"] = _vectors(case, csr, seed)
        state["z"] = torch.empty_like(state["z0"])
        state["cuts"] = torch.empty(case["starts"], device="cuda", dtype=torch.int64)
    else:
        columns = case["starts"] * case["lift"]
        state["y"] = _block(case, columns, seed, 0.3).clamp_(-1, 1)
        state["zbits"] = torch.empty(n, (case["starts"] + 31) // 32, device="cuda", dtype=torch.int32)
        state["cuts"] = torch.empty(case["starts"], device="cuda", dtype=torch.int64)
        state["best"] = torch.empty(1, device="cuda", dtype=torch.int32)
    torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------- one pass

def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "solve":
        res, z, cuts = deco.deco_solve(state["G"], case["starts"], _schedule(case), state["params"], seed,
                                       x0=state["x0"])
        return {"best_cut": res.best_cut, "best_init": res.best_init, "assignment": z, "phase_cuts": cuts}
    if kind == "phase":
        # the caller's block is advanced in place, from its start
        state["y"].copy_(state["y0"])
        if state["v"] is not None:
            state["v"].zero_()
        deco.deco_run_phase(state["G"], case["columns"], state["y"].shape[1], state["y"], state["v"], case["steps"],
                            state["args"])
        return {"y": state["y"]} if state["v"] is None else {"y": state["y"], "v": state["v"]}
    if kind == "batch":
        pop = deco.population(case["candidates"], case["rounds"], case["t_lo"], case["t_hi"])
        p = deco.params(precision=PREC[case["precision"]], init=deco.DECO_INIT_IDI)
        res, best, ex = deco.deco_solve_batch(state["batch"], case["starts"], p, pop, seed, want_assignment=True,
                                              want_round_cuts=True)
        return {"best": best, "assignment": ex["assignment"], "round_cuts": ex["round_cuts"],
                "scores": ex["round_scores"], "e": ex["final_e"], "T": ex["final_T"]}
    if kind == "train":
        m = state["model"]
        m.set_params(state["theta"])   # a fresh fit: the parameters, and Adam's moments at zero
        loss = m.loss_grad(state["batch"], state["z"], state["grad"], feat_seed=seed)
        losses = m.train(state["batch"], state["z"], case["steps"], lr=1e-3, feat_seed=seed)
        return {"loss": loss, "grad": state["grad"], "losses": losses, "theta": m.get_params()}
    if kind == "infer":
        state["model"].infer(state["G"], state["h"], feat_seed=seed, precision=PREC[case["precision"]])
        return {"h": state["h"]}
    if kind == "greedy":
        deco.deco_greedy(state["G"], case["starts"], seed, state["z"], state["cuts"])
        return {"z": state["z"], "cuts": state["cuts"]}
    if kind == "search":
        state["z"].copy_(state["z0"])
        rounds = deco.deco_local_search(state["G"], case["starts"], state["z"], case["max_rounds"], state["cuts"])
        return {"z": state["z"], "cuts": state["cuts"], "rounds": rounds}
    y = state["y"]
    deco.deco_round_cut(state["G"], case["starts"], case["lift"], y.shape[1], PREC[case["precision"]], y,
                        state["zbits"], state["cuts"], state["best"])
    return {"zbits": state["zbits"], "cuts": state["cuts"], "best": state["best"]}


# ---------------------------------------------------------------- work and tolerance

def _csr_bytes(case):
    nnz = case["n"] * case["degree"]
    return 4 * (case["n"] + 1) + nnz * (4 if case["weights"] == "unit" else 8)


def work(case):
    """One pass: the graph and the call's inputs read once, its results written once; the sums over the entries."""
    kind = case["kind"]
    if kind in ("batch", "train"):
        n = case["graphs"] * (case["n_lo"] + case["n_hi"]) / 2
        if kind == "batch":
            nnz = 8 * n
            columns = sum(case["starts"] * (1, 2)[r % 2] for r in range(case["rounds"]))
            return {"bytes": 4 * nnz + 4 * n + n + 8 * case["rounds"] * case["graphs"] * case["starts"],
                    "flops": 2 * nnz * columns * 0.9 * case["t_hi"]}
        h = case["hidden"]
        nnz = n * 0.5 * (8 + 0.055 * (case["n_lo"] + case["n_hi"]) / 2)
        fwd = 2 * n * (8 * h + case["layers"] * 2 * h * h) + 2 * nnz * h * case["layers"]
        passes = case["steps"] + 1
        return {"bytes": 4 * nnz + 5 * n + 4 * (8 * h + case["layers"] * 2 * h * h) * 3, "flops": 3 * fwd * passes}
    n, nnz = case["n"], case["n"] * case["degree"]
    esz = 2 if case.get("precision") == "bf16" else 4
    if kind == "solve":
        rep = case["repeats"]
        flops = 2 * nnz * case["starts"] * (case["steps"] + case["lift"] * case["lift_steps"]) * rep
        out = n + 8 * case["starts"] * len(_schedule(case))
        return {"bytes": _csr_bytes(case) + out + (4 * n * case["starts"] if case["init"] == "explicit" else 0),
                "flops": flops}
    if kind == "phase":
        block = n * case["columns"] * (2 * esz + (8 if case["momentum"] else 0))
        return {"bytes": _csr_bytes(case) + block, "flops": 2 * nnz * case["columns"] * case["steps"]}
    if kind == "infer":
        h = case["hidden"]
        return {"bytes": _csr_bytes(case) + 4 * n,
                "flops": 2 * n * (8 * h + case["layers"] * 2 * h * h) + 2 * nnz * h * case["layers"]}
    B = case["starts"]
    if kind == "greedy":
        return {"bytes": _csr_bytes(case) + n * B, "flops": 2 * nnz * B}
    if kind == "search":
        return {"bytes": _csr_bytes(case) + 2 * n * B, "flops": 4 * nnz * B}
    return {"bytes": _csr_bytes(case) + n * B * case["lift"] * esz + n * B / 8, "flops": nnz * B}


def tolerance(case):
    """Solves, batches, greedy, local search and rounding end in whole numbers: the library's sparse kernels
    perform the same 32-bit operations in one order, so they agree exactly.  A phase's block and the network's
    numbers are sums whose order is free."""
    kind = case["kind"]
    if kind == "phase":
        # about four times the distance to the 64-bit iterate; after some 50 steps entries near the box's
        # threshold between the two faces carry a rounding's difference on
        short = case["steps"] <= 50
        if case["precision"] == "bf16":   # 16-bit storage of every step's iterate
            return {"rel": 2e-2 if short else 0.15}
        return {"rel": 1e-6 if short else 1e-4}
    if kind == "train":
        return {"rel": 3e-3}   # Adam divides by the root of small second moments (gradients alone: 1e-6)
    if kind == "infer":
        return {"rel": 1.6e-2} if case["precision"] == "bf16" else {"rel": 1e-5}
    return "exact"


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

def _philox_word0(v, j, stream, seed):
    """Word 0 of Philox4x32-10 (Salmon et al., SC'11) for counters (v, j, 0, stream), key seed."""
    c = [v.astype(np.uint64), np.full(v.shape, j, np.uint64), np.zeros(v.shape, np.uint64),
         np.full(v.shape, stream, np.uint64)]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64((seed >> 32) & 0xFFFFFFFF)
    mask = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & mask, (k1 + np.uint64(0xBB67AE85)) & mask
    return c[0]


def _features(csr, seed):
    n, rp, _, _ = csr
    deg = np.diff(rp).astype(np.float64)
    x = np.zeros((n, 8))
    x[:, 0] = deg / max(deg.max(), 1.0)
    x[:, 1] = deg / (deg.mean() if deg.mean() > 0 else 1.0)
    x[:, 2] = 1.0 / np.sqrt(deg + 1.0)
    for j in range(5):
        r = _philox_word0(np.arange(n), j, 4, seed)
        x[:, 3 + j] = 2.0 * ((2 * (r >> np.uint64(9)).astype(np.float64) + 1) * 2.0 ** -24) - 1.0
    return torch.as_tensor(x.astype(np.float32).astype(np.float64))


def _net(theta, hidden, layers, x, aggregate):
    """Output o of the network; aggregate(H) is the mean over each node's neighbours."""
    pos = 0

    def take(*shape):
        nonlocal pos
        k = int(np.prod(shape))
        pos += k
        return theta[pos - k:pos].view(*shape)

    h = torch.relu(x @ take(8, hidden) + take(hidden))
    for _ in range(layers):
        ws, wn, b = take(hidden, hidden), take(hidden, hidden), take(hidden)
        h = torch.relu(h @ ws + aggregate(h) @ wn + b)
    return h @ take(hidden) + take(1)


class _Aggregate(torch.autograd.Function):
    @staticmethod
    def forward(ctx, h, A, dinv):
        ctx.A, ctx.dinv = A, dinv
        return dinv[:, None] * (A @ h)

    @staticmethod
    def backward(ctx, g):
        return ctx.A @ (ctx.dinv[:, None] * g), None, None


def _exact_steps(case, csr, y, v, steps):
    A = _adjacency(csr)
    dev = A.device
    y, v = y.to(dev), v.to(dev)
    lap = case["objective"] == "laplacian"
    d = (A @ torch.ones(case["n"], 1, dtype=torch.float64, device=dev)) if lap else None
    factor = 1.0 if lap else 2.0
    alpha, mu = float(np.float32(case["alpha"])), float(np.float32(case["momentum"]))
    for _ in range(steps):
        grad = -(A @ y)
        if lap:
            grad += d * y
        v = mu * v + grad
        y = torch.clamp(y + factor * alpha * v, -1, 1)
    return y, v


def exact(case, seed):
    kind = case["kind"]
    if kind == "phase":
        if case["n"] * case["degree"] * case["columns"] * case["steps"] > 1e11:
            return None
        C = case["columns"]
        y0 = _block(case, C, seed, 0.05).double()
        y, v = _exact_steps(case, _graph(case, seed), y0[:, :C], torch.zeros_like(y0[:, :C]), case["steps"])
        y0[:, :C] = y
        vv = torch.zeros_like(y0)
        vv[:, :C] = v
        return {"y": y0} if not case["momentum"] else {"y": y0, "v": vv}
    if kind == "solve":
        if case["init"] != "explicit" or len(_schedule(case)) > 1:
            return None   # the library's own random starts
        csr = _graph(case, seed)
        y = 2 * _x0(case, seed).double() - 1
        y, _ = _exact_steps(case, csr, y, torch.zeros_like(y), case["steps"])
        cuts, z = _exact_cuts(csr, y > 0)
        best = int(torch.argmax(cuts))
        return {"best_cut": int(cuts[best]), "best_init": best, "assignment": z[:, best].to(torch.uint8).cpu().numpy(),
                "phase_cuts": cuts[None].cpu().numpy()}
    if kind == "round":
        B, lift = case["starts"], case["lift"]
        y = _block(case, B * lift, seed, 0.3).clamp_(-1, 1)[:, :B * lift].double()
        z = y > 0 if lift == 1 else y.view(case["n"], B, lift).sum(2) >= 0
        cuts, _ = _exact_cuts(_graph(case, seed), z)
        pad = torch.zeros(case["n"], (B + 31) // 32 * 32, dtype=torch.int64, device=z.device)
        pad[:, :B] = z
        words = (pad.view(case["n"], -1, 32) << torch.arange(32, device=z.device)).sum(2)
        words = torch.where(words >= 2 ** 31, words - 2 ** 32, words).to(torch.int32)
        return {"zbits": words, "cuts": cuts, "best": torch.argmax(cuts)[None].to(torch.int32)}
    if kind == "infer":
        csr = _graph(case, seed)
        A = _adjacency(csr)
        deg = torch.as_tensor(np.diff(csr[1])).double().to(A.device)
        dinv = torch.where(deg > 0, 1 / deg.clamp(min=1), torch.zeros_like(deg))
        theta = torch.as_tensor(_theta(case["hidden"], case["layers"], seed)).double().to(A.device)
        o = _net(theta, case["hidden"], case["layers"], _features(csr, seed).to(A.device),
                 lambda h: dinv[:, None] * (A @ h))
        return {"h": torch.tanh(o)}
    if kind == "train":
        return _exact_train(case, seed)
    return None


def _exact_cuts(csr, z):
    """Cut of every binary column: (1/2) sum over stored entries of w (z_u xor z_v)."""
    A = _adjacency(csr)
    x = z.to(A.device).double()
    total = A @ torch.ones(csr[0], 1, dtype=torch.float64, device=A.device)
    cuts = (x * (total - A @ x)).sum(0)
    return torch.round(cuts).to(torch.int64), x


def _exact_train(case, seed):
    graphs = _graph_set(case, seed)
    sizes = [g[0] for g in graphs]
    n = sum(sizes)
    off = np.concatenate([[0], np.cumsum(sizes)])
    eoff = np.concatenate([[0], np.cumsum([g[2].size for g in graphs])])
    rp = np.concatenate([g[1][:-1].astype(np.int64) + e for g, e in zip(graphs, eoff)] + [eoff[-1:]])
    ci = np.concatenate([g[2].astype(np.int64) + o for g, o in zip(graphs, off)])
    A = _adjacency((n, rp, ci, None))
    dev = A.device
    deg = torch.as_tensor(np.diff(rp)).double().to(dev)
    dinv = torch.where(deg > 0, 1 / deg.clamp(min=1), torch.zeros_like(deg))
    x = torch.cat([_features(g, seed + i) for i, g in enumerate(graphs)]).to(dev)
    t = (2.0 * _labels(case, seed, n).double() - 1).to(dev)
    gid = torch.as_tensor(np.repeat(np.arange(len(sizes)), sizes)).to(dev)
    size = torch.as_tensor(sizes).double().to(dev)
    theta = torch.as_tensor(_theta(case["hidden"], case["layers"], seed)).double().to(dev).requires_grad_(True)

    def loss_grad():
        o = _net(theta, case["hidden"], case["layers"], x, lambda h: _Aggregate.apply(h, A, dinv))
        zero = torch.zeros(len(sizes), dtype=torch.float64, device=dev)
        lp = zero.index_add(0, gid, torch.nn.functional.softplus(-t * o, threshold=100)) / size
        lm = zero.index_add(0, gid, torch.nn.functional.softplus(t * o, threshold=100)) / size
        loss = torch.minimum(lp, lm).mean()
        g, = torch.autograd.grad(loss, theta)
        return float(loss.detach()), g

    loss0, grad0 = loss_grad()
    m, v = torch.zeros_like(grad0), torch.zeros_like(grad0)
    losses = []
    for k in range(1, case["steps"] + 1):
        loss, g = loss_grad()
        losses.append(loss)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        with torch.no_grad():
            theta -= 1e-3 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
    return {"loss": loss0, "grad": grad0, "losses": np.array(losses), "theta": theta.detach()}
