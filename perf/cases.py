"""Timed cases of the sampler: what a program that uses it calls, over the
range of models that the library is for.

A case is a dict of plain values with a "kind":

  plain     a handle on one model, n plain sweeps, then the labels (and, for
            small models, the marginals) are read
  frame     new potentials for every call (set_factors), n sweeps, marginals
  cluster   Swendsen-Wang or Higdon sweeps of a ferromagnetic model, labels
  blocked   blocked (comb tree) sweeps of a lattice, labels
  learned   sweeps with the learned block proposal, labels
  batch     a round of a batch of uneven graphs: an edit from device memory
            and n sweeps, then its outcome and every class's labels
  meanfield n mean-field iterations from given marginals

listed() holds the listed cases, draw(rng) one more of the same kinds and
ranges, prepare(case, seed) what a program has in hand before the call,
run(state) one pass, work(case) what a pass cannot do without and
exact(case, seed) the float64 value of computed outputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1611_06684_gb300 import mrf as M
from paper_1611_06684_gb300 import workloads as wl

MODES = {"plain": M.MODE_PLAIN, "sw": M.MODE_SW, "higdon": M.MODE_HIGDON, "splash": M.MODE_SPLASH,
         "learned": M.MODE_LEARNED}


def listed():
    return [
        # the paper's first model: a 32 x 32 Ising grid, one chain, a hundred sweeps
        # between two looks at the marginals; the smallest call, one launch
        {"name": "ising32_c1", "kind": "plain", "graph": "grid2d", "nx": 32, "ny": 32, "nz": 1, "L": 2, "C": 1,
         "tables": "ising", "sweeps": 100, "schedule": 1, "marginals": True},
        # the paper's mixing experiment: a 50 x 50 grid, ten chains, ten sweeps between two
        # looks at the labels (the scale reduction factor is computed every ten sweeps)
        {"name": "grid50_c10", "kind": "plain", "graph": "grid2d", "nx": 50, "ny": 50, "nz": 1, "L": 2, "C": 10,
         "tables": "potts", "sweeps": 10, "schedule": 1, "marginals": True},
        # marginals of a model that is new in every call (an image, a frame of a video):
        # potentials from device memory, a short run, the marginals read back
        {"name": "frame320x240_L5_c16", "kind": "frame", "nx": 320, "ny": 240, "nz": 1, "L": 5, "C": 16,
         "sweeps": 10},
        # the benchmark's model: 128^3 lattice, 8 labels, random tables, 64 chains
        {"name": "potts128_L8_c64", "kind": "plain", "graph": "grid3d", "nx": 128, "ny": 128, "nz": 128, "L": 8,
         "C": 64, "tables": "uniform", "sweeps": 2, "schedule": 1, "marginals": False},
        # a lattice of odd sides, an odd number of labels and chains that fill no warp
        {"name": "potts61x47x53_L5_c24", "kind": "plain", "graph": "grid3d", "nx": 61, "ny": 47, "nz": 53, "L": 5,
         "C": 24, "tables": "uniform", "sweeps": 4, "schedule": 1, "marginals": False},
        # fully connected, 4,096 sites (the paper's third family at the benchmark's size)
        {"name": "dense4096_L4_c16", "kind": "plain", "graph": "dense", "N": 4096, "L": 4, "C": 16,
         "tables": "normal", "sweeps": 4, "schedule": 2, "marginals": False},
        # dynamic networks: Erdos-Renyi graphs of 2, 4, 8 and 16 labels, one chain each,
        # one per cent of the edges exchanged, then ten sweeps
        {"name": "er40_c1", "kind": "batch", "graphs": 40, "n_min": 100, "n_max": 20000, "C": 1, "sweeps": 10},
        # Swendsen-Wang on a large ferromagnetic Potts lattice
        {"name": "sw96_L8_c64", "kind": "cluster", "mode": "sw", "nx": 96, "ny": 96, "nz": 96, "L": 8, "C": 64,
         "sweeps": 2},
        # Higdon's partial Swendsen-Wang on a smaller lattice
        {"name": "higdon48_L4_c32", "kind": "cluster", "mode": "higdon", "nx": 48, "ny": 48, "nz": 48, "L": 4,
         "C": 32, "sweeps": 4},
        # blocked sweeps (exact trees inside 4 x 4 x 4 blocks)
        {"name": "splash64_L8_c64", "kind": "blocked", "nx": 64, "ny": 64, "nz": 64, "L": 8, "C": 64, "sweeps": 2},
        # learned block proposals on a preferential-attachment graph
        {"name": "learned_ba50k_L4_c32", "kind": "learned", "N": 50000, "m": 5, "L": 4, "C": 32, "hidden": 256,
         "sweeps": 4},
        # mean field from several starting points
        {"name": "meanfield48_L8_c4", "kind": "meanfield", "nx": 48, "ny": 48, "nz": 48, "L": 8, "C": 4, "iters": 4},
    ]


# ----------------------------------------------------------------------------- draws

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50.0)


def draw(rng):
    kind = rng.choice(["plain", "plain", "plain", "plain", "frame", "batch", "cluster", "cluster", "blocked",
                       "learned", "meanfield"])
    most = max(_cost(c) for c in listed())
    while True:
        L = rng.randint(2, 16)
        if kind == "plain":
            graph = rng.choice(["grid2d", "grid3d", "grid3d", "dense", "random"])
            case = {"kind": "plain", "graph": graph, "L": L, "C": _log(rng, 1, 96), "sweeps": rng.randint(1, 12),
                    "schedule": 1, "marginals": rng.random() < 0.5,
                    "tables": rng.choice(["uniform", "potts", "normal"])}
            if graph == "grid2d":
                case |= {"nx": _log(rng, 8, 700), "ny": _log(rng, 8, 700), "nz": 1}
            elif graph == "grid3d":
                case |= {"nx": _log(rng, 5, 128), "ny": _log(rng, 5, 128), "nz": _log(rng, 5, 128)}
            elif graph == "dense":
                # a site's incidences over a thread block once there are enough of them
                n = _log(rng, 40, 4096)
                case |= {"N": n, "tables": "normal", "schedule": 2 if n >= 600 else 1, "C": min(case["C"], 32),
                         "L": min(L, 6)}
            else:
                case |= {"N": _log(rng, 200, 200000), "k": rng.randint(2, 8)}
        elif kind == "frame":
            case = {"kind": "frame", "nx": _log(rng, 20, 640), "ny": _log(rng, 20, 480), "nz": 1, "L": min(L, 10),
                    "C": _log(rng, 1, 64), "sweeps": rng.randint(2, 20)}
        elif kind == "batch":
            case = {"kind": "batch", "graphs": _log(rng, 4, 40), "n_min": 50, "n_max": _log(rng, 400, 20000),
                    "C": rng.choice([1, 1, 1, 2, 4, 10]), "sweeps": rng.randint(2, 12)}
        elif kind == "cluster":
            case = {"kind": "cluster", "mode": rng.choice(["sw", "higdon"]), "nx": _log(rng, 5, 96),
                    "ny": _log(rng, 5, 96), "nz": _log(rng, 5, 96), "L": L, "C": _log(rng, 1, 96),
                    "sweeps": rng.randint(1, 6)}
        elif kind == "blocked":
            case = {"kind": "blocked", "nx": _log(rng, 5, 96), "ny": _log(rng, 5, 96), "nz": _log(rng, 5, 96), "L": L,
                    "C": _log(rng, 1, 96), "sweeps": rng.randint(1, 6)}
        elif kind == "learned":
            case = {"kind": "learned", "N": _log(rng, 500, 50000), "m": rng.randint(2, 5), "L": min(L, 8),
                    "C": _log(rng, 1, 64), "hidden": rng.choice([64, 128, 256]), "sweeps": rng.randint(1, 6)}
        else:
            case = {"kind": "meanfield", "nx": _log(rng, 5, 96), "ny": _log(rng, 5, 96), "nz": _log(rng, 5, 48),
                    "L": min(L, 10), "C": rng.randint(1, 8), "iters": rng.randint(1, 6)}
        if _cost(case) <= most and _tables(case) <= 6.3e6 * 64:
            return case


def _tables(case):
    """Table floats of a case's model."""
    return _edges(case) * _sq_labels(case)


# ----------------------------------------------------------------------------- sizes

def _sites(case):
    if case["kind"] == "batch":
        return int(case["graphs"] * (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"]))
    return case["N"] if "N" in case else case["nx"] * case["ny"] * case["nz"]


def _edges(case):
    if "nx" in case:
        x, y, z = case["nx"], case["ny"], case["nz"]
        return (x - 1) * y * z + x * (y - 1) * z + x * y * (z - 1)
    if case["kind"] == "batch":
        return int(_sites(case) * 11.5 / 2)                # mean degree U[3, 20]
    if case.get("graph") == "dense":
        return case["N"] * (case["N"] - 1) // 2
    return case["N"] * (case["m"] if "m" in case else case["k"])


def _sq_labels(case):
    """L^2 (mean over the label counts of a batch)."""
    return (4 + 16 + 64 + 256) / 4 if case["kind"] == "batch" else case["L"] ** 2


def _bits(case):
    """Dual bits of an edge (mean over the label counts of a batch)."""
    if case["kind"] == "batch":
        return (1 + 9 + 49 + 225) / 4
    diagonal = case["kind"] in ("cluster", "learned") or case.get("tables") == "potts"
    return case["L"] if diagonal and case["L"] > 2 else (case["L"] - 1) ** 2


def work(case):
    """Bytes and operations of a pass.

    A sweep reads every edge's endpoints and one weight per dual bit, every
    site's unaries, and reads and writes every label once.  Operations: two
    additions per dual bit and chain (one at either end) and the multiplies and
    logic of one 4-word random call (about 60) per 16 dual bits and per label.
    Swendsen-Wang draws one bond per edge and chain instead."""
    N, E, C, m = _sites(case), _edges(case), case["C"], _bits(case)
    L = 7.5 if case["kind"] == "batch" else case["L"]
    if case["kind"] == "meanfield":
        n = case["iters"]
        return {"bytes": n * (E * (8 + 4 * m) + N * 4 * L + 2 * 4 * N * L * C), "flops": n * E * C * m * 12.0}
    n = case["sweeps"]
    weights = 4 * L if case.get("mode") == "sw" else 4 * m
    per_edge = 60.0 if case.get("mode") == "sw" else 60.0 * math.ceil(m / 16) + 2 * m
    b, f = n * (E * (8 + weights) + 4 * N * L + 2 * N * C), n * (E * C * per_edge + N * C * (60.0 + 8 * L))
    if case["kind"] == "learned":
        rows = N / 8 * C                                  # blocks grow to 16 sites, about 6 to 10 in the mean
        h, o = case["hidden"], 16 * L
        f += n * 2.0 * rows * (o * h + h * h + h * o)
    if case["kind"] == "frame":
        b += 4 * E * case["L"] ** 2 + 4 * N * L
    if case["kind"] == "batch":
        b += 0.01 * E * (16 + 4 * _sq_labels(case))
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- models on the device

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)


def _grid_edges(nx, ny, nz):
    """The lattice's edges in canonical order: x-edges, y-edges, z-edges."""
    idx = torch.arange(nx * ny * nz, dtype=torch.int32, device="cuda").reshape(nz, ny, nx)
    s = [idx[:, :, :-1].reshape(-1), idx[:, :-1, :].reshape(-1), idx[:-1].reshape(-1)]
    t = [idx[:, :, 1:].reshape(-1), idx[:, 1:, :].reshape(-1), idx[1:].reshape(-1)]
    return torch.cat(s), torch.cat(t)


def _distinct(N, E, g):
    """About E distinct pairs s < t, in random order."""
    a = torch.randint(0, N, (E,), device="cuda", generator=g)
    b = (a + 1 + torch.randint(0, N - 1, (E,), device="cuda", generator=g)) % N
    key = torch.unique(torch.minimum(a, b) * N + torch.maximum(a, b))
    key = key[torch.randperm(key.numel(), device="cuda", generator=g)]
    return (key // N).to(torch.int32), (key % N).to(torch.int32)


def _ba_edges(N, m, seed):
    """Preferential attachment, m edges per new site: an edge's older end is the
    end of an earlier edge taken at random (so chosen with probability in
    proportion to its degree), found by following the choices back."""
    rng = np.random.default_rng(seed)
    new = np.repeat(np.arange(1, N, dtype=np.int64), m)   # the younger end of every edge
    k = np.arange(new.size, dtype=np.int64)
    first = (new - 1) * m                                 # edges of older sites: k < first
    pick = np.floor(rng.random(new.size) * 2 * first).astype(np.int64)
    old = np.where(first == 0, 0, -1)
    even = (first > 0) & (pick % 2 == 0)
    old[even] = new[pick[even] // 2]
    at = np.where(old < 0, pick // 2, k)                  # the edge whose older end is taken
    while True:
        open_ = old < 0
        if not open_.any():
            break
        got = old[at[open_]]
        where = np.flatnonzero(open_)
        old[where[got >= 0]] = got[got >= 0]
        todo = where[got < 0]
        at[todo] = at[at[todo]]
    return old.astype(np.int32), new.astype(np.int32)


def _tables_like(kind, E, L, N, g):
    """Log tables [E][L][L]: "uniform" U[-0.3, 0.3] per entry, "normal" N(0, (0.2 / sqrt N)^2) per entry
    (the fully connected family), "potts" a coupling U[0, 0.8] on the diagonal, "ising" J s t with J ~ U[0, 0.3]."""
    if kind == "uniform":
        return torch.rand((E, L, L), device="cuda", generator=g).mul_(0.6).sub_(0.3)
    if kind == "normal":
        return torch.randn((E, L, L), device="cuda", generator=g).mul_(0.2 / math.sqrt(N))
    beta = torch.rand((E, 1, 1), device="cuda", generator=g)
    if kind == "ising":
        spin = torch.tensor([-1.0, 1.0], device="cuda")
        return 0.3 * beta * spin[:, None] * spin[None, :]
    return 0.8 * beta * torch.eye(L, device="cuda")


def _model(case, seed):
    """(n_vars, unary, src, dst, pair) on the device."""
    g = _gen(seed)
    L = case["L"]
    if "nx" in case:
        s, t = _grid_edges(case["nx"], case["ny"], case["nz"])
    elif case.get("graph") == "dense":
        s, t = (x.to(torch.int32) for x in torch.triu_indices(case["N"], case["N"], 1, device="cuda"))
    elif case.get("graph") == "random":
        s, t = _distinct(case["N"], _edges(case), g)
    else:
        s, t = (torch.from_numpy(x).cuda() for x in _ba_edges(case["N"], case["m"], seed))
    N, E = _sites(case), s.numel()
    if case["kind"] == "cluster":
        beta = torch.rand((E, 1, 1), device="cuda", generator=g)
        pair, u_std = beta * torch.eye(L, device="cuda"), 0.5
        if L == 2:
            pair = pair.contiguous()
    elif case["kind"] == "learned":
        pair, u_std = _tables_like("potts", E, L, N, g), 1.0
    else:
        pair, u_std = _tables_like(case.get("tables", "uniform"), E, L, N, g), 1.0
    if case.get("tables") == "ising":
        h = 0.5 * torch.randn((N, 1), device="cuda", generator=g)
        unary = torch.cat([-h, h], 1)
    else:
        unary = u_std * torch.randn((N, L), device="cuda", generator=g)
    return N, unary.contiguous(), s.contiguous(), t.contiguous(), pair.contiguous()


# ----------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    stream = torch.cuda.Stream()
    kind = case["kind"]
    state = {"case": case, "stream": stream}
    if kind == "batch":
        return _prepare_batch(case, seed, state)
    N, unary, src, dst, pair = _model(case, seed)
    grid = (case["nx"], case["ny"], case["nz"]) if kind == "blocked" else None
    h = M.MRF(N, case["L"], case["C"], seed=seed, stream=stream.cuda_stream, grid=grid,
              schedule=case.get("schedule", 1), exact_edges=kind == "learned")
    torch.cuda.synchronize()                              # the model was made on torch's current stream
    h.set_factors(unary, src, dst, pair)
    state["h"] = h
    state["labels"] = torch.empty((case["C"], N), dtype=torch.uint8, device="cuda")
    if kind == "frame":
        state["model"] = (unary, src, dst, pair)          # this frame's potentials
    elif kind == "learned":
        blocks = wl.bfs_blocks(wl.Model(N, case["L"], None, src.cpu().numpy(), dst.cpu().numpy(), None), 16, seed=0)
        h.learned_setup(blocks, hidden=case["hidden"], seed=seed)
    elif kind == "meanfield":
        state["q"] = _start_marginals(case, seed).cpu().numpy()
    torch.cuda.synchronize()
    return state


def _start_marginals(case, seed):
    """Starting points [C][N][L]: the softmax of small random fields."""
    z = torch.randn((case["C"], _sites(case), case["L"]), device="cuda", generator=_gen(seed + 77))
    return torch.softmax(0.5 * z, dim=2)


def _er_graphs(case, seed):
    """Graphs of the batched family with distinct uniform pairs, tables U[-0.5, 0.5] and unaries N(0, 1).
    Their sizes, label counts and mean degrees belong to the case; edges and potentials come from the seed."""
    rng = np.random.default_rng(seed)
    models = []
    for sp in wl.er_batch_specs(case["graphs"], case["n_min"], case["n_max"], seed=case["n_max"]):
        N, L = sp.n_vars, sp.n_labels
        E = min(int(round(N * sp.mean_degree / 2)), N * (N - 1) // 4)
        keys = np.zeros(0, np.int64)
        while keys.size < E:
            a = rng.integers(0, N, E)
            b = (a + 1 + rng.integers(0, N - 1, E)) % N
            keys = np.unique(np.concatenate([keys, np.minimum(a, b) * N + np.maximum(a, b)]))
        keys = rng.permutation(keys)[:E]
        unary = rng.standard_normal((N, L), dtype=np.float32)
        pair = rng.random((E, L, L), dtype=np.float32) - np.float32(0.5)
        models.append(wl.Model(N, L, unary, (keys // N).astype(np.int32), (keys % N).astype(np.int32), pair))
    return models


def _prepare_batch(case, seed, state):
    models = _er_graphs(case, seed)
    b = M.MRFBatch([m.n_vars for m in models], [m.n_labels for m in models], case["C"], seed=seed,
                   stream=state["stream"].cuda_stream, schedule=1)
    b.set_factors(models)
    edits = wl.ErBatchEdits(models, [b.graph(g).first_edge_slot for g in range(len(models))], seed=seed + 1)
    arrays = edits.edit(0.01)
    n_rm, n_add, n_pair = (int(arrays[k].shape[0]) for k in (1, 2, 5))
    b.queue_create(n_rm, n_add, n_pair, 64)
    state["b"] = b
    state["n_add"] = n_add
    # as many edges come as go in every class and they take the freed slots, so the
    # same arrays are a valid edit of the next round too
    state["edit"] = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in arrays]
    state["classes"] = [b.class_handle(k) for k in range(b.n_classes())]
    state["labels"] = [torch.empty((v.C, v.N), dtype=torch.uint8, device="cuda") for v in state["classes"]]
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["b"]
        b.queue_load(*state["edit"])
        b.round(case["sweeps"])
        status, slots = b.queue_result(state["n_add"])
        return {"status": status, "slots": slots,
                "labels": [v.get_labels_into(x) for v, x in zip(state["classes"], state["labels"])]}
    h = state["h"]
    if kind == "meanfield":
        return {"q": h.mean_field(state["q"], case["iters"])}
    if kind == "frame":
        h.set_factors(*state["model"])
        h.reset_marginals(0)
        h.sweep(case["sweeps"])
        p, n = h.marginals()
        return {"p": p, "n": n}
    mode = {"plain": "plain", "blocked": "splash", "learned": "learned"}.get(kind) or case["mode"]
    h.sweep(case["sweeps"], MODES[mode])
    out = {"labels": h.get_labels_into(state["labels"])}
    if case.get("marginals"):
        out["p"], out["n"] = h.marginals()
    return out


# ----------------------------------------------------------------------------- float64 values

def exact(case, seed):
    """Mean field (the paper's Section 5.3) in float64: the dual weights of every
    table (Theorem 2 in closed form), the unaries with the tables' constant
    rows, columns and dual terms folded in, then the iterations.  Samples have
    no exact value."""
    if case["kind"] != "meanfield":
        return None
    N, unary, src, dst, pair = _model(case, seed)
    L, E = case["L"], src.numel()
    if E * (L - 1) ** 2 * case["C"] * case["iters"] > 4e9:
        return None
    s, t = src.long(), dst.long()
    w = pair.double()
    l = w[:, 1:, 1:] - w[:, 1:, :1] - w[:, :1, 1:] + w[:, :1, :1]
    a = l.abs()
    size = a + 2 * torch.log1p(torch.sqrt(-torch.expm1(-a)))
    tau = torch.where(l > 0, size, torch.where(l < 0, -size, torch.zeros_like(l)))
    a1 = torch.where(l > 0, 0.5 * (l - size), torch.where(l < 0, 0.5 * (l + size), torch.zeros_like(l)))
    a2 = torch.where(l != 0, 0.5 * (l - size), torch.zeros_like(l))
    fs = w[:, :, 0].clone()
    fs[:, 1:] += a1.sum(2)
    ft = w[:, 0, :] - w[:, :1, 0]
    ft[:, 1:] += a2.sum(1)
    u = unary.double()
    u.index_add_(0, s, fs)
    u.index_add_(0, t, ft)
    q = torch.from_numpy(_start_marginals(case, seed).cpu().numpy()).cuda().double()
    step = max(1, int(1e8 / ((L - 1) ** 2)))
    for _ in range(case["iters"]):
        for c in range(case["C"]):
            F = u.clone()
            for e0 in range(0, E, step):
                e = slice(e0, min(E, e0 + step))
                T = tau[e]
                eta = (-T.clamp(min=0) + T * q[c, s[e], 1:, None] + T.abs() * q[c, t[e], None, 1:])
                pi = torch.sigmoid(eta)
                F[:, 1:].index_add_(0, s[e], (T * pi).sum(2))
                F[:, 1:].index_add_(0, t[e], (T.abs() * pi).sum(1))
            q[c] = torch.softmax(F, dim=1)
    return {"q": q.cpu().numpy()}
