"""The work whose speed is measured: one entry per kind of call a user makes.

A partition (Algorithm 2 of the Sphynx paper) spends its time in Laplacian
block products, preconditioner applications, Gram matrices, the small
Rayleigh-Ritz problems and the multi-jagged cut.  Each is measured through its
own entry point, on the graph classes of this repository's benchmark (27-point
and 5-point meshes, random geometric graphs, R-MAT), in the precisions their
users run; two cases are whole solves.  Graphs are generated on the GPU from
the seed.

    listed()             the fixed cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handle, as a caller holds them
    run(state)           one call (or the calls of one step), with its outputs
    work(case)           bytes and operations the call cannot do without
    exact(case, seed)    the outputs in 64-bit arithmetic, where they are
                         numbers that a plain formula gives
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2105_00578_gb300 as spx

DEV = "cuda"
DTYPES = {"f64": (spx.DT_F64, torch.float64, torch.float64, 8),
          "f32": (spx.DT_F32, torch.float32, torch.float32, 4)}


# ---- the cases ------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one product on the 64 x 64 mesh of the quick-start and smoke
        # partitions, in the default precision; launch and host latency count
        {"name": "product-grid2d-f64", "kind": "product", "graph": "grid2d", "nx": 64, "ny": 64, "nz": 1,
         "weighted": False, "laplacian": "combinatorial", "dtype": "f64", "cols": 4},
        # L H and L X of every LOBPCG iteration on the headline mesh (128^3, 27-point, K = 64: 7 vectors)
        {"name": "product-mesh-f32", "kind": "product", "graph": "mesh27", "nx": 128, "ny": 128, "nz": 128,
         "weighted": False, "laplacian": "generalized", "dtype": "f32", "cols": 7},
        # the same on an irregular graph: power-law degrees, hub rows, normalized problem, K = 256 (9 vectors)
        {"name": "product-rmat-f32", "kind": "product", "graph": "rmat", "scale": 20, "graph_seed": 3,
         "weighted": False, "laplacian": "normalized", "dtype": "f32", "cols": 9},
        # the preconditioner of the headline partition: 24 chain steps with bfloat16 vectors
        {"name": "chain-mesh-mixed", "kind": "chain", "graph": "mesh27", "nx": 128, "ny": 128, "nz": 128,
         "weighted": False, "laplacian": "generalized", "precision": "mixed_bf16", "degree": 25, "cols": 7},
        # the preconditioner in the default precision, on a geometric graph whose vertex
        # numbers say nothing about position, K = 8
        {"name": "chain-rgg-f64", "kind": "chain", "graph": "rgg", "points": 300007, "graph_seed": 4,
         "weighted": False, "laplacian": "combinatorial", "precision": "fp64", "degree": 25, "cols": 4},
        # the preconditioner of a weighted power-law graph, K = 8
        {"name": "chain-rmat-weighted-mixed", "kind": "chain", "graph": "rmat", "scale": 19, "graph_seed": 5,
         "weighted": True, "laplacian": "normalized", "precision": "mixed_bf16", "degree": 25, "cols": 4},
        # one multigrid V-cycle on a mesh of odd sides
        {"name": "vcycle-mesh-f32", "kind": "vcycle", "graph": "mesh27", "nx": 101, "ny": 97, "nz": 89,
         "weighted": False, "laplacian": "combinatorial", "precision": "fp32", "cols": 7},
        # the Gram matrices of a Rayleigh-Ritz step in the default precision, generalized problem
        {"name": "gram-f64", "kind": "gram", "n": 1000003, "nblk": 3, "ld": 8, "bdiag": True},
        # the Rayleigh-Ritz problem of K = 64: 21 columns, 7 wanted
        {"name": "ritz-21", "kind": "ritz", "m": 21, "nev": 7},
        # multi-jagged cut of the headline mesh by six coordinates, and the exact cut of the result
        {"name": "cut-mesh", "kind": "cut", "graph": "mesh27", "nx": 128, "ny": 128, "nz": 128,
         "weighted": False, "dtype": "f32", "K": 64, "vweights": False},
        # the whole eigensolve of a mixed-precision mesh partition, K = 64
        {"name": "solve-mesh-mixed", "kind": "solve", "graph": "mesh27", "nx": 112, "ny": 98, "nz": 80,
         "weighted": False, "laplacian": "generalized", "precision": "mixed_bf16", "degree": 25, "nev": 7},
        # many small graphs in one call, default precision
        {"name": "batch-rgg-f64", "kind": "batch", "count": 24, "n_min": 1000, "n_max": 12000, "K": 8, "graph_seed": 4,
         "precision": "fp64", "degree": 25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, n_lo, n_hi, classes):
    """A graph of about n_lo to n_hi vertices from one of the classes."""
    g = rng.choice(classes)
    n = _log_int(rng, n_lo, n_hi)
    if g == "grid2d":
        nx = max(8, int(math.sqrt(n) * rng.uniform(0.6, 1.6)))
        return {"graph": g, "nx": nx, "ny": max(8, n // nx), "nz": 1, "weighted": rng.random() < 0.2}
    if g == "mesh27":
        s = n ** (1.0 / 3.0)
        nx, ny = max(6, int(s * rng.uniform(0.8, 1.2))), max(6, int(s * rng.uniform(0.8, 1.2)))
        return {"graph": g, "nx": nx, "ny": ny, "nz": max(6, min(n // (nx * ny), 2097152 // (nx * ny))),
                "weighted": rng.random() < 0.15}
    if g == "rgg":
        return {"graph": g, "points": max(2000, min(n, 700001)), "graph_seed": rng.randint(1, 999),
                "weighted": rng.random() < 0.2}
    return {"graph": g, "scale": max(11, min(20, int(round(math.log2(n))))), "graph_seed": rng.randint(1, 999),
            "weighted": rng.random() < 0.3}


def draw(rng):
    kind = rng.choice(["product", "product", "product", "chain", "chain", "chain", "vcycle", "gram", "ritz", "cut",
                       "solve", "batch"])
    if kind == "product":
        c = _draw_graph(rng, 3000, 2000000, ["grid2d", "mesh27", "mesh27", "rgg", "rmat"])
        return {"kind": kind, **c, "laplacian": rng.choice(["combinatorial", "generalized", "normalized"]),
                "dtype": rng.choice(["f32", "f32", "f64"]), "cols": rng.randint(2, 10)}
    if kind == "chain":
        precision = rng.choice(["mixed_bf16", "fp32", "fp64"])
        c = _draw_graph(rng, 8000, 200000 if precision == "fp64" else 1500000, ["mesh27", "mesh27", "rgg", "rmat"])
        if c["graph"] == "rmat":
            c["scale"] = min(c["scale"], 18 if precision == "fp64" else 19)
        # irregular graphs take the normalized problem with this preconditioner (the library's default too)
        lap = "normalized" if c["graph"] == "rmat" else rng.choice(["combinatorial", "generalized", "normalized"])
        return {"kind": kind, **c, "laplacian": lap, "precision": precision, "degree": rng.randint(10, 30),
                "cols": rng.randint(2, 9)}
    if kind == "vcycle":
        return {"kind": kind, **_draw_graph(rng, 20000, 900000, ["mesh27"]), "laplacian": "combinatorial",
                "precision": rng.choice(["fp32", "fp32", "fp64"]), "cols": rng.randint(2, 8)}
    if kind == "gram":
        return {"kind": kind, "n": _log_int(rng, 4000, 1000000), "nblk": rng.randint(1, 3),
                "ld": rng.choice([4, 8, 8]), "bdiag": rng.random() < 0.5}
    if kind == "ritz":
        nev = rng.randint(2, 11)
        return {"kind": kind, "m": rng.choice([nev, 2 * nev, 3 * nev, 3 * nev]), "nev": nev}
    if kind == "cut":
        return {"kind": kind, **_draw_graph(rng, 20000, 2000000, ["mesh27", "rgg", "rmat"]),
                "dtype": rng.choice(["f32", "f64"]), "K": _log_int(rng, 3, 128), "vweights": rng.random() < 0.3}
    if kind == "solve":
        # three different sides, so that no eigenvalue is (nearly) multiple
        nx = rng.randint(36, 112)
        return {"kind": kind, "graph": "mesh27", "nx": nx, "ny": int(0.875 * nx), "nz": int(0.715 * nx),
                "weighted": False, "laplacian": rng.choice(["combinatorial", "generalized"]),
                "precision": "mixed_bf16", "degree": rng.randint(15, 25), "nev": rng.randint(3, 7)}
    return {"kind": kind, "count": rng.randint(4, 24), "n_min": 1000, "n_max": _log_int(rng, 2000, 12000),
            "K": rng.choice([2, 4, 8]), "graph_seed": rng.randint(1, 999), "precision": "fp64",
            "degree": rng.randint(15, 25)}


# ---- graphs, generated on the GPU --------------------------------------------------

class _CSR:
    """row_ptr int64 [n + 1], col int32 [nnz], w float32 [nnz] or None, on the GPU."""

    def __init__(self, n, row_ptr, col, w=None):
        self.n, self.row_ptr, self.col, self.w = n, row_ptr, col, w
        self.nnz = int(col.numel())

    def rows(self):
        return torch.repeat_interleave(torch.arange(self.n, device=DEV), self.row_ptr.diff())


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 12345)
    return g


def _from_directed(n, rows, cols, w=None):
    """CSR of directed entries sorted by (row, column)."""
    order = torch.argsort(rows * n + cols)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return _CSR(n, row_ptr, cols[order].to(torch.int32), None if w is None else w[order].contiguous())


def _edge_weights(count, gen):
    return 0.5 + torch.rand(count, generator=gen, device=DEV)


def _grid(nx, ny, nz, box, gen=None):
    """Mesh graph: the 27-point box stencil, or axis neighbours only."""
    n = nx * ny * nz
    offs = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
            if (dx, dy, dz) != (0, 0, 0) and (box or abs(dx) + abs(dy) + abs(dz) == 1)]
    i = torch.arange(n, device=DEV)
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    ok = torch.stack([(x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
                      for dx, dy, dz in offs], dim=1)
    step = torch.tensor([dx + nx * (dy + ny * dz) for dx, dy, dz in offs], device=DEV)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(ok.sum(1), 0)
    rows, k = ok.nonzero(as_tuple=True)
    cols = rows + step[k]
    w = None
    if gen is not None:   # one weight per undirected edge: drawn at (smaller end, direction)
        table = 0.5 + torch.rand((n, len(offs)), generator=gen, device=DEV)
        up = cols > rows
        w = torch.where(up, table[rows, k], table[cols, len(offs) - 1 - k]).contiguous()
    return _CSR(n, row_ptr, cols.to(torch.int32), w)


def _largest_component(n, a, b):
    """Undirected edges a < b among n vertices -> (vertices, a, b) of the largest component, renumbered in order."""
    label = torch.arange(n, device=DEV)
    while True:
        new = label.clone()
        new.scatter_reduce_(0, a, label[b], "amin")
        new.scatter_reduce_(0, b, label[a], "amin")
        new = torch.minimum(new, new[new])
        new = torch.minimum(new, new[new])
        if torch.equal(new, label):
            break
        label = new
    keep = label == torch.bincount(label, minlength=n).argmax()
    new_id = torch.cumsum(keep, 0) - 1
    m = keep[a]
    return int(keep.sum()), new_id[a[m]], new_id[b[m]]


def _undirected(n, a, b, gen, weighted):
    """CSR of the largest component; `gen` draws its weights."""
    n, a, b = _largest_component(n, a, b)
    w = _edge_weights(a.numel(), gen) if weighted else None
    return _from_directed(n, torch.cat([a, b]), torch.cat([b, a]), None if w is None else torch.cat([w, w]))


# A random graph's edges come from the case's own graph_seed, so that every
# seed of a case has the same sizes; its weights and the vectors come from the seed.

def _rmat(scale, graph_seed, gen, weighted):
    """R-MAT with 16 edge draws per vertex and (0.57, 0.19, 0.19), symmetrised, largest component."""
    n, m, edges = 1 << scale, 16 << scale, _gen(graph_seed)
    src = torch.zeros(m, dtype=torch.int64, device=DEV)
    dst = torch.zeros(m, dtype=torch.int64, device=DEV)
    for level in range(scale):
        u = torch.rand(m, generator=edges, device=DEV)
        src = 2 * src + (u >= 0.76)
        dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    lo, hi = torch.minimum(src, dst), torch.maximum(src, dst)
    key = torch.unique((lo * n + hi)[lo != hi])
    return _undirected(n, key // n, key % n, gen, weighted)


def _rgg(n, graph_seed, gen, weighted):
    """Uniform points in the unit square joined within sqrt(8 / (pi n)), numbered in drawing order; its largest
    component."""
    r = math.sqrt(8.0 / (math.pi * n))
    p = torch.rand((n, 2), generator=_gen(graph_seed), device=DEV, dtype=torch.float64)
    m = max(1, int(1.0 / r))
    cell_xy = (p * m).long().clamp_(max=m - 1)
    cell = cell_xy[:, 1] * m + cell_xy[:, 0]
    order = torch.argsort(cell)
    first = torch.zeros(m * m + 1, dtype=torch.int64, device=DEV)
    first[1:] = torch.cumsum(torch.bincount(cell, minlength=m * m), 0)
    ends_a, ends_b = [], []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            cx, cy = cell_xy[:, 0] + dx, cell_xy[:, 1] + dy
            who = ((cx >= 0) & (cx < m) & (cy >= 0) & (cy < m)).nonzero().squeeze(1)
            c = cy[who] * m + cx[who]
            count = first[c + 1] - first[c]
            a = torch.repeat_interleave(who, count)
            at = torch.arange(a.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(count, 0) - count, count)
            b = order[torch.repeat_interleave(first[c], count) + at]
            near = (a < b) & ((p[a] - p[b]).square().sum(1) <= r * r)
            ends_a.append(a[near])
            ends_b.append(b[near])
    return _undirected(n, torch.cat(ends_a), torch.cat(ends_b), gen, weighted)


def _graph(case, gen):
    if case["graph"] in ("grid2d", "mesh27"):
        return _grid(case["nx"], case["ny"], case["nz"], case["graph"] == "mesh27", gen if case["weighted"] else None)
    if case["graph"] == "rgg":
        return _rgg(case["points"], case["graph_seed"], gen, case["weighted"])
    return _rmat(case["scale"], case["graph_seed"], gen, case["weighted"])


def _sizes(case):
    """Vertices and stored entries: exact for meshes, the expected ones for random graphs."""
    if case["graph"] == "rgg":
        return case["points"] * 0.99, case["points"] * 7.9
    if case["graph"] == "rmat":
        return 0.62 * (1 << case["scale"]), 30.0 * (1 << case["scale"])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    if case["graph"] == "mesh27":
        return n, (3 * nx - 2) * (3 * ny - 2) * (3 * nz - 2) - n
    return n, 2 * (3 * n - ny * nz - nx * nz - nx * ny)


class _Handle:
    """Owns a handle and keeps the device arrays that it adopted alive."""

    def __init__(self, h, *arrays):
        self.h, self.arrays = h, arrays

    def __del__(self):
        spx.sphynx_destroy(self.h)


def _create(g, vtx_w=None):
    return _Handle(spx.sphynx_create(g.row_ptr, g.col, g.w, vtx_w, g.n, g.nnz, spx.DEVICE_PTRS), g, vtx_w)


def _pad(cols):
    return (cols + 3) & ~3


def _block(n, cols, dtype, gen):
    """Random n x round4(cols) block, padding columns zero, as LOBPCG keeps its blocks."""
    x = torch.randn((n, _pad(cols)), generator=gen, device=DEV, dtype=dtype)
    x[:, cols:] = 0
    return x


# ---- prepare and run ------------------------------------------------------------------

def _options(case, seed):
    return spx.options(laplacian=case["laplacian"], precond="amg" if case["kind"] == "vcycle" else "poly",
                       poly_degree=case.get("degree", 25), precision=case["precision"], tol=1e-3, seed=seed % 1000,
                       max_iter=400)


def _chain_input(case, g, gen):
    return _block(g.n, case["cols"], torch.float64 if case["precision"] == "fp64" else torch.float32, gen)


def _spectral_coords(case, g, gen, dtype):
    """Coordinates with the smoothness of low eigenvectors and the small-scale variation of unconverged ones."""
    dims = max(1, case["K"].bit_length() - 1)
    t = torch.arange(g.n, device=DEV, dtype=torch.float64) / g.n
    freq = 1.0 + 3.0 * torch.rand(dims, generator=gen, device=DEV, dtype=torch.float64)
    c = torch.cos(math.pi * t[:, None] * freq * torch.arange(1, dims + 1, device=DEV))
    c = c + 0.3 * torch.randn((g.n, dims), generator=gen, device=DEV, dtype=torch.float64)
    return (c / math.sqrt(g.n)).to(dtype).contiguous()


def _ritz_input(case, gen):
    """G_A and G_B of a block with columns of unequal length, as LOBPCG's X, H and P are."""
    m, n = case["m"], 40 * case["m"]
    s = torch.randn((n, m), generator=gen, device=DEV, dtype=torch.float64)
    s = s * 10.0 ** (2.0 * torch.rand(m, generator=gen, device=DEV, dtype=torch.float64) - 2.0)
    lam = 10.0 ** (3.0 * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64) - 2.0)
    ga, gb = s.T @ (lam[:, None] * s), s.T @ s
    sym = lambda a: (0.5 * (a + a.T)).cpu().numpy()  # noqa: E731
    return np.ascontiguousarray(sym(ga)), np.ascontiguousarray(sym(gb))


def _gram_input(case, gen):
    n, ld, nblk = case["n"], case["ld"], case["nblk"]
    lam = 0.5 + torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    s = [torch.randn((n, ld), generator=gen, device=DEV, dtype=torch.float64) / math.sqrt(n) for _ in range(nblk)]
    ls = [lam[:, None] * b for b in s]
    bd = 1.0 + torch.randint(0, 26, (n,), generator=gen, device=DEV).double() if case["bdiag"] else None
    return s, ls, bd


def _batch_input(case, gen):
    """Weighted geometric graphs, sizes log-uniform, as one block-diagonal host CSR."""
    u = torch.rand(case["count"], generator=_gen(case["graph_seed"]), device=DEV, dtype=torch.float64).cpu().numpy()
    sizes = np.floor(case["n_min"] * (case["n_max"] / case["n_min"]) ** u).astype(np.int64)
    row_ptr, col, w, gptr = [np.zeros(1, np.int64)], [], [], [0]
    for k, n in enumerate(sizes):
        g = _rgg(int(n), case["graph_seed"] + k, gen, True)
        row_ptr.append(g.row_ptr[1:].cpu().numpy() + row_ptr[-1][-1])
        col.append(g.col.cpu().numpy() + np.int32(gptr[-1]))
        w.append(g.w.cpu().numpy())
        gptr.append(gptr[-1] + g.n)
    return np.concatenate(row_ptr), np.concatenate(col), np.concatenate(w), np.array(gptr, np.int64)


def prepare(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "product":
        g = _graph(case, gen)
        code, dtype, out, _ = DTYPES[case["dtype"]]
        x = _block(g.n, case["cols"], dtype, gen)
        return {"kind": kind, "h": _create(g), "lap": case["laplacian"], "code": code, "cols": case["cols"],
                "x": x, "y": torch.zeros(x.shape, device=DEV, dtype=out)}
    if kind in ("chain", "vcycle"):
        g = _graph(case, gen)
        h, opt = _create(g), _options(case, seed)
        spx.sphynx_precond_setup(h.h, opt)
        r = _chain_input(case, g, gen)
        return {"kind": kind, "h": h, "opt": opt, "cols": case["cols"], "r": r, "out": torch.zeros_like(r)}
    if kind == "gram":
        s, ls, bd = _gram_input(case, gen)
        return {"kind": kind, "s": s, "ls": ls, "bd": bd, "ld": case["ld"], "n": case["n"]}
    if kind == "ritz":
        ga, gb = _ritz_input(case, gen)
        return {"kind": kind, "ga": ga, "gb": gb, "active": np.ones(case["m"], np.int32), "nev": case["nev"]}
    if kind == "cut":
        g = _graph(case, gen)
        code, dtype, _, _ = DTYPES[case["dtype"]]
        vw = torch.randint(1, 10, (g.n,), generator=gen, device=DEV) if case["vweights"] else None
        return {"kind": kind, "h": _create(g, vw), "vw": vw, "code": code, "K": case["K"],
                "coords": _spectral_coords(case, g, gen, dtype),
                "part": torch.zeros(g.n, dtype=torch.int32, device=DEV)}
    if kind == "solve":
        g = _graph(case, gen)
        return {"kind": kind, "h": _create(g), "opt": _options(case, seed), "nev": case["nev"],
                "x": torch.zeros((g.n, _pad(case["nev"])), device=DEV)}
    row_ptr, col, w, gptr = _batch_input(case, gen)
    opt = spx.options(laplacian="combinatorial", precond="poly", poly_degree=case["degree"],
                      precision=case["precision"], tol=1e-3, seed=seed % 1000, max_iter=600)
    return {"kind": kind, "h": _Handle(spx.sphynx_create_batch(row_ptr, col, gptr, edge_w=w)), "K": case["K"],
            "count": case["count"], "opt": opt, "part": np.zeros(int(gptr[-1]), np.int32)}


def run(state):
    kind = state["kind"]
    if kind == "product":
        ld = state["x"].shape[1]
        spx.sphynx_laplacian_apply(state["h"].h, state["lap"], state["code"], state["x"], ld, state["y"], ld,
                                   state["cols"])
        return state["y"]
    if kind in ("chain", "vcycle"):
        spx.sphynx_precond_apply(state["h"].h, state["opt"], state["r"], state["out"], state["r"].shape[1],
                                 state["cols"])
        return state["out"]
    if kind == "gram":
        return spx.sphynx_gram(spx.DT_F64, state["s"], state["ls"], state["ld"], state["n"], state["bd"])
    if kind == "ritz":
        theta, y, _ = spx.sphynx_rayleigh_ritz(state["ga"], state["gb"], state["active"], state["nev"], 2.0 ** -53)
        return theta, y
    if kind == "cut":
        dims = state["coords"].shape[1]
        spx.sphynx_mj(state["code"], state["coords"], dims, dims, state["part"].numel(), state["vw"], state["K"],
                      state["part"])
        return (state["part"], *spx.sphynx_eval(state["h"].h, state["part"], state["K"]))
    if kind == "solve":
        _, theta, res, _ = spx.sphynx_eigensolve(state["h"].h, state["opt"], state["nev"], state["x"],
                                                 state["x"].shape[1])
        return state["x"], theta, res
    _, cuts, imbalances, eigs, iters, _, _ = spx.sphynx_partition_batch(state["h"].h, state["K"], state["opt"],
                                                                        state["part"], state["count"])
    return state["part"], cuts, imbalances, eigs, iters


# ---- work: each input read once, each output written once ---------------------------------

def work(case):
    kind = case["kind"]
    if kind == "gram":
        m = case["nblk"] * case["ld"]
        return {"bytes": case["n"] * 8.0 * (2 * m + (1 if case["bdiag"] else 0)) + 16.0 * m * m,
                "flops": 2.0 * case["n"] * m * (m + 1)}
    if kind == "ritz":
        m, nev = case["m"], case["nev"]   # Cholesky, its inverse, the projection and a tridiagonal eigensolve
        return {"bytes": 8.0 * (2 * m * m + m * nev + nev), "flops": m ** 3 * (1 / 3 + 1 / 3 + 2 + 4 / 3)}
    if kind == "batch":
        n = case["count"] * (case["n_max"] - case["n_min"]) / max(1e-9, math.log(case["n_max"] / case["n_min"]))
        return {"bytes": n * (8 + 7.9 * 8 + 4), "flops": 2.0 * 7.9 * n * _pad(case["K"].bit_length()) * case["degree"]}
    n, nnz = _sizes(case)
    graph = 8.0 * (n + 1) + nnz * (8.0 if case["weighted"] else 4.0)
    if kind == "cut":
        dims = max(1, case["K"].bit_length() - 1)
        return {"bytes": graph + n * (dims * DTYPES[case["dtype"]][3] + 4.0 + (8.0 if case["vweights"] else 0.0)),
                "flops": nnz}
    cols = case["nev"] if kind == "solve" else case["cols"]
    size = 8.0 if case.get("dtype") == "f64" or case.get("precision") == "fp64" else 4.0
    products = {"product": 1, "chain": case.get("degree", 1) - 1, "vcycle": 6, "solve": case.get("degree", 1) + 1}[kind]
    return {"bytes": graph + n * size * cols * (1.0 if kind == "solve" else 2.0), "flops": 2.0 * nnz * cols * products}


# ---- the same results in 64-bit arithmetic --------------------------------------------

class _Laplacian:
    """L X in double with torch's sparse product."""

    def __init__(self, g, lap):
        w = torch.ones(g.nnz, dtype=torch.float64, device=DEV) if g.w is None else g.w.double()
        rows, cols = g.rows(), g.col.long()
        self.deg = torch.zeros(g.n, dtype=torch.float64, device=DEV).index_add_(0, rows, w)
        self.normalized = lap == "normalized"
        if self.normalized:
            s = self.deg.rsqrt()
            w = w * s[rows] * s[cols]
        self.a = torch.sparse_csr_tensor(g.row_ptr, cols, w, size=(g.n, g.n))

    def __call__(self, x):
        d = 1.0 if self.normalized else self.deg[:, None]
        return d * x - self.a @ x

    def null(self):
        return self.deg.sqrt() if self.normalized else torch.ones_like(self.deg)


def _mix64(z):
    """SplitMix64's output function."""
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _polynomial_roots(apply, null, n, degree, seed):
    """Harmonic Ritz values of `degree` Lanczos steps from the seeded start vector, with the copies that keep the
    polynomial positive."""
    gamma = np.uint64(0x9E3779B97F4A7C15)
    with np.errstate(over="ignore"):
        key = _mix64(np.uint64(seed) + np.uint64(3) * gamma)
        z = _mix64(key + np.arange(1, n + 1, dtype=np.uint64) * gamma)
    v = torch.from_numpy(2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0).to(DEV)
    null = null / null.norm()
    basis = [null]
    v = v - (null @ v) * null
    v = v / v.norm()
    t = np.zeros((degree, degree))
    for j in range(degree):
        basis.append(v)
        w = apply(v[:, None])[:, 0]
        t[j, j] = float(v @ w)
        q = torch.stack(basis)
        for _ in range(2):
            w = w - q.T @ (q @ w)
        beta = float(w.norm())
        if j + 1 < degree:
            t[j, j + 1] = t[j + 1, j] = beta
        v = w / beta
    m = t @ t
    m[-1, -1] += beta ** 2
    c = np.linalg.inv(np.linalg.cholesky(t))
    m = c @ m @ c.T
    base = np.linalg.eigvalsh(0.5 * (m + m.T))
    roots = list(base)
    lam = base[-1] * np.arange(1, 8193) / 8192
    for _ in range(4):
        p = (1.0 - np.prod([1.0 - lam / x for x in roots], axis=0)) / lam
        k = int(np.argmin(p))
        if p[k] > 0.0:
            break
        roots.append(base[int(np.argmin(np.abs(base - lam[k])))])
    if len(roots) % 2 == 0:
        roots.append(base[-1])
    # largest first, then each root as far as possible from those before it: the factors' order for stability
    left, order = list(roots), []
    while left:
        score = [sum(math.log(abs(x - y)) if x != y else -math.inf for y in order) if order else x for x in left]
        order.append(left.pop(int(np.argmax(score))))
    return order


def exact(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "product":
        g = _graph(case, gen)
        x = _block(g.n, case["cols"], DTYPES[case["dtype"]][1], gen)
        return _Laplacian(g, case["laplacian"])(x.double())
    if kind == "chain":
        g = _graph(case, gen)
        t = _chain_input(case, g, gen).double()
        lap = _Laplacian(g, case["laplacian"])
        roots = _polynomial_roots(lap, lap.null(), g.n, case["degree"], seed % 1000)
        y = torch.zeros_like(t)
        for i, x in enumerate(roots):
            y += t / x
            if i + 1 < len(roots):
                t = t - lap(t) / x
        return y
    if kind == "gram":
        s, ls, bd = _gram_input(case, gen)
        s, ls = torch.cat(s, 1), torch.cat(ls, 1)
        return s.T @ ls, s.T @ (s if bd is None else bd[:, None] * s)
    if kind == "ritz":
        ga, gb = _ritz_input(case, gen)
        d = 1.0 / np.sqrt(np.diag(gb))
        c = np.linalg.inv(np.linalg.cholesky(d[:, None] * gb * d)).T   # upper triangular R^{-1}
        w = c.T @ (d[:, None] * ga * d) @ c
        theta, w = np.linalg.eigh(0.5 * (w + w.T))
        theta, w = theta[:case["nev"]], w[:, :case["nev"]]
        w = w * np.sign(w[np.argmax(np.abs(w), axis=0), np.arange(w.shape[1])])
        return theta, d[:, None] * (c @ w)
    # the multigrid hierarchy is the framework's own choice of aggregates; cuts
    # are whole numbers; a solve stops where its tolerance is met
    return None
