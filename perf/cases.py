"""The work whose speed is looked after: calls a user makes through the public entry points.

A case is one of three kinds of use:
  iter   one const_execute on tensors already in CSF form -- what an iterative decomposition does in its inner
         loop, with the same tensors and new factors;
  step   const_csf_build of every sparse operand, const_execute, release -- a tensor used once;
  csf    const_csf_build and the resulting arrays read back.
over the expressions the library is used for: TTMc and MTTKRP of order 3 and 4 (Secs. 5.2, 5.3 of the paper), the
two-contraction network with banded operands (Sec. 1) and the four-tensor running example with the printed
schedule (Sec. 4.2).  Sizes are those of workloads/generators.py and of the tests, or generic and ragged.
Coordinates are drawn on the device: Zipf slice sizes along the root mode where `slice_s` > 0, Zipf coordinates
inside a slice where `inner_s` > 0, uniform ones otherwise, duplicates drawn again.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2401_04836_b200 as cb

LETTERS = "ijkl"
RANK_LETTERS = "abc"
FACTOR_NAMES = {"ttmc": ("U", "V", "W"), "mttkrp": ("B", "C", "D")}


def _chain(name, kind, family, dims, nnz, ranks, f64=False, slice_s=0.0, inner_s=0.0):
    return {"name": name, "kind": kind, "family": family, "dims": dims, "nnz": nnz, "ranks": ranks, "f64": f64,
            "slice_s": slice_s, "inner_s": inner_s}


def _network(name, kind, n, n_k, band):
    return {"name": name, "kind": kind, "family": "network", "n": n, "n_k": n_k, "band": band, "f64": True}


def listed():
    return [
        # the smallest useful call, repeated: an inner iteration on a tensor of 20 000 nonzeros (latency)
        _chain("iter_ttmc3_20k_r8", "iter", "ttmc", "200x200x200", 20_000, "8x8"),
        # the same tensor used once: many short launches and one wait of the host
        _chain("step_ttmc3_20k_r8", "step", "ttmc", "200x200x200", 20_000, "8x8"),
        # a ragged tensor brought into CSF form in another mode order, its arrays handed on to the user's own code
        {"name": "csf_5m", "kind": "csf", "family": "csf", "dims": "60001x4099x523", "nnz": 5_000_003, "order": "1,2,0",
         "f64": False, "slice_s": 0.0, "inner_s": 0.0},
        # the headline workload: the large skewed order-3 TTMc, built and contracted once
        _chain("step_ttmc3_77m_r16", "step", "ttmc", "12000x9000x29000", 77_000_000, "16x16", slice_s=1.1, inner_s=0.9),
        # an inner iteration on a mid-sized uniform tensor with unequal ranks and odd extents
        _chain("iter_ttmc3_8m_r8x32", "iter", "ttmc", "3001x2503x4007", 8_000_009, "8x32"),
        # order 4, short fibres, the dense stage on the tensor cores
        _chain("iter_ttmc4_50m_r8", "iter", "ttmc", "20000x20000x20000x20000", 50_000_000, "8x8x8", slice_s=1.0),
        # the largest MTTKRP: an ALS sweep's inner product at rank 32
        _chain("iter_mttkrp_100m_r32", "iter", "mttkrp", "50000x50000x50000", 100_000_000, "32", slice_s=1.2),
        # the fp64 network at its full size, and a small odd one used once
        _network("iter_network_1024", "iter", 1024, 128, 32),
        _network("step_network_331", "step", 331, 61, 17),
        # a rank that is no power of two, as users choose them
        _chain("iter_ttmc3_2m_r10x12", "iter", "ttmc", "5003x3001x4001", 2_000_003, "10x12", slice_s=0.8),
        # fp64 MTTKRP of an order-4 tensor
        _chain("iter_mttkrp4_f64_1m_r16", "iter", "mttkrp", "2003x1501x701x301", 1_000_003, "16", f64=True, slice_s=0.8),
        # four sparse operands, two workspaces inside the fused loops
        {"name": "iter_example_64", "kind": "iter", "family": "example", "n": 64, "nnz": 20_000, "f64": True},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["ttmc3", "ttmc3", "mttkrp3", "ttmc4", "csf", "network", "any_rank", "mttkrp4", "example"])
    kind = rng.choice(["iter", "step"])
    skew = rng.choice([0.0, 0.8, 1.1])
    if what == "network":
        n = _log_uniform(rng, 64, 900)
        return _network(None, kind, n, _log_uniform(rng, 16, 128), max(4, n // 32))
    if what == "example":
        n = rng.randint(16, 72)
        return {"name": None, "kind": kind, "family": "example", "n": n, "nnz": int(n ** 3 * rng.uniform(0.02, 0.08)),
                "f64": rng.random() < 0.5}
    small = what in ("any_rank", "mttkrp4")
    nnz = _log_uniform(rng, 5_000, 2_000_000 if small else 30_000_000)
    side = max(20, int(nnz ** 0.5))
    order = 4 if what in ("ttmc4", "mttkrp4") else 3
    dims = "x".join(str(min(60_000, max(20, int(side * rng.uniform(0.3, 3.0)) | 1))) for _ in range(order))
    f64 = small and rng.random() < 0.5
    if what == "csf":
        order = rng.choice(["0,1,2", "1,2,0", "2,0,1"])
        return {"name": None, "kind": "csf", "family": "csf", "dims": dims, "nnz": nnz, "order": order,
                "f64": rng.random() < 0.3, "slice_s": skew, "inner_s": 0.0}
    if what == "ttmc3":
        ranks = f"{rng.choice([8, 16, 32])}x{rng.choice([8, 16, 32])}"
    elif what == "any_rank":
        ranks = f"{rng.randint(3, 32)}x{rng.randint(3, 32)}"
    elif what == "ttmc4":
        ranks = "8x8x8"
    elif what == "mttkrp3":
        ranks = str(rng.choice([8, 16, 32]))
    else:
        ranks = str(rng.randint(4, 32))
    inner = rng.choice([0.0, 0.9]) if what == "ttmc3" else 0.0
    return _chain(None, kind, "mttkrp" if "mttkrp" in what else "ttmc", dims, nnz, ranks, f64, skew, inner)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _dims(case):
    return [int(d) for d in case["dims"].split("x")]


def _ranks(case):
    return [int(r) for r in case["ranks"].split("x")]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _slice_sizes(case, dims):
    """Nonzeros per slice by falling rank, none above half of the slice's cells."""
    n0, nnz = dims[0], case["nnz"]
    w = np.arange(1, n0 + 1, dtype=np.float64) ** -case["slice_s"]
    cum = np.round(np.cumsum(w) / w.sum() * nnz).astype(np.int64)
    sizes = np.diff(cum, prepend=0)
    return np.minimum(sizes, math.prod(dims[1:]) // 2)


def _coordinates(case, dims, gen):
    """One int32 tensor per mode, distinct tuples in random order."""
    dev = "cuda"
    need = torch.zeros(dims[0], dtype=torch.int64, device=dev)
    need[torch.randperm(dims[0], generator=gen, device=dev)] = torch.from_numpy(_slice_sizes(case, dims)).to(dev)
    tables = None
    if case["inner_s"] > 0:
        tables = []
        for d in dims[1:]:
            w = torch.arange(1, d + 1, dtype=torch.float64, device=dev) ** -case["inner_s"]
            tables.append((torch.cumsum(w, 0) / w.sum(), torch.randperm(d, generator=gen, device=dev)))
    cells = math.prod(dims[1:])
    have = None
    for _ in range(6):
        key = torch.repeat_interleave(torch.arange(dims[0], device=dev), need)
        if key.numel() == 0:
            break
        for m, d in enumerate(dims[1:]):
            if tables is None:
                c = torch.randint(0, d, (key.numel(),), generator=gen, device=dev)
            else:
                at = torch.searchsorted(tables[m][0], torch.rand(key.numel(), generator=gen, device=dev, dtype=torch.float64))
                c = tables[m][1][at.clamp_(max=d - 1)]
            key = key * d + c
        if have is not None:
            key = torch.cat([have, key])
        key = torch.sort(key).values
        keep = torch.ones(key.numel(), dtype=torch.bool, device=dev)
        keep[1:] = key[1:] != key[:-1]
        fresh = key[keep]
        got = torch.bincount(fresh // cells, minlength=dims[0])
        need = (need + (torch.bincount(have // cells, minlength=dims[0]) if have is not None else 0) - got).clamp_(min=0)
        have = fresh
    have = have[torch.randperm(have.numel(), generator=gen, device=dev)]
    coords = []
    for d in reversed(dims[1:]):
        coords.append((have % d).to(torch.int32))
        have = have // d
    coords.append(have.to(torch.int32))
    return coords[::-1]


def _banded(n_a, n_b, n_k, band, gen):
    """All (a, b, k) with |a - b| < band, each kept with probability 1/4, in random order."""
    a = torch.arange(n_a, device="cuda").repeat_interleave(2 * band - 1)
    b = a + torch.arange(1 - band, band, device="cuda").repeat(n_a)
    near = (b >= 0) & (b < n_b)
    a, b = a[near], b[near]
    pair, k = torch.nonzero(torch.rand(a.numel(), n_k, generator=gen, device="cuda") < 0.25, as_tuple=True)
    perm = torch.randperm(pair.numel(), generator=gen, device="cuda")
    pair, k = pair[perm], k[perm]
    return [x.to(torch.int32) for x in (a[pair], b[pair], k)]


def _normal(shape, gen, dtype):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64).to(dtype)


def _inputs(case, seed):
    """{sparse name: (coords, vals, dims)}, {dense name: array} -- from the seed alone."""
    gen = _generator(seed)
    dtype = torch.float64 if case["f64"] else torch.float32
    if case["family"] == "network":
        n, n_k, band = case["n"], case["n_k"], case["band"]
        u = _banded(n, n, n_k, band, gen)
        w = _banded(n, n, n_k, band, gen)
        sparse = {"U": (u, _normal(u[0].numel(), gen, dtype), (n, n, n_k)),
                  "W": ([w[2], w[0], w[1]], _normal(w[0].numel(), gen, dtype), (n_k, n, n))}
        return sparse, {"V": _normal((n, n), gen, dtype)}
    if case["family"] == "example":
        n = case["n"]
        sparse = {}
        for name in "ABCD":
            key = torch.randperm(n ** 3, generator=gen, device="cuda")[: case["nnz"]]
            coords = [x.to(torch.int32) for x in (key // (n * n), key // n % n, key % n)]
            sparse[name] = (coords, _normal(case["nnz"], gen, dtype), (n, n, n))
        return sparse, {}
    dims = _dims(case)
    if case["family"] == "csf":
        # one pattern under seeded relabellings of its modes, so that the arrays of every seed have the same lengths
        coords = _coordinates(case, dims, _generator(0))
        perm = torch.randperm(coords[0].numel(), generator=gen, device="cuda")
        coords = [torch.randperm(d, generator=gen, device="cuda").to(torch.int32)[c[perm].long()] for c, d in zip(coords, dims)]
    else:
        coords = _coordinates(case, dims, gen)
    vals = (1.0 - torch.rand(coords[0].numel(), generator=gen, device="cuda", dtype=torch.float64)).to(dtype)
    sparse = {"X": (coords, vals, tuple(dims))}
    if case["family"] == "csf":
        return sparse, {}
    ranks = _ranks(case) * (1 if case["family"] == "ttmc" else len(dims) - 1)
    names = FACTOR_NAMES[case["family"]]
    return sparse, {names[m]: _normal((dims[m + 1], ranks[m]), gen, dtype) for m in range(len(dims) - 1)}


def _schedule(case):
    """(expression, tree, mode orders, loop orders, extents, output shape) of a contraction case."""
    family = case["family"]
    if family == "network":
        n = case["n"]
        return ("Z[i,m] = U[i,j,k] * V[j,l] * W[k,l,m]",
                ["T[i,k,l] = U[i,j,k] * V[j,l]", "Z[i,m] = T[i,k,l] * W[k,l,m]"],
                {"U": (0, 2, 1), "W": (1, 2, 0)}, ["ikjl", "ilmk"],
                {"i": n, "j": n, "k": case["n_k"], "l": n, "m": n}, (n, n))
    if family == "example":
        n = case["n"]
        return ("R[i,j,k] = A[i,p,q] * B[j,p,r] * C[k,q,r] * D[j,k,r]",
                ["X[i,j,q,r] = A[i,p,q] * B[j,p,r]", "Y[i,j,k,r] = X[i,j,q,r] * C[k,q,r]",
                 "R[i,j,k] = Y[i,j,k,r] * D[j,k,r]"],
                {"A": (1, 2, 0), "B": (2, 0, 1), "C": (2, 1, 0), "D": (2, 0, 1)}, ["rjpqi", "rjqki", "rjki"],
                {x: n for x in "ijkpqr"}, (n, n, n))
    dims, ranks = _dims(case), _ranks(case)
    order, names = len(dims), FACTOR_NAMES[family]
    idx = LETTERS[:order]
    extents = dict(zip(idx, dims))
    ranked = RANK_LETTERS[: order - 1] if family == "ttmc" else "r" * (order - 1)
    extents.update(zip(ranked, ranks))
    ref = lambda t, letters: f"{t}[{','.join(letters)}]"
    factors = [ref(names[m], idx[m + 1] + ranked[m]) for m in range(order - 1)]
    out_idx = "i" + (ranked if family == "ttmc" else "r")
    expression = f"{ref('Y', out_idx)} = {ref('X', idx)} * " + " * ".join(factors)
    # the leaf level first, one factor per contraction; each result keeps the levels above and the ranks so far
    tree, loops, left, left_idx = [], [], "X", idx
    for m in range(order - 2, -1, -1):
        done = ranked[m:] if family == "ttmc" else "r"
        res_idx = idx[: m + 1] + done
        result = "Y" if m == 0 else f"T{m}"
        tree.append(f"{ref(result, res_idx)} = {ref(left, left_idx)} * {factors[m]}")
        loops.append(idx[: m + 2] + done)
        left, left_idx = result, res_idx
    shape = (dims[0], *ranks) if family == "ttmc" else (dims[0], ranks[0])
    return expression, tree, {"X": tuple(range(order))}, loops, extents, shape


def prepare(case, seed):
    sparse, dense = _inputs(case, seed)
    state = {"kind": case["kind"], "sparse": sparse, "dense": dense}
    if case["family"] == "csf":
        state["mode_orders"] = {"X": tuple(int(m) for m in case["order"].split(","))}
        return state
    expression, tree, mode_orders, loops, extents, shape = _schedule(case)
    state["mode_orders"] = mode_orders
    state["plan"] = cb.const_plan_create(expression, tree, mode_orders, loops, extents, cb.F64 if case["f64"] else cb.F32)
    state["out"] = torch.empty(shape, dtype=torch.float64 if case["f64"] else torch.float32, device="cuda")
    if case["kind"] == "iter":
        state["handles"] = {n: cb.const_csf_build(c, v, d, mode_orders[n]) for n, (c, v, d) in sparse.items()}
        del state["sparse"]
    return state


def run(state):
    if state["kind"] == "csf":
        coords, vals, dims = state["sparse"]["X"]
        h = cb.const_csf_build(coords, vals, dims, state["mode_orders"]["X"])
        arrays = [a for level in range(len(dims)) for a in cb.const_csf_level(h, level)]
        arrays.append(cb.const_csf_values(h))
        cb.const_destroy(h)
        return arrays
    if state["kind"] == "iter":
        cb.const_execute(state["plan"], {**state["handles"], **state["dense"]}, state["out"])
        return state["out"]
    handles = {n: cb.const_csf_build(c, v, d, state["mode_orders"][n]) for n, (c, v, d) in state["sparse"].items()}
    cb.const_execute(state["plan"], {**handles, **state["dense"]}, state["out"])
    for h in handles.values():
        cb.const_destroy(h)
    return state["out"]


# ------------------------------------------------------------------------------------------------
# work, tolerance, 64-bit results
# ------------------------------------------------------------------------------------------------
def _nodes(case, dims):
    """Expected CSF nodes per level of a chain tensor (slices grouped by size)."""
    sizes = _slice_sizes(case, dims).astype(np.float64)
    n0 = int((sizes > 0).sum())
    levels = [n0]
    classes, counts = np.unique(np.round(np.log(np.maximum(sizes[sizes > 0], 1)) * 16) / 16, return_counts=True)
    for l in range(1, len(dims) - 1):
        cells = math.prod(dims[1 : l + 1])
        total = 0.0
        for c, k in zip(np.exp(classes), counts):
            if case["inner_s"] > 0 and l == 1:
                w = np.arange(1, dims[1] + 1, dtype=np.float64) ** -case["inner_s"]
                total += k * float(-np.expm1(-c * w / w.sum()).sum())
            else:
                total += k * cells * -math.expm1(-c / cells)
        levels.append(int(total))
    levels.append(int(sizes.sum()))
    return levels


def work(case):
    v = 8 if case["f64"] else 4
    family = case["family"]
    if family == "network":
        n, n_k, band = case["n"], case["n_k"], case["band"]
        nnz = (n * (2 * band - 1) - band * (band - 1)) * n_k // 4
        csf = 2 * nnz * (4 + v) + 8 * (n * n_k + n * (2 * band - 1))
        coo = 2 * nnz * (12 + v)
        return {"bytes": (coo if case["kind"] == "step" else csf) + 2 * v * n * n, "flops": 2 * 2 * n * nnz}
    if family == "example":
        n, nnz = case["n"], case["nnz"]
        # X[i,q] += A * B and Y[i,k] += X * C per (r, j) as a dense range where fusion leaves one, R from D's nonzeros
        flops = 2 * nnz * nnz // n + 2 * nnz * n * n + 2 * nnz * n
        return {"bytes": 4 * nnz * (12 + v) + n ** 3 * v, "flops": flops}
    dims = _dims(case)
    order = len(dims)
    n = _nodes(case, dims)
    csf = n[-1] * (4 + v) + 8 * sum(n[:-1])
    coo = n[-1] * (4 * order + v)
    if family == "csf":
        return {"bytes": coo + csf, "flops": 0}
    ranks = _ranks(case)
    flops, width = 0, 1
    for m in range(order - 2, -1, -1):
        width = width * ranks[m] if family == "ttmc" else ranks[0]
        flops += 2 * width * n[m + 1]
    rows = sum(d * (ranks[m] if family == "ttmc" else ranks[0]) for m, d in enumerate(dims[1:]))
    out = dims[0] * math.prod(ranks)
    return {"bytes": (coo if case["kind"] == "step" else csf) + v * (rows + out), "flops": flops}


def tolerance(case):
    if case["family"] == "csf":
        return "exact"
    # measured against exact(): fp64 up to 2.3e-15, fp32 up to 6.5e-7, order-4 TTMc (split tf32 operands) 8e-6
    if case["f64"]:
        return {"rel": 1e-14}
    order4 = case["family"] == "ttmc" and case["dims"].count("x") == 3
    return {"rel": 3e-5 if order4 else 3e-6}


def _exact_chain(case, sparse, dense):
    (coords, vals, dims), ranks = sparse["X"], _ranks(case)
    factors = [f.double() for f in dense.values()]
    shape = (dims[0], *ranks) if case["family"] == "ttmc" else (dims[0], ranks[0])
    step = 4_000_000
    if case["family"] == "mttkrp":
        out = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for a in range(0, vals.numel(), step):
            part = vals[a : a + step].double()[:, None]
            for c, f in zip(coords[1:], factors):
                part = part * f[c[a : a + step].long()]
            out.index_add_(0, coords[0][a : a + step].long(), part)
        return out
    order = torch.argsort(coords[0].long() * dims[1] + coords[1].long())
    i, j = coords[0][order], coords[1][order]
    new = torch.ones(order.numel(), dtype=torch.bool, device="cuda")
    new[1:] = (i[1:] != i[:-1]) | (j[1:] != j[:-1])
    fibre = torch.cumsum(new, 0) - 1
    fi, fj = i[new].long(), j[new].long()
    width = math.prod(ranks[1:])
    t = torch.zeros(fi.numel(), width, dtype=torch.float64, device="cuda")
    step = max(1, step * 16 // width)
    for a in range(0, order.numel(), step):
        o = order[a : a + step]
        part = vals[o].double()[:, None]
        for c, f in zip(coords[2:], factors[1:]):
            part = (part[:, :, None] * f[c[o].long()][:, None, :]).flatten(1)
        t.index_add_(0, fibre[a : a + step], part)
    out = torch.zeros(dims[0], ranks[0], width, dtype=torch.float64, device="cuda")
    edges = torch.searchsorted(fi, torch.arange(dims[0] + 1, device="cuda")).tolist()
    for s in range(dims[0]):
        a, b = edges[s], edges[s + 1]
        if a < b:
            torch.mm(factors[0][fj[a:b]].t(), t[a:b], out=out[s])
    return out.view(shape)


def exact(case, seed):
    if case["family"] == "csf":
        return None
    sparse, dense = _inputs(case, seed)
    if case["family"] in ("ttmc", "mttkrp"):
        return _exact_chain(case, sparse, dense)
    full = {}
    for name, (coords, vals, dims) in sparse.items():
        full[name] = torch.zeros(dims, dtype=torch.float64, device="cuda")
        full[name][tuple(c.long() for c in coords)] = vals.double()
    if case["family"] == "network":
        v = dense["V"].double()
        z = torch.zeros(case["n"], case["n"], dtype=torch.float64, device="cuda")
        for k in range(case["n_k"]):
            z += full["U"][:, :, k] @ v @ full["W"][k]
        return z
    r = torch.zeros(case["n"], case["n"], case["n"], dtype=torch.float64, device="cuda")
    for x in range(case["n"]):                                   # one value of the index r at a time
        w = torch.einsum("ipq,jp,kq->ijk", full["A"], full["B"][:, :, x], full["C"][:, :, x])
        r += w * full["D"][None, :, :, x]
    return r
