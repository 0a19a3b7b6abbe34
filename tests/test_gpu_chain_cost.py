"""Chains cut by cost (leaves, and for every slice as much again as it costs beyond them), against fp64 sums over the nonzeros."""
import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from tests.gpu_util import assert_close

pytestmark = pytest.mark.gpu

NAMES = {"ttmc": "UVW", "mttkrp": "BCD"}


def coordinates(sizes, dims, rng):
    """`sizes[s]` distinct nonzeros in slice s, in random order."""
    cells = int(np.prod(dims[1:], dtype=np.int64))
    inside = [(rng.integers(0, cells) + np.arange(z, dtype=np.int64) * (cells // z)) % cells for z in sizes]
    slices = np.repeat(np.arange(len(sizes)), [x.size for x in inside])
    key = np.concatenate(inside)
    perm = rng.permutation(key.size)
    slices, key = slices[perm], key[perm]
    coords = []
    for d in reversed(dims[1:]):
        coords.append((key % d).astype(np.int32))
        key = key // d
    return [slices.astype(np.int32)] + coords[::-1]


def sizes_of(what, rng):
    if what == "forties":                                  # with long fibres: a million leaves in short slices
        return np.full(26_000, 40)
    if what == "ones":                                     # every slice one leaf: chunks end in the cost behind a leaf
        return np.ones(60_000, np.int64)
    if what == "giant in front":                           # one slice over hundreds of warps, then a tail of short ones
        return np.concatenate([[180_000], rng.integers(1, 9, 20_000)])
    if what.startswith("short chunks"):                    # of little more than a slice's own cost: some warps get no leaf
        n, k = (110_000, 1800) if what == "short chunks" else (240_000, 4000)
        return (n / 6 * np.arange(1, k + 1) ** -1.1).astype(np.int64) + rng.integers(1, 40, k)
    z = (180_000 * np.arange(1, 24_001) ** -1.1).astype(np.int64) + 1
    return np.concatenate([z[:1], rng.permutation(z[1:])])


@pytest.mark.parametrize("ranks", [(8, 16), (16, 16)])
def test_short_slices_of_long_fibres(ranks):
    test_slices_of_all_sizes("long fibres", 3, ranks, cb.F32, "forties")


@pytest.mark.parametrize("what", ["ones", "giant in front", "zipf", "short chunks", "short chunks, more of them"])
@pytest.mark.parametrize("family,order,ranks,dtype", [
    ("ttmc", 3, (8, 8), cb.F32), ("ttmc", 3, (16, 32), cb.F32), ("ttmc", 3, (20, 27), cb.F64), ("mttkrp", 3, (8,), cb.F32),
    ("mttkrp", 3, (32,), cb.F32), ("mttkrp", 4, (12,), cb.F64), ("ttmc", 4, (8, 8, 8), cb.F32), ("long fibres", 3, (16, 16), cb.F32)])
def test_slices_of_all_sizes(family, order, ranks, dtype, what):
    rng = np.random.default_rng(len(what) + order + sum(ranks))
    long_fibres, family = family == "long fibres", "ttmc" if family == "long fibres" else family
    sizes = sizes_of(what, rng)
    if long_fibres:
        sizes = np.maximum(sizes, 16)                      # fibres of several leaves: two level-1 coordinates
    dims = (len(sizes), 2, 300_000) if long_fibres else (len(sizes), 700, 900) if order == 3 else (len(sizes), 90, 80, 100)
    coords = [torch.from_numpy(c).cuda() for c in coordinates(sizes, dims, rng)]
    t = torch.float32 if dtype == cb.F32 else torch.float64
    g = torch.Generator(device="cuda").manual_seed(1)
    vals = torch.randn(coords[0].numel(), generator=g, device="cuda", dtype=torch.float64).to(t)
    every = ranks if family == "ttmc" else ranks * (order - 1)
    fac = [torch.randn(d, r, generator=g, device="cuda", dtype=torch.float64).to(t) for d, r in zip(dims[1:], every)]

    idx, ranked, names = "ijkl"[:order], "abc"[: order - 1] if family == "ttmc" else "r" * (order - 1), NAMES[family]
    ref = lambda n, letters: f"{n}[{','.join(letters)}]"
    f = [ref(names[m], idx[m + 1] + ranked[m]) for m in range(order - 1)]
    out_idx = "i" + (ranked if family == "ttmc" else "r")
    tree, loops, left, left_idx = [], [], "X", idx
    for m in range(order - 2, -1, -1):
        done = ranked[m:] if family == "ttmc" else "r"
        name = "Y" if m == 0 else f"T{m}"
        tree.append(f"{ref(name, idx[: m + 1] + done)} = {ref(left, left_idx)} * {f[m]}")
        loops.append(idx[: m + 2] + done)
        left, left_idx = name, idx[: m + 1] + done
    ext = dict(zip(idx, dims))
    ext.update(zip(ranked, every))
    plan = cb.const_plan_create(f"{ref('Y', out_idx)} = {ref('X', idx)} * " + " * ".join(f), tree, {"X": tuple(range(order))}, loops, ext, dtype)
    h = cb.const_csf_build(coords, vals, dims, tuple(range(order)))
    out = torch.full((dims[0], *ranks), float("nan"), dtype=t, device="cuda")
    cb.const_execute(plan, {"X": h, **dict(zip(names, fac))}, out)
    assert cb.const_last_device_status(plan) == 0

    width = int(np.prod(ranks))
    S, A = (torch.zeros(dims[0], width, dtype=torch.float64, device="cuda") for _ in range(2))
    step = 40_000
    for a in range(0, vals.numel(), step):
        part = vals[a : a + step].double()[:, None]
        for c, x in zip(coords[1:], fac):
            row = x.double()[c[a : a + step].long()]
            part = (part[:, :, None] * row[:, None, :]).flatten(1) if family == "ttmc" else part * row
        S.index_add_(0, coords[0][a : a + step].long(), part)
        A.index_add_(0, coords[0][a : a + step].long(), part.abs())
    assert_close(out.cpu().numpy().reshape(dims[0], width), S.cpu().numpy(), A.cpu().numpy(), np.float32 if dtype == cb.F32 else np.float64)
