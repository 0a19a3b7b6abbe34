"""The leaf-balanced chain kernels against the oracle: ranks around their widths, fp32 and fp64, orders 3 and 4, windows that
end inside fibres and slices, chunks that end anywhere, and the same schedule on the generic executor."""
import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from oracle import contract as oc
from workloads import generators as gen
from workloads import mttkrp_workload, ttmc3_workload, ttmc4_workload
from tests.gpu_util import assert_close, build_csf, oracle, run_workload, to_dev

pytestmark = pytest.mark.gpu
NAMES = {"ttmc": "UVW", "mttkrp": "BCD"}


def run_chain(family, dims, ranks, X, fac, dtype, generic=False):
    """A fully fused chain over X at the given ranks; returns (output, S, A)."""
    order, idx = len(dims), "ijkl"
    ranked = "abc"[: order - 1] if family == "ttmc" else "r" * (order - 1)
    ref = lambda t, letters: f"{t}[{','.join(letters)}]"
    f = [ref(NAMES[family][m], idx[m + 1] + ranked[m]) for m in range(order - 1)]
    out_idx = "i" + (ranked if family == "ttmc" else "r")
    expr = f"{ref('Y', out_idx)} = {ref('X', idx[:order])} * " + " * ".join(f)
    tree, loops, left, left_idx = [], [], "X", idx[:order]
    for m in range(order - 2, -1, -1):
        done = ranked[m:] if family == "ttmc" else "r"
        name = "Y" if m == 0 else f"T{m}"
        tree.append(f"{ref(name, idx[: m + 1] + done)} = {ref(left, left_idx)} * {f[m]}")
        loops.append(idx[: m + 2] + done)
        left, left_idx = name, idx[: m + 1] + done
    ext = dict(zip(idx, dims))
    ext.update(zip(ranked, ranks))
    plan = cb.const_plan_create(expr, tree, {"X": tuple(range(order))}, loops, ext, dtype)
    if generic:
        cb.const_plan_set_generic_executor(plan, True)
    ops = {"X": build_csf(X, tuple(range(order)))}
    ops.update({n: to_dev(a) for n, a in fac.items()})
    shape = (dims[0], *ranks) if family == "ttmc" else (dims[0], ranks[0])
    out = torch.full(shape, float("nan"), dtype=torch.float32 if dtype == cb.F32 else torch.float64, device="cuda")
    cb.const_execute(plan, ops, out)
    assert cb.const_last_device_status(plan) == 0
    S, A = oc.nary_einsum(expr, dict(fac, X=(X.coords, X.vals)), ext)
    return out.cpu().numpy(), S, A


def inputs(family, dims, ranks, nnz, dtype, seed):
    rng = np.random.default_rng(seed)
    np_type = np.float32 if dtype == cb.F32 else np.float64
    X = gen._uniform_tensor(dims, nnz, rng, "pm1", np_type)
    fac = {n: rng.standard_normal((d, r)).astype(np_type) for n, d, r in zip(NAMES[family], dims[1:], ranks)}
    return X, fac


@pytest.mark.parametrize("dtype", [cb.F32, cb.F64])
@pytest.mark.parametrize("family,dims,ranks", [
    ("ttmc", (9, 11, 300), (1, 1)), ("ttmc", (9, 11, 300), (7, 9)), ("ttmc", (40, 30, 20), (10, 12)),
    ("ttmc", (40, 30, 20), (17, 31)), ("ttmc", (40, 30, 20), (32, 32)), ("ttmc", (3, 2, 2000), (24, 8)),
    ("ttmc", (12, 10, 9, 8), (8, 8, 8)), ("ttmc", (12, 10, 9, 8), (3, 5, 7)), ("ttmc", (2, 3, 4, 200), (8, 1, 6)),
    ("mttkrp", (30, 20, 25), (1,)), ("mttkrp", (30, 20, 25), (5,)), ("mttkrp", (30, 20, 25), (33,)),
    ("mttkrp", (2, 5, 900), (70,)), ("mttkrp", (12, 10, 9, 8), (16,)), ("mttkrp", (12, 10, 9, 8), (3,)),
    ("mttkrp", (3, 4, 5, 150), (40,)),
])
def test_ranks_around_the_widths(family, dims, ranks, dtype):
    ranks = ranks if family == "ttmc" else ranks * (len(dims) - 1)
    for nnz in (1, 31, 65, min(2500, int(np.prod(dims)))):
        X, fac = inputs(family, dims, ranks, nnz, dtype, 7 * nnz + len(dims))
        out, S, A = run_chain(family, dims, ranks, X, fac, dtype)
        assert_close(out, S, A, X.vals.dtype)


@pytest.mark.parametrize("family,dims,ranks", [("ttmc", (25, 20, 30), (6, 10)), ("mttkrp", (20, 9, 8, 7), (5, 5, 5))])
def test_agrees_with_the_generic_executor(family, dims, ranks):
    X, fac = inputs(family, dims, ranks, 1500, cb.F64, 3)
    a, S, A = run_chain(family, dims, ranks, X, fac, cb.F64)
    b, _, _ = run_chain(family, dims, ranks, X, fac, cb.F64, generic=True)
    assert_close(a, S, A, np.float64)
    assert_close(b, S, A, np.float64)


def test_generic_executor_on_off_and_on_again():
    """One plan of family "tree" that the chain kernels take: which kernels run is seen in the profile."""
    w = ttmc3_workload((25, 20, 30), 1500, (6, 10), value="pm1", config_id=31)
    S, A = oracle(w)
    plan = cb.const_plan_create(w.expression, w.tree, w.mode_orders, w.loop_orders, w.extents, cb.F32)
    assert cb.const_plan_family(plan) == "tree"
    ops = {"X": build_csf(w.sparse["X"], w.mode_orders["X"])}
    ops.update({n: to_dev(a) for n, a in w.dense.items()})
    for generic in (None, True, False, True, True, False):
        if generic is not None:
            cb.const_plan_set_generic_executor(plan, generic)
        out = torch.full(w.out_shape, float("nan"), device="cuda")
        cb.const_profile_enable(True)
        cb.const_execute(plan, ops, out)
        prof = cb.const_profile_read()
        cb.const_profile_enable(False)
        assert ("tree_kernel" in prof) == bool(generic) and ("chain3_kernel" in prof) == (not generic), (generic, prof)
        assert_close(out.cpu().numpy(), S, A, np.float32)


@pytest.mark.parametrize("family,ranks", [("ttmc", (7, 10)), ("mttkrp", (6, 6))])
def test_rows_a_tensor_does_not_name_stay_out(family, ranks):
    """A factor row that no nonzero reads may hold anything: neither padding nor unused records may touch it."""
    X, fac = inputs(family, (20, 15, 30), ranks, 700, cb.F32, 5)
    X = gen.SparseOperand([X.coords[0], np.maximum(X.coords[1], 1), X.coords[2]], X.vals, X.dims)
    key = np.unique(np.stack(X.coords), axis=1, return_index=True)[1]
    X = gen.SparseOperand([np.ascontiguousarray(c[key]) for c in X.coords], np.ascontiguousarray(X.vals[key]), X.dims)
    keep = X.coords[2] > 0
    X = gen.SparseOperand([np.ascontiguousarray(c[keep]) for c in X.coords], np.ascontiguousarray(X.vals[keep]), X.dims)
    clean, S, A = run_chain(family, X.dims, ranks, X, fac, cb.F32)
    for f in fac.values():
        f[0] = np.inf
    dirty, _, _ = run_chain(family, X.dims, ranks, X, fac, cb.F32)
    assert_close(dirty, S, A, np.float32)
    assert_close(clean, S, A, np.float32)


def test_chunks_of_a_large_skewed_tensor():
    """Several windows per chunk, slices over many chunks and many slices per chunk; long and short fibres."""
    for dims, nnz, inner in (((300, 4000, 900), 400_000, None), ((40, 30, 20000), 400_000, None), ((5000, 700, 800), 300_000, 0.9)):
        w = ttmc3_workload(dims, nnz, (9, 12), slice_s=1.1, inner_s=inner, value="pm1", config_id=21)
        out, _ = run_workload(w)
        S, A = oracle(w)
        assert_close(out, S, A, np.float32)
    w = mttkrp_workload((4000, 350, 300), 300_000, 20, slice_s=1.2, value="unit", config_id=22)
    out, _ = run_workload(w)
    S, A = oracle(w)
    assert_close(out, S, A, np.float32)
    w = ttmc4_workload((300, 40, 30, 50), 200_000, 6, slice_s=1.0, value="pm1", config_id=23)
    out, _ = run_workload(w)
    S, A = oracle(w)
    assert_close(out, S, A, np.float32)


@pytest.mark.parametrize("rank", [(8, 8), (16, 16), (32, 32), (8, 32)])
def test_short_fibres_of_a_tensor_above_a_million(rank):
    """The size and fibre length from which order-3 TTMc at a family rank takes the record walk."""
    w = ttmc3_workload((60, 40_000, 5000), 1_100_000, rank, slice_s=0.6, inner_s=None, value="pm1", config_id=24)
    out, handles = run_workload(w)
    rows = np.arange(0, 60, 7)
    S, A = oracle(w, rows)
    assert_close(out, S, A, np.float32, rows)


@pytest.mark.parametrize("family,dims,ranks,dtype", [("ttmc", (25, 20, 30), (6, 10), cb.F32), ("mttkrp", (20, 9, 8, 7), (5, 5, 5), cb.F64)])
def test_without_memory_for_padded_factors(family, dims, ranks, dtype):
    """The generic executor needs none: the call succeeds there, and nothing of the failed request stays behind."""
    X, fac = inputs(family, dims, ranks, 1500, dtype, 3)
    cb.const_debug_set(3, 1)
    try:
        out, S, A = run_chain(family, dims, ranks, X, fac, dtype)
    finally:
        cb.const_debug_set(3, 0)
    assert_close(out, S, A, X.vals.dtype)
    out, S, A = run_chain(family, dims, ranks, X, fac, dtype)
    assert_close(out, S, A, X.vals.dtype)


@pytest.mark.parametrize("dtype", [cb.F32, cb.F64])
@pytest.mark.parametrize("family,ranks,dims", [("ttmc", (8, 8), (2000, 50, 60)), ("ttmc", (16, 8), (2000, 50, 60)), ("mttkrp", (8, 8), (2000, 50, 60)),
                                               ("ttmc", (8, 8, 8), (150, 12, 10, 9)), ("mttkrp", (5, 5, 5), (400, 12, 10, 9))])
@pytest.mark.parametrize("nnz", [592, 593, 2369, 9473])
def test_short_slices_dealt_out_in_small_chunks(family, ranks, dims, dtype, nnz):
    """Chunks of one leaf, of a few, and of up to 64: around the numbers of warps that are resident at once (148 SMs times
    4 to 32), with slices of one leaf and of several chunks."""
    X, fac = inputs(family, dims, ranks, nnz, dtype, nnz + len(dims))
    hot = X.coords[0] % 7 == 0                                 # a seventh of the nonzeros into three slices
    X = gen.SparseOperand([np.where(hot, X.coords[0] % 3, X.coords[0]).astype(np.int32)] + list(X.coords[1:]), X.vals, X.dims)
    key = np.sort(np.unique(np.ravel_multi_index([c.astype(np.int64) for c in X.coords], dims), return_index=True)[1])
    X = gen.SparseOperand([np.ascontiguousarray(c[key]) for c in X.coords], np.ascontiguousarray(X.vals[key]), X.dims)
    out, S, A = run_chain(family, dims, ranks, X, fac, dtype)
    assert_close(out, S, A, X.vals.dtype)


def test_ttmc3_below_a_million_in_slices_of_several_windows():
    """The size and slice length from which order-3 TTMc takes the record walk below a million nonzeros, and just below."""
    for dims, nnz, rank in (((5000, 400, 700), 100_100, (8, 8)), ((5000, 400, 700), 99_000, (8, 8)), ((7000, 400, 700), 110_000, (16, 16)),
                            ((7500, 400, 700), 110_000, (16, 16)), ((5000, 400, 700), 110_000, (32, 32))):
        w = ttmc3_workload(dims, nnz, rank, slice_s=0.3, inner_s=None, value="pm1", config_id=25)
        out, _ = run_workload(w)
        S, A = oracle(w)
        assert_close(out, S, A, np.float32)


@pytest.mark.parametrize("extent,fused", [(40_000, True), (41_000, False)])
def test_factors_that_dwarf_the_nonzeros(extent, fused):
    """Copying a factor whole costs more than a few nonzeros are worth: from 256 padded entries per nonzero on the generic
    executor, which reads only the rows that occur, does the work."""
    w = ttmc3_workload((30, extent, extent), 5_001, (10, 12), value="pm1", config_id=33)
    assert (2 * extent * 16 <= 256 * 5_001) == fused
    cb.const_profile_enable(True)
    out, _ = run_workload(w)
    prof = cb.const_profile_read()
    cb.const_profile_enable(False)
    assert ("pad_factors" in prof) == fused and ("tree_kernel" in prof) == (not fused), prof
    S, A = oracle(w)
    assert_close(out, S, A, np.float32)


@pytest.mark.parametrize("family,ranks", [("ttmc", (8, 8)), ("ttmc", (7, 9)), ("mttkrp", (16, 16)), ("ttmc", (8, 8, 8)), ("ttmc", (5, 6, 7)), ("mttkrp", (8, 8, 8))])
@pytest.mark.parametrize("long_fibres", [False, True])
def test_products_are_formed_in_the_order_of_the_schedule(family, ranks, long_fibres):
    """Leaf value times leaf factor first, then level by level upwards: large values and leaf factors small enough to bring
    them back leave no intermediate beyond fp32, though the value times any other factor would be."""
    dims = (12, 10, 9, 11)[: len(ranks) + 1]
    X, fac = inputs(family, dims, ranks, 900, cb.F32, 51)
    if not long_fibres:                                        # one leaf to a node: the leaf coordinate from the others
        at = np.unique(np.ravel_multi_index([c.astype(np.int64) for c in X.coords[:-1]], dims[:-1]), return_index=True)[1]
        X = gen.SparseOperand([np.ascontiguousarray(c[at]) for c in X.coords], np.ascontiguousarray(X.vals[at]), X.dims)
    X = gen.SparseOperand(X.coords, X.vals * np.float32(2.0 ** 90), X.dims)
    names = NAMES[family][: len(ranks)]
    for n in names[:-1]:
        fac[n] = fac[n] * np.float32(2.0 ** 45)
    fac[names[-1]] = fac[names[-1]] * np.float32(2.0 ** -100)
    out, S, A = run_chain(family, dims, ranks, X, fac, cb.F32)
    assert_close(out, S, A, np.float32)


@pytest.mark.parametrize("dims,slice_s,inner", [
    ((40, 3, 60_000), None, None),         # 120 fibres of 27 000 leaves, each over many warps
    ((1, 3000, 2500), None, None),         # one slice
    ((3000, 5000, 400), 1.1, None),        # slices of all sizes, a hot one over hundreds of warps, fibres of a few leaves
    ((500_000, 40, 50), 0.5, None),        # more slices than a search takes in two steps, most of them of a few leaves
    ((900, 1050, 3000), None, None),       # slices of 1011 fibres, 3.4 leaves each
    ((900, 1100, 3000), None, None),       # of 1052: equal leaves again
    ((1100, 1100, 3000), None, None),      # fibres of 2.8 leaves: equal leaves again
])
def test_parts_of_equal_cost(dims, slice_s, inner):
    """From three million nonzeros on order-3 TTMc cuts the tensor by leaves and fibres together: parts begin inside fibres,
    at fibres, and at slices."""
    for rank in ((8, 8), (16, 16), (32, 32)) if dims[0] <= 40 else ((8, 8), (8, 16)):
        w = ttmc3_workload(dims, 3_100_000, rank, slice_s=slice_s, inner_s=inner, value="pm1", config_id=26)
        out, _ = run_workload(w)
        present = np.unique(w.sparse["X"].coords[0])
        rows = np.unique(np.concatenate([present[:: max(1, present.size // 40)], present[-1:]]))
        S, A = oracle(w, rows)
        assert_close(out, S, A, np.float32, rows)
        absent = np.setdiff1d(np.arange(dims[0]), present)
        assert not out[absent].any()
