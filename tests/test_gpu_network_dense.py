"""The two-contraction network where its operands have locality (the fp64 matrix pipe), and where they do not, or must not be
written out densely: against the oracle, element by element."""
import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from workloads import generators as gen
from workloads import network_workload
from tests.gpu_util import assert_close, oracle, run_workload, to_dev

pytestmark = pytest.mark.gpu


def kernels_of(w):
    """Output and the time of each kernel (a kernel that leaves the work to another returns at once)."""
    cb.const_profile_enable(True)
    out, _ = run_workload(w)
    prof = cb.const_profile_read()
    cb.const_profile_enable(False)
    return out, prof


@pytest.mark.parametrize("n,n_k,band,keep", [
    (331, 61, 17, 0.25),      # nothing a multiple of a tile
    (300, 128, 12, 0.3),      # a full tile of k
    (260, 150, 12, 0.3),      # two tiles of k, the second of 22
    (400, 7, 39, 0.6),        # the widest range of m that qualifies with four slices together (80)
    (400, 9, 40, 0.6),        # one that does not (82)
    (603, 33, 3, 1.0),        # narrow and full
])
def test_banded(n, n_k, band, keep):
    w = network_workload(n, n_k, band, keep, config_id=61)
    out, prof = kernels_of(w)
    assert "network_t" in prof and "network_kernel" in prof
    S, A = oracle(w)
    assert_close(out, S, A, np.float64)


def matrix_form_alone(w):
    """The output where only the matrix form is let run: zero if the device hands the work on."""
    cb.const_debug_set(2, 6)
    try:
        out, _ = run_workload(w)
    finally:
        cb.const_debug_set(2, 0)
    return out


def bands(n, n_k, band_u, band_w, keep_u, keep_w):
    """U and W of two bands of their own."""
    w = network_workload(n, n_k, band_u, keep_u, config_id=65)
    w.sparse["W"] = network_workload(n, n_k, band_w, keep_w, config_id=66).sparse["W"]
    return w


@pytest.mark.parametrize("band_u,band_w,keep_u,keep_w,taken", [
    (48, 10, 0.6, 0.6, True),        # 95 neighbouring j of 96
    (49, 10, 0.6, 0.6, False),       # 97
    (10, 39, 0.6, 0.6, True),        # four slices of W together: 80 neighbouring m of 80
    (10, 40, 0.6, 0.6, False),       # 82
    (16, 16, 0.17, 0.17, True),      # 6 to 7 dense multiply-adds per sparse one
    (16, 16, 0.1, 0.1, False),       # 11
])
def test_which_operands_the_matrix_form_takes(band_u, band_w, keep_u, keep_w, taken):
    w = bands(500, 24, band_u, band_w, keep_u, keep_w)
    S, A = oracle(w)
    out, _ = run_workload(w)
    assert_close(out, S, A, np.float64)
    alone = matrix_form_alone(w)
    if taken:
        assert_close(alone, S, A, np.float64)
    else:
        assert not alone.any()


def test_the_matrix_form_rounds_no_more_than_the_gather_form():
    """Relative 2-norm of the error of either form; the sums over k and l must not run in one chain of additions (which gave
    3.0e-16 here against 2.6e-16 of the gather form)."""
    w = network_workload(331, 61, 17, 0.25, config_id=68)
    S, _ = oracle(w)
    matrix = matrix_form_alone(w)
    cb.const_debug_set(3, 1)                                     # no memory for T: the gather form
    try:
        gather, _ = run_workload(w)
    finally:
        cb.const_debug_set(3, 0)
    error = [np.linalg.norm(x - S) for x in (matrix, gather)]
    assert 0 < error[0] <= error[1]


def test_an_infinity_in_a_later_chunk():
    """Products of the first chunk of slices have been added to Z when a T of the second turns out not to be finite: Z starts
    again in the gather form.  (T of 1024 slices takes 335 MB, a chunk at most 256.)"""
    w = network_workload(1024, 40, 6, 0.5, config_id=67)
    U = w.sparse["U"]
    keep = U.coords[1] != 1000
    w.sparse["U"] = gen.SparseOperand([np.ascontiguousarray(c[keep]) for c in U.coords], np.ascontiguousarray(U.vals[keep]), U.dims)
    rows = np.concatenate([np.arange(0, 1024, 61), np.arange(994, 1007)])
    S, A = oracle(w, rows)
    assert_close(matrix_form_alone(w), S, A, np.float64, rows)
    w.dense["V"][1000] = np.inf
    out, prof = kernels_of(w)
    assert prof["network_t"][0] == 2
    assert_close(out, S, A, np.float64, rows)
    assert not matrix_form_alone(w).any()


def scattered(n, n_k, nnz, seed):
    w = network_workload(n, n_k, 4, 0.25, config_id=62)
    rng = np.random.default_rng(seed)
    w.sparse["U"] = gen._uniform_tensor((n, n, n_k), nnz, rng, "normal", np.float64)
    w.sparse["W"] = gen._uniform_tensor((n_k, n, n), nnz, rng, "normal", np.float64)
    return w


def test_operands_without_locality():
    w = scattered(400, 20, 150_000, 1)
    out, prof = kernels_of(w)
    assert "network_t" in prof                                 # (asked for, and handed on by the device)
    S, A = oracle(w)
    assert_close(out, S, A, np.float64)
    assert not matrix_form_alone(w).any()


def test_rows_and_slices_missing():
    """Slices of U and W without nonzeros, ranges at both ends of the extents."""
    w = network_workload(400, 40, 10, 0.5, config_id=63)
    for name, m in (("U", 0), ("W", 1)):
        op = w.sparse[name]
        keep = (op.coords[m] % 5 != 2) & (op.coords[m] < 390)
        w.sparse[name] = gen.SparseOperand([np.ascontiguousarray(c[keep]) for c in op.coords], np.ascontiguousarray(op.vals[keep]), op.dims)
    out, _ = kernels_of(w)
    S, A = oracle(w)
    assert_close(out, S, A, np.float64)


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_values_no_nonzero_reads(value):
    """A row of V that no nonzero of U reads may hold anything, though it lies inside the ranges that are written out."""
    w = network_workload(400, 40, 10, 0.5, config_id=64)
    U = w.sparse["U"]
    keep = U.coords[1] != 150
    w.sparse["U"] = gen.SparseOperand([np.ascontiguousarray(c[keep]) for c in U.coords], np.ascontiguousarray(U.vals[keep]), U.dims)
    S, A = oracle(w)
    w.dense["V"][150] = value
    out, prof = kernels_of(w)
    assert "network_t" in prof
    assert_close(out, S, A, np.float64)
    assert not matrix_form_alone(w).any()


def test_more_rows_than_a_grid_has():
    """One l and eight k: a chunk of the intermediate holds 4 194 304 slices of U, 65 536 rows of blocks."""
    n = 4_194_300
    rng = np.random.default_rng(66)
    i = np.arange(n, dtype=np.int32)
    u = [i, i % 90, i % 8]
    k, m = (x.ravel().astype(np.int32) for x in np.mgrid[0:8, 0:8])
    uv, wv, V = rng.standard_normal(n), rng.standard_normal(64), rng.standard_normal((90, 1))
    plan = cb.const_plan_create("Z[i,m] = U[i,j,k] * V[j,l] * W[k,l,m]", ["T[i,k,l] = U[i,j,k] * V[j,l]", "Z[i,m] = T[i,k,l] * W[k,l,m]"],
                                {"U": (0, 2, 1), "W": (1, 2, 0)}, ["ikjl", "ilmk"], {"i": n, "j": 90, "k": 8, "l": 1, "m": 8}, cb.F64)
    U = cb.const_csf_build([to_dev(c) for c in u], to_dev(uv), (n, 90, 8), (0, 2, 1))
    W = cb.const_csf_build([to_dev(k), to_dev(0 * k), to_dev(m)], to_dev(wv), (8, 1, 8), (1, 2, 0))
    out = torch.full((n, 8), float("nan"), dtype=torch.float64, device="cuda")
    cb.const_execute(plan, {"U": U, "V": to_dev(V), "W": W}, out)
    assert cb.const_last_device_status(plan) == 0
    S = (uv * V[u[1], 0])[:, None] * wv.reshape(8, 8)[u[2]]
    assert np.all(np.abs(out.cpu().numpy() - S) <= 1e-12 * np.abs(S))


def test_without_memory_for_the_intermediate():
    """The gather form needs none."""
    w = network_workload(331, 61, 17, 0.25, config_id=61)
    cb.const_debug_set(3, 1)
    try:
        out, prof = kernels_of(w)
    finally:
        cb.const_debug_set(3, 0)
    assert "network_t" not in prof
    S, A = oracle(w)
    assert_close(out, S, A, np.float64)
