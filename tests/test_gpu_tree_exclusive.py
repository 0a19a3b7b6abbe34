"""Generic executor: updates of a shared workspace without atomics (fp64, a dense innermost range, enough updates per step of
the loop around it), and the same statement dealt out where an iteration has too few, against the oracle."""
import json
import os

import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from oracle import contract as oc
from workloads import generators as gen
from tests.gpu_util import assert_close, build_csf

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


@pytest.mark.parametrize("dtype,i,nnz_c,kernel", [
    (cb.F64, 64, 4000, "tree_step_kernel"),        # in step: 28 x 64 updates per value of q for 256 threads
    (cb.F64, 61, 4000, "tree_step_kernel"),        # rows made odd already, an extent that does not divide the group
    (cb.F64, 64, 200, "tree_step_kernel"),         # too few: dealt out, by the same kernel
    (cb.F64, 40, 4000, "tree_kernel"),             # workspaces that let more than four blocks run on an SM
    (cb.F32, 128, 4000, "tree_kernel"),            # fp32: always dealt out, padded rows
])
def test_running_example_with_large_workspaces(dtype, i, nnz_c, kernel):
    with open(os.path.join(GOLDEN, "running_example_schedule.json")) as f:
        g = json.load(f)
    rng = np.random.default_rng(i + nnz_c)
    ext = {"i": i, "j": 4, "k": 48, "p": 5, "q": 48, "r": 3}
    shape = {"A": "ipq", "B": "jpr", "C": "kqr", "D": "jkr"}
    nnz = {"A": 2500, "B": 40, "C": nnz_c, "D": 300}
    np_type = np.float32 if dtype == cb.F32 else np.float64
    sparse = {t: gen._uniform_tensor(tuple(ext[x] for x in idx), nnz[t], rng, "pm1", np_type) for t, idx in shape.items()}
    plan = cb.const_plan_create(g["expression"], g["tree"], g["mode_orders"], g["loop_orders"], ext, dtype)
    ops = {n: build_csf(op, g["mode_orders"][n]) for n, op in sparse.items()}
    out = torch.full((i, 4, 48), float("nan"), dtype=torch.float32 if dtype == cb.F32 else torch.float64, device="cuda")
    cb.const_profile_enable(True)
    cb.const_execute(plan, ops, out)
    prof = cb.const_profile_read()
    cb.const_profile_enable(False)
    assert [k for k in prof if k.startswith("tree")] == [kernel]
    assert cb.const_last_device_status(plan) == 0
    S, A = oc.nary_einsum(g["expression"], {t: (op.coords, op.vals) for t, op in sparse.items()}, ext)
    assert np.count_nonzero(A) > 0
    assert_close(out.cpu().numpy(), S, A, np_type)
