"""The gather form of the two-contraction network where its tiles (eight i by eight l) outnumber a 32-bit count."""
import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_l", [
    (40_003, 40_001),          # 25 million tiles
    (372_003, 372_001),        # 2.16e9, above 2^31
    (403, 600_001),            # 75 001 tiles of l, above the 65 535 rows of a grid
])
def test_tiles_beyond_a_grid(n, n_l):
    """Z_im = U_ijk V_jl W_klm with n slices of one nonzero and W nonzero in a few l only, the first and the last among
    them: tile numbers reach from 0 to n / 8 times n_l / 8."""
    rng = np.random.default_rng(n)
    i = np.arange(n)
    u = [i.astype(np.int32), (i % 2).astype(np.int32), (i // 2 % 3).astype(np.int32)]
    l = np.array([0, 7, 8, n_l // 2, n_l - 9, n_l - 1])
    w = [np.tile(np.arange(3), l.size).astype(np.int32), np.repeat(l, 3).astype(np.int32), (np.arange(3 * l.size) % 2).astype(np.int32)]
    uv, wv, V = rng.standard_normal(n), rng.standard_normal(w[0].size), rng.standard_normal((2, n_l))
    plan = cb.const_plan_create("Z[i,m] = U[i,j,k] * V[j,l] * W[k,l,m]", ["T[i,k,l] = U[i,j,k] * V[j,l]", "Z[i,m] = T[i,k,l] * W[k,l,m]"],
                                {"U": (0, 2, 1), "W": (1, 2, 0)}, ["ikjl", "ilmk"], {"i": n, "j": 2, "k": 3, "l": n_l, "m": 2}, cb.F64)
    assert cb.const_plan_family(plan) == "network"
    U = cb.const_csf_build([to_dev(c) for c in u], to_dev(uv), (n, 2, 3), (0, 2, 1))
    W = cb.const_csf_build([to_dev(c) for c in w], to_dev(wv), (3, n_l, 2), (1, 2, 0))
    out = torch.full((n, 2), float("nan"), dtype=torch.float64, device="cuda")
    cb.const_execute(plan, {"U": U, "V": to_dev(V), "W": W}, out)
    assert cb.const_last_device_status(plan) == 0
    S, A = np.zeros((n, 2)), np.zeros((n, 2))
    for k, at, m, v in zip(w[0], w[1], w[2], wv):
        term = np.where(u[2] == k, uv * V[u[1], at] * v, 0.0)
        S[:, m] += term
        A[:, m] += np.abs(term)
    assert np.all(np.abs(out.cpu().numpy() - S) <= 1e-12 * A)
