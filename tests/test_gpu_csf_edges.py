"""CSF compression at the edges of its tiles, against the CSF oracle."""
import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from oracle import csf as ocsf
from workloads import generators as gen
from tests.gpu_util import assert_csf_equal, build_csf, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz", [1, 2, 63, 64, 65, 255, 257, 2047, 2049, 4097])
def test_edges_of_the_compression_tiles(nnz):
    """Two keys per lane, 64 per step, 256 per warp, 2048 per block; every order; results that start at an odd address."""
    rng = np.random.default_rng(nnz)
    for dims in ((90, 80), (30, 20, 40), (9, 12, 8, 11)):
        op = gen._uniform_tensor(dims, min(nnz, int(np.prod(dims))), rng, "pm1", np.float32)
        order = tuple(reversed(range(len(dims))))
        h = build_csf(op, order)
        assert_csf_equal(h, op, order)
        n0 = cb.const_csf_level(h, 0)[1].numel()
        assert cb.const_csf_work_lists(h)[0].numel() == n0 + 1
        # the allocation-free build into arrays that are 4 bytes off any larger boundary
        n = op.nnz
        pos = [torch.empty(n + 2, dtype=torch.int32, device="cuda")[1:] for _ in dims]
        crd = [torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:] for _ in dims]
        vals = torch.empty(n, dtype=torch.float32, device="cuda")
        sizes = cb.const_csf_build_noalloc([to_dev(c.astype(np.int32)) for c in op.coords], to_dev(op.vals), dims, order, pos, crd, vals)
        opos, ocrd, ovals = ocsf.build(op.coords, op.vals, order)
        for l in range(len(dims)):
            np.testing.assert_array_equal(crd[l][: sizes[l]].cpu().numpy(), ocrd[l])
            np.testing.assert_array_equal(pos[l][: opos[l].size].cpu().numpy(), opos[l])
        assert vals.cpu().numpy().tobytes() == ovals.tobytes()
