"""The CSF builder's splitter sort against the CSF oracle and against its radix sort, array for array."""
import itertools

import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from workloads import generators as gen
from tests.gpu_util import assert_csf_equal, build_csf, csf_to_host, to_dev

pytestmark = pytest.mark.gpu

RADIX, SPLIT = 1, 2


@pytest.fixture(autouse=True)
def default_path():
    yield
    for what in range(5):
        cb.const_debug_set(what, 0)


def built(op, order, path):
    cb.const_debug_set(4, path)
    h = build_csf(op, order)
    return (*csf_to_host(h), cb.const_csf_work_lists(h)[0].cpu().numpy())


def assert_same(op, order):
    a, b = built(op, order, RADIX), built(op, order, SPLIT)
    for x, y in zip(a[0] + a[1] + [a[3]], b[0] + b[1] + [b[3]]):
        np.testing.assert_array_equal(x, y)
    assert a[2].tobytes() == b[2].tobytes()


def operand(key, dims, dtype=np.float32, shuffle=True):
    rng = np.random.default_rng(key.size)
    key = rng.permutation(key) if shuffle else key
    coords = []
    for d in reversed(dims):
        coords.append((key % d).astype(np.int32))
        key = key // d
    return gen.SparseOperand(coords[::-1], rng.standard_normal(coords[0].size).astype(dtype), dims)


# one part, the edges of a tile (2048) and of a chunk (4096), several parts and buckets; every order, key widths up to 64 bits
@pytest.mark.parametrize("nnz", [1, 2, 1365, 1366, 2048, 2049, 4095, 4097, 30_011, 200_003])
def test_against_the_oracle(nnz):
    rng = np.random.default_rng(nnz)
    for dims, dtype in (((1700, 900), np.float32), ((90, 80, 170), np.float64), ((65536, 65536, 65536, 65536), np.float32)):
        op = gen._uniform_tensor(dims, nnz, rng, "pm1", dtype)
        for order in (tuple(range(len(dims))), tuple(reversed(range(len(dims))))):
            cb.const_debug_set(4, SPLIT)
            assert_csf_equal(build_csf(op, order), op, order)


@pytest.mark.parametrize("dims,nnz", [((1, 1, 900_000), 400_000), ((900_000, 1, 1), 400_000), ((3, 700, 701), 1_300_000),
                                      ((5003, 3001, 4001), 1_300_001), ((2003, 1501, 701, 301), 500_003)])
def test_every_mode_order_against_the_radix_sort(dims, nnz):
    rng = np.random.default_rng(nnz)
    cells = int(np.prod(dims, dtype=np.int64))
    key = rng.permutation(cells)[:nnz] if cells < 4 * nnz else np.unique(rng.integers(0, cells, nnz))
    op = operand(key, dims, np.float64 if len(dims) == 4 else np.float32)
    for order in itertools.islice(itertools.permutations(range(len(dims))), 0, None, 5 if len(dims) == 4 else 2):
        assert_same(op, order)


def test_scan_over_many_blocks():
    """Above 4096 blocks of the count kernel (8.4 M nonzeros) the radix path scans them with kernels of their own."""
    dims = (3001, 2503, 4007)
    key = np.unique(np.random.default_rng(9).integers(0, int(np.prod(dims, dtype=np.int64)), 9_000_000))
    assert key.size > 4096 * 2048
    assert_same(operand(key, dims), (1, 0, 2))


@pytest.mark.parametrize("what", ["sorted", "reversed", "banded", "clusters", "one slice"])
def test_distributions(what):
    """Sorted input (all lanes one way), keys crowded into a part of their range (bins of bins, then the network), a giant slice."""
    rng = np.random.default_rng(7)
    dims = (65536, 65536, 65536)
    if what in ("sorted", "reversed"):
        key = np.sort(np.unique(rng.integers(0, 2 ** 48, 600_000)))[:: 1 if what == "sorted" else -1]
    elif what == "banded":
        i = np.repeat(np.arange(20_000, dtype=np.int64), 30)
        j = i + np.tile(np.arange(30), 20_000)
        key = np.unique((i * 65536 + j) * 65536 + (7 * i + j) % 65536)
    elif what == "clusters":
        key = np.unique(np.exp2(rng.random(700_000) * 47.9).astype(np.int64))
    else:
        key = (41 << 32) + rng.permutation(2 ** 24)[:600_000].astype(np.int64)
    op = operand(key, dims, shuffle=what not in ("sorted", "reversed"))
    assert_same(op, (0, 1, 2))
    assert_same(op, (2, 0, 1))


@pytest.mark.parametrize("tail", [3, 200, 500, 1300])
@pytest.mark.parametrize("dims", [(2, 1 << 21, 1 << 21, 1 << 21), (4, 1 << 21, 1 << 21, 1 << 20), (1 << 16,) * 4])
def test_largest_key_of_64_bits(dims, tail):
    """The last corner of extents that fill 64 bits, in a part that begins in the first slice: its number is the largest there is."""
    rng = np.random.default_rng(tail)
    nnz = 300_000
    for shrink in (0, 4, 8) * 2:                           # the tail, in the last slice, is spread over it or lies close to the corner
        coords = [rng.integers(0, d, nnz).astype(np.int32) for d in dims]
        coords[0][:] = 0
        near = [d >> shrink for d in dims[2:]]
        inside = rng.permutation(np.unique(rng.integers(0, near[0] * near[1], 2 * tail)))[:tail]
        inside[0] = 0
        for c, d, back in zip(coords, dims, (0, 0, inside // near[1], inside % near[1])):
            c[:tail] = d - 1 - back
        perm = rng.permutation(nnz)
        op = gen.SparseOperand([c[perm] for c in coords], rng.standard_normal(nnz).astype(np.float32), dims)
        assert_same(op, (0, 1, 2, 3))


def test_errors_and_the_way_back_to_the_radix_sort():
    rng = np.random.default_rng(3)
    op = gen._uniform_tensor((300, 1000, 777), 500_003, rng, "pm1", np.float32)
    cb.const_debug_set(4, SPLIT)

    def status(coords):
        with pytest.raises(cb.ConstError) as e:
            cb.const_csf_build([to_dev(c) for c in coords], to_dev(op.vals), op.dims, (0, 1, 2))
        return e.value.status

    twice = [c.copy() for c in op.coords]
    for c in twice:
        c[400_000] = c[5]
    assert status(twice) == 4
    assert status([np.zeros_like(c) for c in op.coords]) == 4        # one part outgrows its room: sorted again by digits
    for bad in (-1, 1000, 2 ** 31 - 1):
        far = [c.copy() for c in op.coords]
        far[1][123_456] = bad
        assert status(far) == 5
    cb.const_debug_set(3, 1)                                         # no memory for it
    cb.const_profile_enable(True)
    h = build_csf(op, (0, 1, 2))
    names = cb.const_profile_read()
    cb.const_profile_enable(False)
    assert "rs_onesweep" in names and "part_sort" not in names
    assert_csf_equal(h, op, (0, 1, 2))


@pytest.mark.parametrize("path", [3, 4])
def test_the_radix_sort_runs_behind_the_splitters(path):
    """A valid tensor whose build gives up (3), or finds no memory for the upper levels beside its arena (4), when the values and leaf
    coordinates have been written already."""
    rng = np.random.default_rng(5)
    for dims, dtype in (((300, 1000, 777), np.float32), ((70, 80, 90, 100), np.float64), ((5003, 3001), np.float32)):
        op = gen._uniform_tensor(dims, 300_007, rng, "pm1", dtype)
        cb.const_debug_set(4, path)
        cb.const_profile_enable(True)
        h = build_csf(op, tuple(range(len(dims))))
        names = cb.const_profile_read()
        cb.const_profile_enable(False)
        assert "part_sort" in names and "rs_onesweep" in names and "part_nodes" not in names
        assert_csf_equal(h, op, tuple(range(len(dims))))
    with pytest.raises(cb.ConstError):
        cb.const_debug_set(4, 5)


def test_chunk_wait_times_out_and_recovers():
    rng = np.random.default_rng(4)
    op = gen._uniform_tensor((300, 1000, 777), 300_007, rng, "pm1", np.float32)
    cb.const_debug_set(4, SPLIT)
    cb.const_debug_set(0, 200)
    cb.const_debug_set(1, 1)
    with pytest.raises(cb.ConstError) as e:
        build_csf(op, (0, 1, 2))
    assert e.value.status == 8
    cb.const_debug_set(1, 0)
    cb.const_debug_set(0, 0)
    assert_csf_equal(build_csf(op, (0, 1, 2)), op, (0, 1, 2))


@pytest.mark.parametrize("nnz", [1366, 2048, 4097])
def test_chunks_that_nobody_waits_for(nnz):
    """One coordinate throughout: one bucket of several parts, which up to a tile no other tile appends to.  Its chunk is not published, so
    it cannot be sampled; published, the coordinate occurs twice."""
    op = operand(np.full(nnz, 123_456_789), (300, 1000, 777))
    for withhold, status in ((1, 8), (0, 4)):
        cb.const_debug_set(4, SPLIT)
        cb.const_debug_set(0, 200)
        cb.const_debug_set(1, withhold)
        with pytest.raises(cb.ConstError) as e:
            build_csf(op, (0, 1, 2))
        assert e.value.status == status


@pytest.mark.parametrize("nnz", [1, 500, 2048])
def test_parts_are_sorted_without_the_early_word(nnz):
    """Signals withheld where nothing has to wait for a chunk: the blocks that sort parts are not told that they may start, and wait."""
    op = operand(np.arange(nnz, dtype=np.int64) * 99_991, (300, 1000, 777))
    cb.const_debug_set(4, SPLIT)
    cb.const_debug_set(1, 1)
    assert_csf_equal(build_csf(op, (0, 1, 2)), op, (0, 1, 2))
    assert_csf_equal(build_csf(op, (2, 0, 1)), op, (2, 0, 1))


def test_which_sort_runs():
    """The line: 200 000 nonzeros, and 700 000 nonzeros times radix passes beyond two."""
    for dims, nnz, split in (((2000, 3000, 4000), 340_000, False), ((2000, 3000, 4000), 360_000, True), ((512, 512, 512), 690_000, False),
                             ((512, 512, 512), 710_000, True), ((20000, 20000, 20000, 20000), 190_000, False),
                             ((20000, 20000, 20000, 20000), 210_000, True)):
        coords = [torch.randint(0, d, (nnz,), device="cuda", dtype=torch.int32) for d in dims]
        cb.const_profile_enable(True)
        try:
            cb.const_csf_build(coords, torch.ones(nnz, device="cuda"), dims, tuple(range(len(dims))))
        except cb.ConstError as e:                                   # drawn with repetition: some occur twice
            assert e.status == 4
        names = cb.const_profile_read()
        cb.const_profile_enable(False)
        assert ("part_sort" in names) == split and ("rs_onesweep" in names) != split


@pytest.mark.parametrize("nnz", [1023, 1025, 50_000, 199_999, 200_001, 410_001, 900_001])
def test_tile_sizes_of_the_radix_sort(nnz):
    """Tiles of 1024, 2048 and 4096 keys, whose passes start before the one before has ended."""
    rng = np.random.default_rng(nnz)
    for dims, dtype in (((331, 331, 64), np.float64), ((1201, 993, 1503), np.float32)):
        op = gen._uniform_tensor(dims, nnz, rng, "pm1", dtype)
        for order in ((0, 1, 2), (2, 0, 1)):
            cb.const_debug_set(4, RADIX)
            for _ in range(3):
                h = build_csf(op, order)
            assert_csf_equal(h, op, order)
