"""const_execute recorded into CUDA graphs and replayed, and the work lists of the tensor-core stage across streams."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2401_04836_b200 as cb
from workloads import network_workload, ttmc3_workload, ttmc4_workload
from tests.gpu_util import assert_close, build_csf, oracle, to_dev

pytestmark = pytest.mark.gpu


class Setup:
    def __init__(self, w, tensor_stage=False):
        self.w, self.dtype = w, cb.F32 if w.dtype == np.float32 else cb.F64
        self.plan = cb.const_plan_create(w.expression, w.tree, w.mode_orders, w.loop_orders, w.extents, self.dtype)
        if tensor_stage:
            cb.const_plan_set_tensor_stage(self.plan, True)
        self.handles = {n: build_csf(op, w.mode_orders[n]) for n, op in w.sparse.items()}
        self.dense = {n: to_dev(a) for n, a in w.dense.items()}
        self.out = torch.full(w.out_shape, float("nan"), dtype=torch.float32 if self.dtype == cb.F32 else torch.float64, device="cuda")

    def execute(self, handles=None, out=None):
        cb.const_execute(self.plan, {**(handles or self.handles), **self.dense}, self.out if out is None else out)

    def check(self):
        S, A = oracle(self.w)
        assert_close(self.out.cpu().numpy(), S, A, self.w.dtype)


def replay_twice(s, graph):
    for _ in range(2):
        s.out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        s.check()


def first_execute(s, stream, **kw):
    """The first execute of a plan, which sets its status word up, on the stream that will capture."""
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        s.execute(**kw)
    torch.cuda.synchronize()


def capture(s, stream):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.execute()
    return graph


@pytest.mark.parametrize("what", ["chain", "padded chain", "network, matrix form", "network, gather form", "generic executor"])
def test_execute_in_a_graph(what):
    """Clearing with an early start of the fused kernel, scratch for padded factors, the device-decided network."""
    if what == "chain":
        s = Setup(ttmc3_workload((120, 90, 80), 20_000, 8, slice_s=1.1, value="pm1", config_id=41))
    elif what.startswith("network"):
        s = Setup(network_workload(*((331, 61, 17) if "matrix" in what else (100, 20, 8)), 0.25, config_id=42))
    else:
        s = Setup(ttmc3_workload((120, 90, 80), 20_000, (10, 12), slice_s=1.1, value="pm1", config_id=43))
        if what == "generic executor":
            cb.const_plan_set_generic_executor(s.plan, True)
    stream = torch.cuda.Stream()
    first_execute(s, stream)
    s.check()
    graph = capture(s, stream)
    replay_twice(s, graph)
    if what.startswith("network, m"):                            # new values under the same graph
        s.dense["V"].mul_(0.5)
        s.w.dense["V"] = s.w.dense["V"] * 0.5
        replay_twice(s, graph)


def tensor_workload(order):
    if order == 4:
        return ttmc4_workload((300, 40, 30, 50), 80_000, 8, slice_s=1.0, value="pm1", config_id=3)
    return ttmc3_workload((500, 300, 700), 120_000, 16, slice_s=1.1, inner_s=0.9, value="unit", config_id=2)


@pytest.mark.parametrize("order", [3, 4])
def test_first_use_of_the_tensor_stage_inside_a_capture(order):
    s = Setup(tensor_workload(order), tensor_stage=True)
    other = Setup(tensor_workload(order), tensor_stage=True)
    other.plan = s.plan                                          # the plan has been used, the tensor has not
    stream = torch.cuda.Stream()
    first_execute(other, stream)
    graph = capture(s, stream)
    replay_twice(s, graph)
    assert cb.const_csf_bin_counts(s.handles["X"]) == cb.const_csf_bin_counts(other.handles["X"])
    s.execute()                                                  # and with lists of the handle's own now
    torch.cuda.synchronize()
    s.check()


def test_capture_behind_lists_that_another_stream_is_still_building():
    """The first use on one stream is not waited for: the graph has to."""
    s = Setup(tensor_workload(4), tensor_stage=True)
    warm = Setup(tensor_workload(4), tensor_stage=True)
    warm.plan = s.plan
    stream = torch.cuda.Stream()
    first_execute(warm, stream)
    side, scrap, graph = torch.cuda.Stream(), torch.empty_like(s.out), torch.cuda.CUDAGraph()
    s.out.fill_(float("nan"))
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)                           # about 0.2 s in front of the lists
        s.execute(out=scrap)
    with torch.cuda.stream(stream):                              # (torch.cuda.graph would wait for the device first)
        graph.capture_begin()
        s.execute()
        graph.capture_end()
        graph.replay()
    assert not side.query()                                      # the lists are still to come
    torch.cuda.synchronize()
    s.check()


def test_lists_outlive_the_stream_they_were_built_in():
    """A stream of the caller's own is where the lists are first needed; it is gone when they are asked for, used on another
    stream, and released."""
    rt = ctypes.CDLL("libcudart.so.12")
    for again in range(3):
        s = Setup(tensor_workload(4), tensor_stage=True)
        raw = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(raw), 1) == 0
        torch.cuda.synchronize()
        cb.const_execute(s.plan, {**s.handles, **s.dense}, s.out, stream=raw.value)
        assert rt.cudaStreamSynchronize(raw) == 0 and rt.cudaStreamDestroy(raw) == 0
        s.check()
        counts = cb.const_csf_bin_counts(s.handles["X"])
        assert counts["light"] + counts["heavy"] + counts["giant"] == np.unique(s.w.sparse["X"].coords[0]).size
        s.out.fill_(float("nan"))
        s.execute()
        torch.cuda.synchronize()
        s.check()
        for h in s.handles.values():
            cb.const_destroy(h)


def test_tensor_stage_on_a_second_stream_behind_lists_of_the_first():
    s, warm = Setup(tensor_workload(3), tensor_stage=True), Setup(tensor_workload(3), tensor_stage=True)
    warm.execute()                                               # (loading a kernel waits for the device)
    first, second, scrap = torch.cuda.Stream(), torch.cuda.Stream(), torch.empty_like(s.out)
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(400_000_000)
        s.execute(out=scrap)
    with torch.cuda.stream(second):
        s.execute()
    assert not first.query()
    second.synchronize()
    s.check()
