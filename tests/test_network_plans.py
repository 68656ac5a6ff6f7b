"""What a network keeps from its layer handles (step lists with their addresses, captured graphs) never outlives them: checked
on the CPU with stand-ins for the native calls that say which handles a pass would have used."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1805_07941_b200 import binding, workloads as wl
from paper_1805_07941_b200.network import QNetwork


class FakeConv:
    count = 0
    live = set()

    def __init__(self, *args, **kw):
        FakeConv.count += 1
        self.value = FakeConv.count
        FakeConv.live.add(self.value)
        self.handle = ctypes.c_void_p(self.value)

    def describe(self):
        return "igemm/box"

    def run(self, *args, **kw):
        assert self.handle, "a destroyed handle was run"

    def run_maxabs(self, *args, **kw):
        return np.float32(1.0)

    def destroy(self):
        FakeConv.live.discard(self.value)
        self.handle = ctypes.c_void_p()

    __del__ = destroy


class FakeSteps:
    last = None

    def __init__(self, steps):
        self.steps = steps

    def run(self, address):
        handles = [s["handle"].value for s in self.steps if "handle" in s]
        if None in handles:
            raise binding.QconvError(binding.ERR_BAD_ARG, "NULL handle")
        assert set(handles) <= FakeConv.live, "the pass holds a destroyed handle"
        FakeSteps.last = self


@pytest.fixture
def network(monkeypatch):
    monkeypatch.setattr(binding, "QConv", FakeConv)
    monkeypatch.setattr(binding, "Steps", FakeSteps)
    monkeypatch.setattr(binding, "qquantize_f32", lambda *a, **k: None)
    monkeypatch.setattr(binding, "qmaxpool_i8", lambda *a, **k: None)
    monkeypatch.setattr(binding, "qcalib_collect", lambda *a, **k: dict(maxabs=np.float32(1.0)))
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    binding.build_library()
    net = wl.resnet50(batch=3, res=32, width=16, blocks=(1, 1, 1, 1))
    weights = {nd["name"]: wl.gen_weights(nd, 0) for nd in net["nodes"] if nd["op"] == "conv"}
    return QNetwork(net, weights, device="cpu"), torch.zeros(net["input"])


def failing_after(calls, real):
    left = [calls]

    def call(*args, **kw):
        left[0] -= 1
        if left[0] < 0:
            raise binding.QconvError(binding.ERR_BAD_SHIFT, "stand-in")
        return real(*args, **kw)
    return call


@pytest.mark.parametrize("calls", [0, 3])
def test_a_calibration_that_raises_leaves_no_address_of_a_destroyed_handle(network, monkeypatch, calls):
    qn, x = network
    qn.calibrate(x)
    qn.run(x[:2])
    qn.run(x)
    qn.graph = object()                                      # (stands for a capture)
    with monkeypatch.context() as m:
        m.setattr(binding, "qrequant_shifts", failing_after(calls, binding.qrequant_shifts))
        with pytest.raises(binding.QconvError):
            qn.calibrate(x)
    assert qn.graph is None
    qn.run(x[:2])                                            # (old and new handles, all of them alive)
    qn.calibrate(x)
    qn.run(x[:2])


def test_a_calibration_that_raises_while_a_handle_is_replaced(network, monkeypatch):
    qn, x = network
    qn.calibrate(x)
    qn.run(x[:2])
    with monkeypatch.context() as m:
        m.setattr(qn, "_make_handle", failing_after(2, qn._make_handle))
        with pytest.raises(binding.QconvError):
            qn.calibrate(x)
    with pytest.raises(binding.QconvError) as e:             # the layer's old handle is gone, a new one was not made
        qn.run(x[:2])
    assert e.value.code == binding.ERR_BAD_ARG


def test_parameters_that_fail_to_load(network, monkeypatch):
    qn, x = network
    qn.calibrate(x)
    qn.run(x[:2])
    params, e_buf = dict(qn.params), dict(qn.e_buf)
    with monkeypatch.context() as m:
        m.setattr(qn, "_make_handle", failing_after(4, qn._make_handle))
        with pytest.raises(binding.QconvError):
            qn.load_params(params, e_buf)
    qn.run(x[:2])
    qn.load_params(params, e_buf).run(x[:2])


def test_handles_and_buffers_that_the_caller_replaces_are_the_ones_used(network):
    qn, x = network
    qn.calibrate(x)
    qn.run(x[:2])
    name = next(nd["name"] for nd in qn.net["nodes"] if nd["op"] == "conv")
    qn.handles[name] = FakeConv()
    qn.run(x[:2])
    assert qn.handles[name].value in [s["handle"].value for s in FakeSteps.last.steps if "handle" in s]
    qn.bufs[qn.last] = torch.zeros_like(qn.bufs[qn.last])
    qn.run(x[:2])
    assert FakeSteps.last.steps[-1]["d_y"] == qn.bufs[qn.last].data_ptr()
    kept = FakeSteps.last
    qn.run(x[:2])
    assert FakeSteps.last is kept                            # (an unchanged network's list is made once)
    qn.handles[name].destroy()
    with pytest.raises(binding.QconvError):
        qn.run(x[:2])


def test_destroyed_networks_keep_nothing(network):
    qn, x = network
    qn.calibrate(x)
    qn.run(x[:2])
    qn.graph = object()
    qn.destroy()
    assert qn.graph is None and not qn.handles
    with pytest.raises(KeyError):
        qn.run(x[:2])
