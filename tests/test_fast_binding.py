"""The native checks of the forward calls: what they do not take goes through binding.py's own, which raise as ever."""
import sys

import numpy as np
import pytest
import torch

import paper_2110_09195_b200 as snn
import workloads as wl
from paper_2110_09195_b200 import binding


def test_anything_unusual_is_left_to_the_python_checks():
    """Where there is no GPU: CPU tensors, and arguments of other kinds, do no harm."""
    fast = binding._load_fast()
    x, y = torch.zeros((1, 4, 4, 1), dtype=torch.int32), torch.zeros((1, 4, 4, 16))
    desc = bytes(48)
    for args in ((desc, x, y, 0, 0), (desc[:40], x, y, 0, 0), (None, x, y, 0, 0), (desc, [x], y, 0, 0), (desc, x, y, 0),
                 (desc, x, y, 7, 0), (desc, x, y, 0.0, 0), (desc, x, y, 0, None)):
        assert fast.layer_forward(*args) == -1
    for args in ((desc, [x], [y], 0), (desc, (x,), [y], 0), (desc[:16], [], [], 0), (desc, [x, x], [y, y], 0)):
        assert fast.group_forward(*args) == -1
    assert fast.stack_forward(desc, x, y, 0) == -1 and fast.stack_forward(desc, x, y, None) == -1


class _Library:
    """Stands in for the C library where there is no GPU: notes the calls, and every one of them succeeds."""

    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append(name)
            if name.endswith("_create"):
                args[-1]._obj.value = 1   # the handle, passed by reference
            return 0
        return call


class _Layer(snn.SnnConv):
    def __del__(self):   # a handle of _Library must not reach the library, whenever it is collected
        pass


class _Group(snn.SnnConvGroup):
    __del__ = _Layer.__del__


@pytest.fixture
def without_module(monkeypatch):
    lib = _Library()
    monkeypatch.setattr(binding, "_lib", lib)
    monkeypatch.setattr(binding, "_fast", None)
    monkeypatch.setattr(binding, "_raw_stream", lambda device, stream: 0)
    monkeypatch.setitem(sys.modules, "paper_2110_09195_b200._snn_fast", None)   # importing it raises
    monkeypatch.delattr("paper_2110_09195_b200._snn_fast", raising=False)
    return lib


def test_a_layer_needs_neither_torch_nor_the_module(without_module, monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", None)   # importing it raises
    layer = _layer(wl.LayerShape(40, 72, 9, 7, 1, 1), cls=_Layer)
    assert without_module.calls == ["snn_conv_create"] and binding._fast is None
    layer.destroy()


def test_without_the_module_the_python_checks_make_the_calls(without_module):
    with pytest.warns(RuntimeWarning, match="checked in Python"):
        layer = _layer(wl.LayerShape(40, 72, 9, 7, 1, 1), device=-1, cls=_Layer)   # (where torch says that CPU tensors live)
    x, out = torch.zeros((2, 9, 7, 2), dtype=torch.int32), torch.zeros((2, 9, 7, 72))
    assert layer.forward(x, out=out) is out
    group = _Group([layer], [(2, 9, 7)])
    outs = [out]
    assert group.forward([x], outs) is outs
    assert without_module.calls == ["snn_conv_create", "snn_conv_forward", "snn_conv_group_create", "snn_conv_group_forward"]
    with pytest.raises(snn.SnnError):
        layer.forward(x, out=out[:1])
    with pytest.raises(snn.SnnError):
        group.forward([x[:1]], outs)
    group.destroy()
    layer.destroy()


def test_a_module_built_for_another_torch_is_not_used(monkeypatch):
    assert binding._load_fast().TORCH_VERSION == torch.__version__
    monkeypatch.setattr(binding, "_fast", None)
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    with pytest.warns(RuntimeWarning, match="not 0.0.1"):
        assert binding._load_fast().layer_forward(bytes(48), None, None, 0, 0) == -1
    assert binding._fast is binding._PythonChecks


def _layer(shape, seed=3, act_type=snn.ACT_BIN, device=0, cls=snn.SnnConv):
    p = wl.draw_layer_params(shape, 5, seed)
    return cls(shape.c_in, shape.c_out, 5, p.codebook, p.idx_packed, p.alpha, shape.stride, shape.pad, act_type, device)


@pytest.mark.gpu
@pytest.mark.parametrize("act_type", [snn.ACT_BIN, snn.ACT_F16])
def test_both_ways_launch_the_same(act_type):
    shape = wl.LayerShape(40, 72, 9, 7, 2, 1)
    layer, other = _layer(shape, 3, act_type), _layer(shape, 4, act_type)
    if act_type == snn.ACT_BIN:
        x = torch.from_numpy(wl.pack_activation_bits(wl.draw_activation_bits(shape, 3, 1)).view(np.int32)).cuda()
    else:
        x = torch.randn((3, 9, 7, 40), dtype=torch.float16, device="cuda")
    stream = torch.cuda.current_stream()
    for out_type in (snn.OUT_F32, snn.OUT_I32, snn.OUT_BITS) if act_type == snn.ACT_BIN else (snn.OUT_F32,):
        a, b = layer.alloc_out(3, 9, 7, out_type), layer.alloc_out(3, 9, 7, out_type)
        layer.forward(x, out=a, out_type=out_type)
        layer.forward(x, out=b, out_type=out_type, stream=stream)
        assert torch.equal(a, b)
        group = snn.SnnConvGroup([layer, other], [(3, 9, 7)] * 2)
        outs, want = group.alloc_outs(out_type), group.alloc_outs(out_type)
        group.forward([x, x], outs, out_type=out_type)
        group.forward((x, x), tuple(want), out_type=out_type)   # (not lists: the Python checks)
        assert all(torch.equal(p, q) for p, q in zip(outs, want)) and torch.equal(outs[0], a)


@pytest.mark.gpu
def test_the_usual_call_is_taken_and_any_other_left():
    """The native checks make a valid call themselves; with one argument changed they launch nothing and leave it."""
    fast = binding._load_fast()
    layer = _layer(wl.LayerShape(40, 72, 9, 7, 2, 1))
    group, stack = snn.SnnConvGroup([layer, layer], [(3, 9, 7)] * 2), snn.SnnConvStack([layer], 3, 9, 7)
    x, y = torch.zeros((3, 9, 7, 2), dtype=torch.int32, device="cuda"), layer.alloc_out(3, 9, 7)
    bits, sums = layer.alloc_out(3, 9, 7, snn.OUT_BITS), layer.alloc_out(3, 9, 7, snn.OUT_I32)
    base = (layer._desc, x, y, snn.OUT_F32, snn.PATH_AUTO)
    no_x = [x.cpu(), x.float(), x[:2], x[..., :1].contiguous(), x.transpose(1, 2), x[0], x.to_sparse(), None, [x]]
    no_y = [y.cpu(), sums, y[:2], y[..., :71].contiguous(), y.transpose(1, 2), bits, None, [y]]

    class Tensor(torch.Tensor):
        pass
    no_x.append(x.as_subclass(Tensor))

    def launches(call, *args):
        before = snn.kernel_launches()
        return call(*args), snn.kernel_launches() - before

    for good in (base, (layer._desc, x.view(torch.uint32), *base[2:]), (layer._desc, x, bits, snn.OUT_BITS, 0),
                 (layer._desc, x, sums, snn.OUT_I32, 0), (layer._desc, torch.nn.Parameter(x, requires_grad=False), *base[2:])):
        st, n = launches(fast.layer_forward, *good)
        assert st == 0 and n >= 1
    for i, values in enumerate(([layer._desc[:40], None, bytearray(layer._desc)], no_x, no_y, [snn.OUT_I32, snn.OUT_BITS, 7, -1, 0.0, True, None],
                                [7, -1, None])):
        for v in values:
            assert launches(fast.layer_forward, *base[:i], v, *base[i + 1:]) == (-1, 0), (i, v)

    base = (group._desc, [x, x], [y, y.clone()], snn.OUT_F32)
    assert launches(fast.group_forward, *base) == (0, 1)
    for i, values in enumerate(([group._desc[:-8], group._desc[:47], None], [[x], (x, x), [x, x, x], *([x, v] for v in no_x), *([v, x] for v in no_x)],
                                [[y], (y, y), *([y, v] for v in no_y)], [snn.OUT_I32, 7, None])):
        for v in values:
            assert launches(fast.group_forward, *base[:i], v, *base[i + 1:]) == (-1, 0), (i, v)

    base = (stack._desc, x, y, snn.OUT_F32)
    assert launches(fast.stack_forward, *base) == (0, 1)
    for i, values in enumerate(([stack._desc[:47], None], no_x, no_y, [snn.OUT_I32, 7, None])):
        for v in values:
            assert launches(fast.stack_forward, *base[:i], v, *base[i + 1:]) == (-1, 0), (i, v)
    torch.cuda.synchronize()


@pytest.mark.gpu
def test_wrong_tensors_are_refused():
    shape = wl.LayerShape(40, 72, 9, 7, 1, 1)
    layer = _layer(shape)
    x = torch.zeros((2, 9, 7, 2), dtype=torch.int32, device="cuda")
    out = layer.alloc_out(2, 9, 7)
    wide = torch.zeros((2, 9, 7, 144), device="cuda")
    for act, o in ((x.cpu(), out), (x.float(), out), (x[..., :1], out), (x.transpose(1, 2), out), (x, out.cpu()), (x, out.int()),
                   (x, out[:1]), (x, wide[..., ::2]), (x[0], out)):
        with pytest.raises(snn.SnnError):
            layer.forward(act, out=o)
        with pytest.raises(snn.SnnError):
            snn.SnnConvGroup([layer], [(2, 9, 7)]).forward([act], [o])
    with pytest.raises(snn.SnnError):
        layer.forward(x, out=out, out_type=9)
    shifted = torch.zeros(x.numel() + 1, dtype=torch.int32, device="cuda")[1:].view(x.shape)   # 4 bytes past a boundary of 16
    with pytest.raises(snn.SnnError):
        layer.forward(shifted, out=out)
    assert layer.forward(x[:0], out=out[:0]).numel() == 0
    layer.destroy()
    with pytest.raises(snn.SnnError):
        layer.forward(x, out=out)


@pytest.mark.gpu
def test_the_current_stream_is_used():
    shape = wl.LayerShape(32, 32, 32, 32, 1, 1)
    layer = _layer(shape)
    x = torch.zeros((4, 32, 32, 1), dtype=torch.int32, device="cuda")
    out = layer.alloc_out(4, 32, 32)
    layer.forward(x, out=out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):      # a launch on any other stream would break the capture
        layer.forward(x, out=out)
    want = out.clone()
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def _static_arguments(c_in=40, c_out=24, n=2, h=9, w=7, tau=4, seed=5, device="cuda"):
    shape = wl.LayerShape(c_in, c_out, h, w, 1, 1)
    p = wl.draw_layer_params(shape, tau, seed)
    x = torch.from_numpy(wl.pack_activation_bits(wl.draw_activation_bits(shape, n, seed)).view(np.int32)).to(device)
    return [c_in, c_out, tau, np.asarray(p.codebook, np.uint16), np.asarray(p.idx_packed, np.uint8), np.asarray(p.alpha, np.float32), x,
            torch.empty((n, h, w, c_out), dtype=torch.float32, device=device), 1, 1, snn.OUT_F32, 0]


def _with(args, i, v):
    return [*args[:i], v, *args[i + 1:]]


# arguments the library would read wrongly, each in the place of a good one
_NOT_PLAIN = [(0, 40.0), (0, 513), (1, 25), (2, 5), (2, True), (3, [1] * 16), (3, np.zeros(16, np.int16)), (3, np.zeros(32, np.uint16)[::2]),
              (3, np.zeros(15, np.uint16)), (4, bytes(480)), (4, np.zeros(479, np.uint8)), (5, np.zeros(24)), (5, np.zeros(24, ">f4")), (5, torch.zeros(24)),
              (6, None), (7, None), (8, 3), (9, 2), (10, 2), (11, -1), (11, 1)]


def test_the_arrays_of_the_no_allocation_call_are_numpys_own():
    fast = binding._load_fast()
    args = _static_arguments(device="cpu")
    assert fast.static_forward(*args) == -1 and fast.static_forward(*args[:-1]) == -1
    for i, v in _NOT_PLAIN:
        assert fast.static_forward(*_with(args, i, v)) == -1


@pytest.mark.gpu
def test_the_no_allocation_call_both_ways():
    args = _static_arguments()
    fast = binding._load_fast()
    first = snn.forward_static(*args).clone()
    lists = _with(_with(_with(args, 3, args[3].tolist()), 5, args[5].astype(np.float64)), 7, torch.zeros_like(first))   # converted in Python
    assert fast.static_forward(*lists) == -1 and torch.equal(snn.forward_static(*lists), first)
    layer = snn.SnnConv(*args[:6])
    assert torch.equal(layer.forward(args[6]), first)
    for i, v in _NOT_PLAIN:
        assert fast.static_forward(*_with(args, i, v)) == -1
    for i, v in ((1, 25), (2, 5), (3, args[3][:-1]), (4, args[4][:-1]), (7, first[:1]), (8, 3)):
        with pytest.raises(snn.SnnError):
            snn.forward_static(*_with(args, i, v))
    with pytest.raises(snn.SnnError):   # refused by the library: said as ever
        snn.forward_static(*_with(args, 5, np.full(24, np.nan, np.float32)))
    layer.destroy()
