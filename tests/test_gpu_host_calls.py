"""The native part of the binding takes the plain case of a call and leaves every other one to the general
path: the same results with and without given outputs, on given streams, for subclasses and wrapped tensors,
the same errors as ever, and the straight-through estimator inside autograd."""
from __future__ import annotations

import ctypes
import subprocess
import threading

import numpy as np
import pytest
import torch
import torch.autograd.forward_ad as fwad
from torch.overrides import TorchFunctionMode
from torch.utils._python_dispatch import TorchDispatchMode

import paper_2604_00529_b200 as mxq
from paper_2604_00529_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture
def general(monkeypatch):
    """Runs a call through the general path alone."""
    class Off:
        def __getattr__(self, name):
            return (lambda *a: 1) if name == "run_prepared" else (lambda *a: None)

    def run(fn):
        host = binding._host
        binding._host = Off()
        try:
            return fn()
        finally:
            binding._host = host
    mxq.load_library()
    return run


def same(a, b):
    if isinstance(a, torch.Tensor):
        return a.dtype == b.dtype and a.shape == b.shape and a.device == b.device and torch.equal(
            a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))
    return type(a) is type(b) and len(a) == len(b) and all(same(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("shape", [(1, 32), (7, 96), (130, 256)])
def test_native_calls_equal_the_general_path(general, dtype, shape):
    x = torch.randn(*shape, device="cuda").to(dtype)
    n = x.numel()
    codes, scales = mxq.quantize(x, "e4m3")
    dst = torch.empty(n, dtype=dtype, device="cuda")
    calls = [
        lambda: mxq.quantize(x, "int6"),
        lambda: mxq.quantize(torch.nn.Parameter(x), "e2m1", 32),
        lambda: mxq.quantize(x, "e4m3", codes=torch.empty_like(codes), scales=torch.empty_like(scales)),
        lambda: mxq.slice_scale(codes, scales, n, "e4m3", "e2m3"),
        lambda: mxq.slice_scale_multi(codes, scales, n, "e4m3", ["e2m3", "e2m1", "e3m3"]),
        lambda: mxq.slice_scale_multi(codes, scales, n, "e4m3", []),
        lambda: mxq.dequantize(codes, scales, n, "e4m3", dtype=dtype),
        lambda: mxq.dequantize(codes, scales, n, "e4m3"),
        lambda: mxq.dequantize(codes, scales, n, "e4m3", dst=dst),
        lambda: mxq.quantize_tiled(x, "e3m2"),
        lambda: mxq.slice_scale_tiled(codes, scales, *shape, "e4m3", "e2m1"),
        lambda: mxq.fake_quant(x, "int4", 16, mxq.FQ_VIA_ANCHOR),
        lambda: mxq.fake_quant_bwd(x),
        lambda: mxq.fake_quant(x, "int4", stream=torch.cuda.Stream()) if torch.cuda.synchronize() is None else None,
    ]
    for call in calls:
        got = call()
        torch.cuda.synchronize()
        want = general(call)
        torch.cuda.synchronize()
        assert same(got, want)
    low, low_scales = torch.empty(n // 2, dtype=torch.uint8, device="cuda"), torch.empty_like(scales)
    p = mxq.prepare_slice_scale(codes, scales, n, "e4m3", "e2m1", 32, low, low_scales)
    p()
    assert same((low, low_scales), general(lambda: mxq.slice_scale(codes, scales, n, "e4m3", "e2m1")))


def test_refused_calls_stay_refused():
    x = torch.randn(64, 64, device="cuda")
    codes, scales = mxq.quantize(x, "int8")
    n = x.numel()
    for error, call in [
        (ValueError, lambda: mxq.quantize(x.t(), "int8")),
        (ValueError, lambda: mxq.quantize(x.cpu(), "int8")),
        (TypeError, lambda: mxq.quantize(x.half(), "int8")),
        (KeyError, lambda: mxq.quantize(x, "int9")),
        (mxq.MxqError, lambda: mxq.quantize(x.view(-1)[:40], "int8")),
        (mxq.MxqError, lambda: mxq.quantize(x.view(-1)[1:33], "int8")),
        (mxq.MxqError, lambda: mxq.quantize(x, "int8", 48)),
        (mxq.MxqError, lambda: mxq.quantize(x, "int8", 0)),
        (mxq.MxqError, lambda: mxq.slice_scale(codes, scales, n, "int8", "e2m1")),
        (mxq.MxqError, lambda: mxq.slice_scale_multi(codes, scales, n, "int8", ["int4", "e2m1"])),
        (ValueError, lambda: mxq.dequantize(codes, scales.cpu(), n, "int8")),
        (TypeError, lambda: mxq.dequantize(codes, scales, n, "int8", dtype=torch.float16)),
        (ValueError, lambda: mxq.quantize_tiled(x.view(-1), "e4m3")),
        (mxq.MxqError, lambda: mxq.quantize_tiled(x, "int8")),
        (mxq.MxqError, lambda: mxq.fake_quant(x, "int4", 32, 7)),
        (ValueError, lambda: mxq.fake_quant_ste(x.t().requires_grad_(), "int4")),
        (RuntimeError, lambda: torch.func.vmap(lambda t: mxq.fake_quant(t, "int4"))(x)),
        (RuntimeError, lambda: torch.func.vmap(lambda t: t * mxq.fake_quant_ste(x, "int4").sum())(x)),
        (RuntimeError, lambda: torch.func.grad(lambda t: mxq.fake_quant_ste(t, "int4").sum())(x)),
    ]:
        with pytest.raises(error):
            call()


@pytest.mark.parametrize("copy_grad", [False, True])
def test_straight_through_gradient(general, copy_grad):
    x = torch.randn(8, 64, device="cuda").requires_grad_()
    g = torch.randn(8, 64, device="cuda")

    def step():
        y = mxq.fake_quant_ste(x * 2, "e2m1", 32, mxq.FQ_VIA_ANCHOR, copy_grad)
        return (y.detach(), *torch.autograd.grad(y * 3, x, g, retain_graph=True))

    assert same(step(), general(step))
    node = mxq.fake_quant_ste(x * 2, "e2m1", copy_grad=copy_grad).grad_fn
    assert "CppFunction" in type(node).__name__ and "Mul" in type(node.next_functions[0][0]).__name__
    with torch.no_grad():
        assert not mxq.fake_quant_ste(x, "e2m1").requires_grad
    assert not mxq.fake_quant_ste(x.detach(), "e2m1").requires_grad
    (first,) = torch.autograd.grad(mxq.fake_quant_ste(x, "e2m1", copy_grad=copy_grad).pow(3).sum(), x, create_graph=True)
    assert first.requires_grad != copy_grad                     # the copied gradient is a constant, as through the general path


@pytest.mark.parametrize("copy_grad", [False, True])
def test_hooks_batched_gradients_and_forward_mode(general, copy_grad):
    x = torch.randn(8, 64, device="cuda").requires_grad_()

    def ste(t):
        return mxq.fake_quant_ste(t, "int4", 32, mxq.FQ_VIA_ANCHOR, copy_grad)

    def hooked():
        leaf, seen = x.detach().clone().requires_grad_(), []
        y = ste(leaf * 2)
        y.retain_grad()
        y.register_hook(lambda g: seen.append(g) or g * 2)
        y.grad_fn.register_prehook(lambda go: (go[0] * 3,))
        y.grad_fn.register_hook(lambda gi, go: seen.append(gi[0]) or seen.append(go[0]))
        y.pow(2).sum().backward()
        return (leaf.grad, y.grad, *seen)

    def strided():
        return torch.autograd.grad(ste(x * 2), x, torch.arange(512.0, device="cuda").view(64, 8).t())

    for step in (hooked, strided):
        assert same(step(), general(step))
    grads = torch.randn(3, 8, 64, device="cuda")

    def batched():
        return torch.autograd.grad(ste(x), x, grads, is_grads_batched=True)

    if copy_grad:                                               # a copy needs memory of its own: refused as ever
        for run in (lambda fn: fn(), general):
            with pytest.raises(RuntimeError, match="storage"):
                run(batched)
    else:
        assert same(batched(), (grads,)) and same(general(batched), (grads,))
    with fwad.dual_level(), pytest.raises(NotImplementedError):
        ste(fwad.make_dual(x.detach(), torch.ones_like(x)))


def test_a_refused_backward_raises_the_library_s_error(general):
    x = torch.randn(8, 64, device="cuda").requires_grad_()
    g = torch.randn(513, device="cuda")[1:].view(8, 64)                # contiguous, not 32-byte aligned

    def step():
        with pytest.raises(mxq.MxqError) as e:
            torch.autograd.grad(mxq.fake_quant_ste(x, "int4", copy_grad=True), x, g)
        return (e.value.status, str(e.value))

    status, text = step()
    assert (status, text) == general(step) and "MXQ_ERR_ALIGN" in text


def per_tensor_calls():
    """One plain call of every native function, all outputs left to it; nothing but arguments is prepared."""
    x = torch.randn(64, 128, device="cuda")
    codes, scales = mxq.quantize(x, "e4m3")
    n, leaf = x.numel(), torch.randn(8, 64, device="cuda").requires_grad_()
    h = binding._host
    return {
        "quantize": lambda: h.quantize(x, "int6", 32, None, None, None),
        "slice_scale": lambda: h.slice_scale(codes, scales, n, "e4m3", "e2m3", 32, None, None, None),
        "slice_scale_multi": lambda: h.slice_scale_multi(codes, scales, n, "e4m3", ["e2m3", "e2m1"], 32, None, None),
        "dequantize": lambda: h.dequantize(codes, scales, n, "e4m3", 32, torch.float32, None, None),
        "quantize_tiled": lambda: h.quantize_tiled(x, "e4m3", 32, None, None, None),
        "slice_scale_tiled": lambda: h.slice_scale_tiled(codes, scales, 64, 128, "e4m3", "e2m1", 32, None, None, None),
        "fake_quant": lambda: h.fake_quant(x, "int4", 32, mxq.FQ_VIA_ANCHOR, None, None),
        "fake_quant_bwd": lambda: h.fake_quant_bwd(x, None, None),
        "fake_quant_ste": lambda: h.fake_quant_ste(leaf, "int4", 32, mxq.FQ_VIA_ANCHOR, False),
    }


class Sub(torch.Tensor):
    pass


class FunctionMode(TorchFunctionMode):
    def __torch_function__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


class DispatchMode(TorchDispatchMode):
    def __torch_dispatch__(self, func, types, args=(), kwargs=None):
        return func(*args, **(kwargs or {}))


def test_the_plain_case_is_handled_natively_and_nothing_else():
    calls = per_tensor_calls()
    for name, call in calls.items():
        assert call() is not None, name
        with FunctionMode():
            assert call() is None, name
        with DispatchMode():
            assert call() is None, name
    h, x = binding._host, torch.randn(64, 128, device="cuda")
    codes, scales = h.quantize(x, "e4m3", 32, None, None, None)
    n, stream = x.numel(), torch.cuda.current_stream()
    out = torch.empty_like(codes)
    assert h.quantize(x, "e4m3", 32, out, scales, None)[0] is out
    for given in (out.cpu(), out.view(2, -1).t(), out.as_subclass(Sub)):
        assert h.quantize(x, "e4m3", 32, given, None, None) is None
    for src in (x.as_subclass(Sub), x.t(), x.cpu(), x.half(), x.to_sparse(), x.to("meta"), None):
        assert h.quantize(src, "e4m3", 32, None, None, None) is None
        assert h.fake_quant(src, "int4", 32, 0, None, None) is None
        assert h.fake_quant_ste(src, "int4", 32, 0, False) is None
    assert h.quantize(x, "e4m3", 32, None, None, stream) is None
    assert h.slice_scale(codes, scales, n, "e4m3", "e2m1", 32, None, None, stream) is None
    assert h.slice_scale(codes, scales, float(n), "e4m3", "e2m1", 32, None, None, None) is None
    assert h.slice_scale_multi(codes, scales, n, "e4m3", iter(["e2m1"]), 32, None, None) is None
    assert h.dequantize(codes, scales, n, "e4m3", 32, torch.float16, None, None) is None
    assert h.fake_quant(x, "int4", True, 0, None, None) is None
    with fwad.dual_level():
        assert h.fake_quant_ste(fwad.make_dual(x.clone(), torch.ones_like(x)), "int4", 32, 0, False) is None
    seen = []
    torch.jit.trace(lambda t: seen.append(h.fake_quant_ste(t * 2, "int4", 32, 0, False)) or t * 2, (x,), check_trace=False)
    torch.func.vmap(lambda t: seen.append(h.fake_quant_ste(x, "int4", 32, 0, False)) or t)(x)
    torch.func.grad(lambda t: (seen.append(h.fake_quant(t, "int4", 32, 0, None, None)), t.sum())[1])(x)
    assert seen == [None, None, None]


def test_subclasses_modes_and_threads_get_the_results_of_the_general_path(general):
    x = torch.randn(64, 128, device="cuda")
    sub = x.as_subclass(Sub)
    want = general(lambda: (*mxq.quantize(x, "int6"), mxq.fake_quant(x, "int4"), mxq.fake_quant_ste(x, "int4")))

    def all_of(t):
        return (*mxq.quantize(t, "int6"), mxq.fake_quant(t, "int4"), mxq.fake_quant_ste(t, "int4"))

    assert all(type(a) is type(b) for a, b in zip(all_of(sub), general(lambda: all_of(sub))))
    got = [tuple(t.as_subclass(torch.Tensor) for t in all_of(sub))]
    for mode in (FunctionMode, DispatchMode, torch.inference_mode, torch.no_grad):
        with mode():
            got.append(all_of(x))
    stream = torch.cuda.current_stream()

    def worker():
        with torch.cuda.stream(stream):
            got.append(all_of(x))

    threads = [threading.Thread(target=worker) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert len(got) == 9
    for g in got:
        assert all(torch.equal(a, b) for a, b in zip(g, want))


def test_launches_and_allocations_leave_the_interpreter_s_lock_to_other_threads(tmp_path):
    """A launch waits when the queue is full and an allocation may wait for the device.  Every entry point is
    replaced by PyGILState_Check (0 -- the status of success -- without the lock, 1 with it), and the outputs come from an
    allocator that notes the same."""
    calls = per_tensor_calls()
    torch.cuda.synchronize()
    src = tmp_path / "note.c"
    src.write_text("int PyGILState_Check(void);\nint notes, held;\nint (*device_malloc)(void **, unsigned long);\n"
                   "int (*device_free)(void *);\n"
                   "void *take(long n, int device, void *stream) { void *p = 0; ++notes; held += PyGILState_Check();"
                   " return device_malloc(&p, (unsigned long)n) ? 0 : p; }\n"
                   "void give(void *p, long n, int device, void *stream) { device_free(p); }\n")
    so = str(tmp_path / "note.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", so, str(src)], check=True)
    note, runtime, lib = ctypes.CDLL(so), ctypes.CDLL("libcudart.so.12"), mxq.load_library()

    def address(f):
        return ctypes.cast(f, ctypes.c_void_p).value

    ctypes.c_void_p.in_dll(note, "device_malloc").value = address(runtime.cudaMalloc)
    ctypes.c_void_p.in_dll(note, "device_free").value = address(runtime.cudaFree)
    allocator = torch.cuda.memory.CUDAPluggableAllocator(so, "take", "give")
    real = {name: address(getattr(lib, name)) for name in binding._HOST_CALLS}
    checks = {name: a if name.endswith("_bytes") else address(ctypes.pythonapi.PyGILState_Check) for name, a in real.items()}
    p = mxq.prepare_fake_quant(torch.empty(32, device="cuda"), "int4", 32, 0, torch.empty(32, device="cuda"))
    binding._host.bind(checks, binding.FORMATS, torch.nn.Parameter, mxq.MxqError)
    try:
        assert binding._host.run_prepared(p.kind, p.packed) == 0
        for name, call in calls.items():
            before = ctypes.c_int.in_dll(note, "notes").value
            with torch.cuda.use_mem_pool(torch.cuda.MemPool(allocator.allocator())):
                assert call() is not None, name + " launches with the lock held"
            assert ctypes.c_int.in_dll(note, "notes").value > before
            assert ctypes.c_int.in_dll(note, "held").value == 0, name + " allocates with the lock held"
    finally:
        binding._host.bind(real, binding.FORMATS, torch.nn.Parameter, mxq.MxqError)


def test_a_failed_launch_among_several_is_not_enqueued_again():
    x = torch.randn(64, 128, device="cuda")
    codes, scales = mxq.quantize(x, "int8")
    real = {name: ctypes.cast(getattr(mxq.load_library(), name), ctypes.c_void_p).value for name in binding._HOST_CALLS}
    failed = ctypes.CFUNCTYPE(ctypes.c_int)(lambda: -7)                 # MXQ_ERR_CUDA, whatever was launched before it
    binding._host.bind({**real, "mxq_slice_scale_multi": ctypes.cast(failed, ctypes.c_void_p).value}, binding.FORMATS,
                       torch.nn.Parameter, mxq.MxqError)
    try:
        with pytest.raises(mxq.MxqError, match="mxq_slice_scale_multi.*MXQ_ERR_CUDA"):
            mxq.slice_scale_multi(codes, scales, x.numel(), "int8", ["int7", "int6", "int5", "int4", "int3"])
    finally:
        binding._host.bind(real, binding.FORMATS, torch.nn.Parameter, mxq.MxqError)


def test_graph_capture_and_side_stream():
    x = torch.randn(64, 128, device="cuda")
    want = [t.clone() for t in mxq.quantize(x, "e4m3")]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        mxq.quantize(x, "e4m3")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        codes, scales = mxq.quantize(x, "e4m3")
        low = mxq.slice_scale(codes, scales, x.numel(), "e4m3", "e2m1")
    codes.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert same((codes, scales), tuple(want))
    assert np.array_equal(low[0].cpu().numpy(), mxq.slice_scale(*want, x.numel(), "e4m3", "e2m1")[0].cpu().numpy())
