"""The bounds-checked build of the library (libmxq_debug.so, -DMXQ_DEBUG): every entry point on the
sizes where index arithmetic goes wrong first -- one block, one warp's worth, ragged tails, several
tiles -- with exactly sized buffers.  With correct arguments the checker must have looked at every
launch and counted no violation, and the results must still be the oracle's.  The checker's teeth are
shown with the library's own test hook, which registers every range a few bytes short: the kernels'
last (legitimate) accesses are then counted and skipped, while no access ever leaves a real buffer."""
import ctypes
import os

import numpy as np
import pytest
import torch

from oracle import mxq_oracle as orc
from paper_2604_00529_b200 import inputs
from paper_2604_00529_b200.binding import FORMATS, _DqItem, _FqItem, _Item, _PairItem, _QItem, _TiledItem

from gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
LIB = os.path.join(os.path.dirname(HERE), "paper_2604_00529_b200", "libmxq_debug.so")


class Info(ctypes.Structure):
    _fields_ = [("enabled", ctypes.c_int), ("checked_launches", ctypes.c_uint), ("violations", ctypes.c_uint),
                ("first_address", ctypes.c_ulonglong), ("first_bytes", ctypes.c_uint)]


@pytest.fixture(scope="module")
def D():
    if not os.path.exists(LIB):
        pytest.fail("libmxq_debug.so is not built: python -m paper_2604_00529_b200.build --debug")
    L = ctypes.CDLL(LIB)
    vp, sz, i = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
    L.mxq_quantize.argtypes = [vp, i, sz, i, i, vp, vp, vp]
    L.mxq_slice_scale.argtypes = [vp, vp, sz, i, i, i, vp, vp, vp]
    L.mxq_dequantize.argtypes = [vp, vp, sz, i, i, vp, i, vp]
    L.mxq_fake_quant.argtypes = [vp, i, sz, i, i, i, vp, vp]
    L.mxq_fake_quant_bwd.argtypes = [vp, i, sz, vp, vp]
    L.mxq_slice_scale_batched.argtypes = [ctypes.POINTER(_Item), i, i, i, i, vp]
    L.mxq_slice_scale_batched_static.argtypes = [ctypes.POINTER(_Item), i, i, i, i, vp]
    L.mxq_quantize_batched.argtypes = [ctypes.POINTER(_QItem), i, i, i, i, vp]
    L.mxq_dequantize_batched.argtypes = [ctypes.POINTER(_DqItem), i, i, i, i, vp]
    L.mxq_fake_quant_batched.argtypes = [ctypes.POINTER(_FqItem), i, i, i, i, i, vp]
    L.mxq_quantize_tiled.argtypes = [vp, i, sz, sz, i, i, vp, vp, vp]
    L.mxq_tiled_scales_bytes.argtypes = [sz, sz]
    L.mxq_tiled_scales_bytes.restype = sz
    L.mxq_debug_report.argtypes = [ctypes.POINTER(Info), i]
    L.mxq_debug_trim_ranges.argtypes = [sz]
    return L


def report(L, reset=True):
    info = Info()
    assert L.mxq_debug_report(ctypes.byref(info), 1 if reset else 0) == 0
    return info


def u8(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")          # exactly sized: no slack behind the data


def P(t):
    return t.data_ptr()


SIZES = [32, 64, 32 * 31, 32 * 32, 32 * 33, 32 * 64, 32 * 65, 32 * 2051]   # one block ... tiles plus a ragged tail


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("anchor,low", [("int8", "int4"), ("int8", "int6"), ("e4m3", "e2m3"), ("e4m3", "e2m1"), ("int8", "int7")])
def test_single_tensor_entry_points_stay_inside_their_buffers(D, n, anchor, low):
    stream = torch.cuda.current_stream().cuda_stream
    x = inputs.to_bf16_bits((np.random.default_rng(n).standard_normal(n) * 0.3).astype(np.float32))
    xd = to_dev(x)
    report(D)
    codes, scales = u8(n), u8(n // 32)
    assert D.mxq_quantize(P(xd), 1, n, FORMATS[anchor], 32, P(codes), P(scales), stream) == 0
    b = orc.bits(low)
    lc, ls = u8(n * b // 8), u8(n // 32)
    assert D.mxq_slice_scale(P(codes), P(scales), n, 32, FORMATS[anchor], FORMATS[low], P(lc), P(ls), stream) == 0
    y = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    y32 = torch.empty(n, dtype=torch.float32, device="cuda")
    assert D.mxq_dequantize(P(lc), P(ls), n, FORMATS[low], 32, P(y), 1, stream) == 0
    assert D.mxq_dequantize(P(lc), P(ls), n, FORMATS[low], 32, P(y32), 0, stream) == 0
    f = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    g = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    assert D.mxq_fake_quant(P(xd), 1, n, FORMATS[low], 32, 1, P(f), stream) == 0
    assert D.mxq_fake_quant_bwd(P(f), 1, n, P(g), stream) == 0
    info = report(D)
    assert info.enabled == 1 and info.checked_launches == 6
    assert info.violations == 0, "first bad access: %#x (%d bytes)" % (info.first_address, info.first_bytes)
    wc, ws = orc.quantize(x, anchor)
    w4, s4 = orc.slice_scale(wc, ws, anchor, low)
    assert np.array_equal(to_host(codes), orc.pack(wc, 8)) and np.array_equal(to_host(scales), ws)
    assert np.array_equal(to_host(lc), orc.pack(w4, b)) and np.array_equal(to_host(ls), s4)
    want = orc.dequantize(w4, s4, low, out_dtype=orc.BF16)
    assert np.array_equal(to_host(y), want) and np.array_equal(to_host(f), want) and np.array_equal(to_host(g), want)
    assert np.array_equal(to_host(y32).view(np.uint32), orc.dequantize(w4, s4, low).view(np.uint32))


def test_batched_entry_points_stay_inside_their_buffers(D):
    stream = torch.cuda.current_stream().cuda_stream
    sizes = [32, 32 * 65, 64, 32 * 700, 32 * 33, 32 * 2051, 32 * 7]
    rng = np.random.default_rng(3)
    xs = [inputs.to_bf16_bits((rng.standard_normal(n) * 2.0 ** rng.integers(-8, 8)).astype(np.float32)) for n in sizes]
    xd = [to_dev(x) for x in xs]
    codes = [u8(n) for n in sizes]
    scales = [u8(n // 32) for n in sizes]
    lc = [u8(n // 2) for n in sizes]
    ls = [u8(n // 32) for n in sizes]
    lc2 = [u8(n // 2) for n in sizes]
    ls2 = [u8(n // 32) for n in sizes]
    y = [torch.empty(n, dtype=torch.bfloat16, device="cuda") for n in sizes]
    f = [torch.empty(n, dtype=torch.bfloat16, device="cuda") for n in sizes]
    k = len(sizes)
    report(D)
    q = (_QItem * k)(*[_QItem(P(xd[j]), sizes[j], P(codes[j]), P(scales[j])) for j in range(k)])
    assert D.mxq_quantize_batched(q, k, 1, FORMATS["e4m3"], 32, stream) == 0
    it = (_Item * k)(*[_Item(P(codes[j]), P(scales[j]), sizes[j], P(lc[j]), P(ls[j])) for j in range(k)])
    assert D.mxq_slice_scale_batched(it, k, 32, FORMATS["e4m3"], FORMATS["e2m1"], stream) == 0
    it2 = (_Item * k)(*[_Item(P(codes[j]), P(scales[j]), sizes[j], P(lc2[j]), P(ls2[j])) for j in range(k)])
    assert D.mxq_slice_scale_batched_static(it2, k, 32, FORMATS["e4m3"], FORMATS["e2m1"], stream) == 0
    dq = (_DqItem * k)(*[_DqItem(P(lc[j]), P(ls[j]), sizes[j], P(y[j])) for j in range(k)])
    assert D.mxq_dequantize_batched(dq, k, FORMATS["e2m1"], 32, 1, stream) == 0
    fq = (_FqItem * k)(*[_FqItem(P(xd[j]), P(f[j]), sizes[j]) for j in range(k)])
    assert D.mxq_fake_quant_batched(fq, k, 1, FORMATS["e2m1"], 32, 1, stream) == 0
    rows, cols = 130, 160                                   # edge tiles in both directions
    xm = to_dev(inputs.to_bf16_bits(rng.standard_normal(rows * cols).astype(np.float32)))
    tc, tt = u8(rows * cols), u8(D.mxq_tiled_scales_bytes(rows, cols // 32))
    assert D.mxq_quantize_tiled(P(xm), 1, rows, cols, FORMATS["e4m3"], 32, P(tc), P(tt), stream) == 0
    info = report(D)
    assert info.enabled == 1 and info.checked_launches == 6
    assert info.violations == 0, "first bad access: %#x (%d bytes)" % (info.first_address, info.first_bytes)
    for j, x in enumerate(xs):
        wc, ws = orc.quantize(x, "e4m3")
        w4, s4 = orc.slice_scale(wc, ws, "e4m3", "e2m1")
        assert np.array_equal(to_host(lc[j]), orc.pack(w4, 4)) and np.array_equal(to_host(ls[j]), s4), j
        assert np.array_equal(to_host(lc2[j]), orc.pack(w4, 4)) and np.array_equal(to_host(ls2[j]), s4), j
        want = orc.dequantize(w4, s4, "e2m1", out_dtype=orc.BF16)
        assert np.array_equal(to_host(y[j]), want) and np.array_equal(to_host(f[j]), want), j


@pytest.mark.parametrize("src,lows", [("int8", ["int7", "int6", "int5", "int3"]), ("e4m3", ["e3m3", "e2m3", "e2m1"])])
@pytest.mark.parametrize("units,block", [(1, 32), (31, 16), (257, 16), (258, 64), (516, 128), (771, 32)])
def test_target_sets_pairs_and_padding_stay_inside_their_buffers(D, src, lows, units, block):
    """The kernels that read an anchor once for several targets, block 16, and the CTAs that write the padding of tiled
    scales, in the bounds-checked build."""
    vp, i = ctypes.c_void_p, ctypes.c_int
    D.mxq_slice_scale_multi.argtypes = [vp, vp, ctypes.c_size_t, i, i, i, ctypes.POINTER(i), ctypes.POINTER(vp), ctypes.POINTER(vp), vp]
    D.mxq_slice_scale_pair_batched.argtypes = [ctypes.POINTER(_PairItem), i, i, i, i, i, vp]
    D.mxq_slice_scale_tiled_batched.argtypes = [ctypes.POINTER(_TiledItem), i, i, i, i, vp]
    stream = torch.cuda.current_stream().cuda_stream
    rng = np.random.default_rng(units)
    n, k = units * 32, len(lows)
    hc, hs = rng.integers(0, 256, n).astype(np.uint8), rng.integers(0, 256, n // block).astype(np.uint8)
    codes, scales = to_dev(hc), to_dev(hs)
    fmts = (i * k)(*[FORMATS[f] for f in lows])
    launches = 0
    report(D)
    sets = [(u8(n * orc.bits(f) // 8), u8(n // block)) for f in lows]
    assert D.mxq_slice_scale_multi(P(codes), P(scales), n, block, FORMATS[src], k, fmts, (vp * k)(*[P(c) for c, _ in sets]),
                                   (vp * k)(*[P(s) for _, s in sets]), stream) == 0
    one = [(u8(n * orc.bits(f) // 8), u8(n // block)) for f in lows]
    for f, (c, s) in zip(lows, one):
        assert D.mxq_slice_scale(P(codes), P(scales), n, block, FORMATS[src], FORMATS[f], P(c), P(s), stream) == 0
    launches += 1 + k
    results = list(zip(lows * 2, sets + one))
    if block >= 32:
        pair = [(u8(n * orc.bits(f) // 8), u8(n // block)) for f in lows[:2]]
        item = (_PairItem * 1)(_PairItem(P(codes), P(scales), n, P(pair[0][0]), P(pair[0][1]), P(pair[1][0]), P(pair[1][1])))
        assert D.mxq_slice_scale_pair_batched(item, 1, block, FORMATS[src], FORMATS[lows[0]], FORMATS[lows[1]], stream) == 0
        launches += 1
        results += list(zip(lows[:2], pair))
    if block == 32 and src == "e4m3":
        rows, kb = (units // 3, 3) if units >= 3 else (1, units)
        nbytes = D.mxq_tiled_scales_bytes(rows, kb)
        tiled = [(u8(rows * kb * 16), u8(nbytes)) for _ in range(2)]
        items = (_TiledItem * 2)(*[_TiledItem(P(codes), P(scales), rows, kb * 32, P(c), P(s)) for c, s in tiled])
        assert D.mxq_slice_scale_tiled_batched(items, 2, 32, FORMATS[src], FORMATS["e2m1"], stream) == 0
        launches += 1
    info = report(D)
    assert info.checked_launches == launches
    assert info.violations == 0, "first bad access: %#x (%d bytes)" % (info.first_address, info.first_bytes)
    for f, (c, s) in results:
        wc, ws = orc.slice_scale(hc, hs, src, f, block)
        assert np.array_equal(to_host(c), orc.pack(wc, orc.bits(f))) and np.array_equal(to_host(s), ws), f
    if block == 32 and src == "e4m3":
        wc, ws = orc.slice_scale(hc, hs, src, "e2m1", 32)
        want = orc.tile_scales(ws[:rows * kb].reshape(rows, kb), rows, kb)
        for c, s in tiled:
            assert np.array_equal(to_host(c), orc.pack(wc[:rows * kb * 32], 4)) and np.array_equal(to_host(s), want)


@pytest.mark.parametrize("block", [16, 32])
def test_two_unit_kernels_stay_inside_their_buffers(D, block):
    """A launch large enough for two lane units per thread, with a ragged last warp."""
    stream = torch.cuda.current_stream().cuda_stream
    n = (148 * 8 * 256 + 5) * 32
    period = 1004 * 32                                            # the data repeats; no multiple of a tile
    rng = np.random.default_rng(block)
    hc, hs = rng.integers(0, 256, period).astype(np.uint8), rng.integers(0, 256, period // block).astype(np.uint8)

    def whole(pattern, count):
        p = to_dev(pattern)
        return p.repeat(-(-count // p.numel()))[:count].contiguous()

    codes, scales = whole(hc, n), whole(hs, n // block)
    lc, ls = u8(n * 6 // 8), u8(n // block)
    y = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    report(D)
    assert D.mxq_slice_scale(P(codes), P(scales), n, block, FORMATS["e4m3"], FORMATS["e2m3"], P(lc), P(ls), stream) == 0
    assert D.mxq_dequantize(P(lc), P(ls), n, FORMATS["e2m3"], block, P(y), 1, stream) == 0
    info = report(D)
    assert info.checked_launches == 2
    assert info.violations == 0, "first bad access: %#x (%d bytes)" % (info.first_address, info.first_bytes)
    wc, ws = orc.slice_scale(hc, hs, "e4m3", "e2m3", block)
    assert torch.equal(lc, whole(orc.pack(wc, 6), lc.numel())) and torch.equal(ls, whole(ws, ls.numel()))
    want = orc.dequantize(wc, ws, "e2m3", block, orc.BF16)
    assert torch.equal(y.view(torch.int16), whole(want.view(np.uint16), n).view(torch.int16))


def test_the_checker_counts_and_skips_what_leaves_a_registered_range(D):
    """Ranges registered 32 bytes short: the kernel's stores and loads of the last 32 bytes of each
    buffer are outside them, are counted, and are skipped (the output keeps its fill there)."""
    stream = torch.cuda.current_stream().cuda_stream
    n = 32 * 64
    x = inputs.to_bf16_bits(np.random.default_rng(1).standard_normal(n).astype(np.float32))
    xd = to_dev(x)
    y = torch.full((n,), 7.0, dtype=torch.bfloat16, device="cuda")
    report(D)
    assert D.mxq_debug_trim_ranges(32) == 1
    try:
        assert D.mxq_fake_quant(P(xd), 1, n, FORMATS["int8"], 32, 0, P(y), stream) == 0
        info = report(D)
    finally:
        D.mxq_debug_trim_ranges(0)
    assert info.checked_launches == 1 and info.violations == 2            # one load and one store of 32 bytes
    assert info.first_bytes == 32 and info.first_address in (P(xd) + 2 * n - 32, P(y) + 2 * n - 32)
    got = to_host(y)
    want = orc.fake_quant(x, "int8")
    assert np.array_equal(got[:-16], want[:-16])
    assert np.all(got[-16:] == 0x40E0)                                     # 7.0 in BF16: the store was skipped
    # and with whole ranges again the same call is clean
    assert D.mxq_fake_quant(P(xd), 1, n, FORMATS["int8"], 32, 0, P(y), stream) == 0
    info = report(D)
    assert info.violations == 0 and np.array_equal(to_host(y), want)


def test_release_build_reports_that_it_is_not_a_debug_build():
    import paper_2604_00529_b200 as mxq
    L = mxq.load_library()
    L.mxq_debug_report.argtypes = [ctypes.POINTER(Info), ctypes.c_int]
    info = Info()
    assert L.mxq_debug_report(ctypes.byref(info), 0) == 0 and info.enabled == 0 and info.violations == 0
    L.mxq_debug_trim_ranges.argtypes = [ctypes.c_size_t]
    assert L.mxq_debug_trim_ranges(64) == 0


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("src,dst", [("int7", "int5"), ("int5", "int3"), ("e3m3", "e2m2"), ("e3m2", "e2m1")])
def test_stored_lower_formats_stay_inside_their_buffers(D, n, src, dst):
    """The unpacking of sources below eight bits, and the FP32 reconstruction's aligned words round 5- and 3-byte pieces."""
    stream = torch.cuda.current_stream().cuda_stream
    rng = np.random.default_rng(n)
    hc = rng.integers(0, 1 << orc.bits(src), n).astype(np.uint8)
    hs = rng.integers(0, 256, n // 32).astype(np.uint8)
    codes, scales = to_dev(orc.pack(hc, orc.bits(src))), to_dev(hs)
    report(D)
    lc, ls = u8(n * orc.bits(dst) // 8), u8(n // 32)
    assert D.mxq_slice_scale(P(codes), P(scales), n, 32, FORMATS[src], FORMATS[dst], P(lc), P(ls), stream) == 0
    y32 = torch.empty(n, dtype=torch.float32, device="cuda")
    assert D.mxq_dequantize(P(lc), P(ls), n, FORMATS[dst], 32, P(y32), 0, stream) == 0
    info = report(D)
    assert info.enabled == 1 and info.checked_launches == 2
    assert info.violations == 0, "first bad access: %#x (%d bytes)" % (info.first_address, info.first_bytes)
    wc, ws = orc.slice_scale(hc, hs, src, dst)
    assert np.array_equal(to_host(lc), orc.pack(wc, orc.bits(dst))) and np.array_equal(to_host(ls), ws)
    assert np.array_equal(to_host(y32).view(np.uint32), orc.dequantize(wc, ws, dst).view(np.uint32))
