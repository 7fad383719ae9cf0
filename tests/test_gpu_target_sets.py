"""Several targets from one read of the anchor: every set of lower formats against the oracle, at the sizes
where a tile of 256 lane units (8192 codes) begins, ends and is left ragged, with all byte values as codes
(E4M3 NaN codes among them) and as scale bytes."""
from __future__ import annotations

import itertools

import numpy as np
import pytest
import torch

import paper_2604_00529_b200 as mxq
from oracle import mxq_oracle as orc
from gpu_util import FP_FORMATS, INT_FORMATS, Guarded, bits_equal, to_dev, to_host

LOWER = {"int8": INT_FORMATS[1:], "e4m3": FP_FORMATS[1:]}


def _input(src, n, block, seed):
    rng = np.random.default_rng(seed)
    codes = rng.integers(0, 256, n).astype(np.uint8)
    codes[:min(n, 256)] = np.arange(min(n, 256))
    if seed % 2:
        codes[(codes & 0x7F) == 0x7F] = 5                     # an anchor without NaN codes: the other route
    return codes, rng.integers(0, 256, n // block).astype(np.uint8)


@pytest.mark.gpu
@pytest.mark.parametrize("units,block", [(1, 32), (4, 128), (31, 16), (255, 32), (256, 64), (257, 16), (516, 128), (771, 32)])
@pytest.mark.parametrize("src", ["int8", "e4m3"])
def test_every_set_of_targets(src, units, block):
    n = units * 32
    for seed, size in enumerate(range(2, len(LOWER[src]) + 1)):
        codes, scales = _input(src, n, block, units + seed)
        want = {f: orc.slice_scale(codes, scales, src, f, block) for f in LOWER[src]}
        dc, ds = to_dev(codes), to_dev(scales)
        for fmts in itertools.combinations(LOWER[src], size):
            fmts = fmts if size % 2 else fmts[::-1]
            outs = [(Guarded(mxq.codes_bytes(n, f)), Guarded(n // block)) for f in fmts]
            mxq.slice_scale_multi(dc, ds, n, src, fmts, block, [(c.view, s.view) for c, s in outs])
            torch.cuda.synchronize()
            for f, (c, s) in zip(fmts, outs):
                c.check()
                s.check()
                assert bits_equal(to_host(c.view), orc.pack(want[f][0], orc.bits(f))), (fmts, f)
                assert bits_equal(to_host(s.view), want[f][1]), (fmts, f)


@pytest.mark.gpu
@pytest.mark.parametrize("src,fmts", [("int8", ["int4", "int4"]), ("int8", ["int8", "int6", "int2", "int6", "int8"]),
                                      ("e4m3", ["e4m3", "e2m1"]), ("e4m3", ["e3m3", "e2m2", "e3m3", "e4m3", "e2m3"])])
def test_repeated_formats_and_the_anchor_itself(src, fmts):
    n = 300 * 32
    codes, scales = _input(src, n, 32, 2)
    for f, (c, s) in zip(fmts, mxq.slice_scale_multi(to_dev(codes), to_dev(scales), n, src, fmts, 32)):
        wc, ws = orc.slice_scale(codes, scales, src, f, 32)
        assert bits_equal(to_host(c), orc.pack(wc, orc.bits(f))) and bits_equal(to_host(s), ws), f


@pytest.mark.gpu
@pytest.mark.parametrize("src", ["int8", "e4m3"])
def test_every_pair_over_a_set_of_tensors(src):
    sizes = [32, 255 * 32, 64, 256 * 32, 257 * 32, 96, 700 * 32]
    tensors = [_input(src, n, 32, k) for k, n in enumerate(sizes)]
    dev = [(to_dev(c), to_dev(s)) for c, s in tensors]
    want = {f: [orc.slice_scale(c, s, src, f, 32) for c, s in tensors] for f in LOWER[src]}
    for a, b in itertools.permutations(LOWER[src], 2):
        outs = [[Guarded(mxq.codes_bytes(n, a)), Guarded(n // 32), Guarded(mxq.codes_bytes(n, b)), Guarded(n // 32)] for n in sizes]
        mxq.slice_scale_pair_batched([(c, s, n, *(g.view for g in o)) for (c, s), n, o in zip(dev, sizes, outs)], src, a, b)
        torch.cuda.synchronize()
        for k, o in enumerate(outs):
            for g in o:
                g.check()
            for f, gc, gs in ((a, o[0], o[1]), (b, o[2], o[3])):
                assert bits_equal(to_host(gc.view), orc.pack(want[f][k][0], orc.bits(f))), (a, b, f, k)
                assert bits_equal(to_host(gs.view), want[f][k][1]), (a, b, f, k)
