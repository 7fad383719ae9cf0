"""The bytes of the tiled scale buffer that no block covers are written as 0 by the producing kernel: shapes on
both sides of the 128-row and 4-column edges, one row, and padding that takes several CTAs; the buffer
starts poisoned."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2604_00529_b200 as mxq
from oracle import mxq_oracle as orc
from gpu_util import Guarded, bits_equal, to_dev, to_host


@pytest.mark.gpu
@pytest.mark.parametrize("kb", [1, 3, 4, 6, 129, 448])
@pytest.mark.parametrize("rows", [1, 33, 127, 128, 129, 1000])
def test_every_byte_of_the_tiled_buffer_is_written(rows, kb):
    n = rows * kb * 32
    x = np.random.default_rng(rows * 1000 + kb).standard_normal(n).astype(np.float32)
    wc, ws = orc.quantize(x, "e4m3", 32)
    want = orc.tile_scales(ws.reshape(rows, kb), rows, kb)
    out = Guarded(mxq.tiled_scales_bytes(rows, kb))
    codes, _ = mxq.quantize_tiled(to_dev(x).view(rows, kb * 32), "e4m3", 32, tiled_scales=out.view)
    torch.cuda.synchronize()
    out.check()
    assert bits_equal(to_host(out.view), want) and bits_equal(to_host(codes), orc.pack(wc, 8))
    lc, ls = orc.slice_scale(wc, ws, "e4m3", "e2m1", 32)
    want = orc.tile_scales(ls.reshape(rows, kb), rows, kb)
    one, two = Guarded(out.nbytes), Guarded(out.nbytes)
    low, _ = mxq.slice_scale_tiled(codes, to_dev(ws), rows, kb * 32, "e4m3", "e2m1", 32, out_tiled_scales=one.view)
    other = torch.empty_like(low)
    first = (to_dev(wc[:32]), to_dev(ws[:1]), 1, 32, torch.empty(16, dtype=torch.uint8, device="cuda"),
             torch.empty(512, dtype=torch.uint8, device="cuda"))
    mxq.slice_scale_tiled_batched([first, (codes, to_dev(ws), rows, kb * 32, other, two.view), first], "e4m3", "e2m1", 32)
    torch.cuda.synchronize()
    for t, c in ((one, low), (two, other)):
        t.check()
        assert bits_equal(to_host(t.view), want) and bits_equal(to_host(c), orc.pack(lc, 4))
