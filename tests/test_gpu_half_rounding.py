"""The conversions that round on the FP16 pipe and those that start from a stored lower format: where the packed arithmetic
could go wrong (BF16 subnormals, the smallest scales, halfway points, clipped ends) and where its tiles end."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2604_00529_b200 as mxq
from oracle import mxq_oracle as orc
from gpu_util import Guarded, INT_FORMATS, bits_equal, first_diff, gpu_dequantize, gpu_quantize, gpu_slice_scale, ss_pairs, to_dev, to_host

pytestmark = pytest.mark.gpu

# lane units of 32 codes: one, around a warp tile (64), around a CTA's (256)
UNITS = [1, 63, 65, 255, 257, 515]


@pytest.mark.parametrize("block", [16, 32, 128])
@pytest.mark.parametrize("fmt", INT_FORMATS)
def test_bf16_blocks_of_every_exponent(fmt, block):
    """Blocks whose largest element walks through every BF16 exponent, subnormals included, each filled with patterns of
    the eight binades below it; then a block of zeros and one of the smallest subnormal behind each."""
    rng = np.random.default_rng(block)
    rows = []
    for exponent in range(0, 255):
        low = max(0, exponent - 8) << 7
        for _ in range(2):
            rows.append(rng.integers(low, (exponent + 1) << 7, block) | rng.integers(0, 2, block) << 15)
        rows.append(np.zeros(block, np.int64))
        rows.append(np.full(block, 1) | rng.integers(0, 2, block) << 15)
    x = np.concatenate(rows).astype(np.uint16)
    x = np.resize(x, -(-x.size // 128) * 128)
    codes, scales = gpu_quantize(x, fmt, block)
    wc, ws = orc.quantize(x, fmt, block)
    assert bits_equal(scales, ws), first_diff(scales, ws)
    assert bits_equal(codes, orc.pack(wc, orc.bits(fmt))), first_diff(codes, orc.pack(wc, orc.bits(fmt)))


def halfway_points(fmt, s):
    """Blocks of every multiple of 1/4 below the next binade that BF16 holds with its BF16 neighbours, both signs, times 2^s; each block's
    scale byte is 127 + s.  (The neighbours of 0 are subnormals, which an exponent shift does not scale: signed zeros.)"""
    top = 1 << (orc.bits(fmt) - 1)
    r = np.arange(0, 4 * top, dtype=np.float32) / 4
    bits = (r.view(np.uint32) >> 16).astype(np.int64)
    near = np.concatenate([bits, np.maximum(bits - 1, 0), np.minimum(bits + 1, int(np.float32(top).view(np.uint32) >> 16) - 1)])
    near = np.concatenate([near, near | 0x8000])
    near = np.resize(near, -(-near.size // 31) * 31).reshape(-1, 31)
    fix = np.full((near.shape[0], 1), int(np.float32(top / 2).view(np.uint32) >> 16))      # sets the block's exponent
    blocks = np.concatenate([near, fix], axis=1)
    field = blocks >> 7 & 0xFF
    assert np.all((field == 0) | (1 <= field + s) & (field + s <= 254))
    return np.where(field, blocks + s * 128, blocks & 0x8000).reshape(-1).astype(np.uint16)


@pytest.mark.parametrize("s", [-60, -20, -7, 0, 5, 40])
@pytest.mark.parametrize("fmt", INT_FORMATS)
def test_bf16_halfway_points(fmt, s):
    """Ties go away from zero, their neighbours do not follow them, the upper end is clipped, under each of six scales."""
    x = halfway_points(fmt, s)
    wc, ws = orc.quantize(x, fmt)
    assert np.all(ws == 127 + s)                                     # no block lost to a larger element than meant
    assert np.unique(wc).size == (1 << orc.bits(fmt)) - 1            # every code but -2^(b-1), which is never produced
    codes, scales = gpu_quantize(x, fmt)
    assert bits_equal(scales, ws), first_diff(scales, ws)
    assert bits_equal(codes, orc.pack(wc, orc.bits(fmt))), first_diff(codes, orc.pack(wc, orc.bits(fmt)))


@pytest.mark.parametrize("src,dst", [p for p in ss_pairs(all_pairs=True) if orc.bits(p[0]) < 8 and p[0] != p[1]], ids=lambda v: v)
@pytest.mark.parametrize("block", [16, 32])
def test_a_stored_lower_format_goes_lower(src, dst, block):
    rng = np.random.default_rng(block)
    for units in UNITS:
        n = 32 * units
        codes = rng.integers(0, 1 << orc.bits(src), n).astype(np.uint8)
        scales = rng.integers(0, 256, n // block).astype(np.uint8)
        got_c, got_s = gpu_slice_scale(orc.pack(codes, orc.bits(src)), scales, n, src, dst, block)
        wc, ws = orc.slice_scale(codes, scales, src, dst, block)
        assert bits_equal(got_s, ws), (units, first_diff(got_s, ws))
        assert bits_equal(got_c, orc.pack(wc, orc.bits(dst))), (units, first_diff(got_c, orc.pack(wc, orc.bits(dst))))


@pytest.mark.parametrize("fmt", ["int7", "int6", "int5", "int3", "e3m3", "e3m2", "e2m3", "e2m2"])
def test_reconstruction_to_f32_of_pieces_that_are_no_vector(fmt):
    """Every length of a tile's ragged end: 1 ... 33 blocks, then around the tiles of a warp and of a CTA."""
    rng = np.random.default_rng(7)
    for units in list(range(1, 34)) + UNITS[1:]:
        n = 32 * units
        codes = rng.integers(0, 1 << orc.bits(fmt), n).astype(np.uint8)
        scales = rng.integers(0, 256, units).astype(np.uint8)
        got = gpu_dequantize(orc.pack(codes, orc.bits(fmt)), scales, n, fmt)
        want = orc.dequantize(codes, scales, fmt)
        assert bits_equal(got, want), (units, first_diff(got, want))


@pytest.mark.parametrize("fmt", ["int7", "int6", "int5", "int3", "e3m3", "e2m3", "e2m2"])
def test_batched_reconstruction_to_f32_of_pieces_that_are_no_vector(fmt):
    """The same pieces in one launch over tensors that end inside a warp's tile: lanes beyond an end read its last piece."""
    rng = np.random.default_rng(11)
    sets = []
    for units in [1, 2, 15, 16, 17, 33, 65, 257]:
        n = 32 * units
        codes = rng.integers(0, 1 << orc.bits(fmt), n).astype(np.uint8)
        scales = rng.integers(0, 256, units).astype(np.uint8)
        sets.append((to_dev(orc.pack(codes, orc.bits(fmt))), to_dev(scales), n, Guarded(4 * n, torch.float32), orc.dequantize(codes, scales, fmt)))
    mxq.dequantize_batched([(c, s, n, y.view) for c, s, n, y, _ in sets], fmt)
    torch.cuda.synchronize()
    for _, _, n, y, want in sets:
        y.check()
        assert bits_equal(to_host(y.view), want), (n, first_diff(to_host(y.view), want))
