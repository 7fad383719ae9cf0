"""Both sides of every rule that picks a kernel shape by size: one lane unit per thread under eight CTAs per SM (148 x 8
CTAs of 256 units; half that for the reconstruction of four and fewer bits) and two above, the item tables of 64 entries
and the largest ones.  Small tensors never reach the two-unit kernels, so their ragged ends, blocks, NaN codes and scale
halves are checked here, at the sizes where real launches run them."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_2604_00529_b200 as mxq
from oracle import mxq_oracle as orc
from paper_2604_00529_b200 import inputs
from gpu_util import Guarded, bits_equal, first_diff, to_dev, to_host

pytestmark = pytest.mark.gpu

CTA = 256                                     # lane units of 32 codes that a CTA of the two-unit kernels covers
PERIOD = 4 * 251                              # units after which the data repeats: no multiple of a tile


def repeated(pattern: np.ndarray, n: int) -> torch.Tensor:
    p = to_dev(pattern)
    return p.repeat(-(-n // p.numel()))[:n].contiguous()


def codes_and_scales(fmt: str, block: int, seed: int):
    """One period of packed codes (every byte value; units with and without E4M3 NaN codes) and of scale bytes."""
    rng = np.random.default_rng(seed)
    n = PERIOD * 32
    codes = rng.integers(0, 1 << orc.bits(fmt), n).astype(np.uint8)
    if fmt == "e4m3":
        units = codes.reshape(-1, 32)
        units[::2][(units[::2] & 0x7F) == 0x7F] = 5
        units[1::2, 7] = 0xFF
    return codes, rng.integers(0, 256, n // block).astype(np.uint8)


def unit_counts(ctas: int):
    """One whole CTA below the rule's limit, just behind it with a ragged CTA, and above it with a ragged warp."""
    return [(ctas - 1) * CTA, (ctas - 1) * CTA + 4, ctas * CTA + 132]


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("dst", ["e3m3", "e3m2", "e2m3", "e2m2"])
def test_slice_scale_on_both_sides_of_the_small_launch_rule(dst, block):
    codes, scales = codes_and_scales("e4m3", block, block)
    wc, ws = orc.slice_scale(codes, scales, "e4m3", dst, block)
    packed = orc.pack(wc, orc.bits(dst))
    for units in unit_counts(148 * 8):
        n = units * 32
        oc, os_ = Guarded(mxq.codes_bytes(n, dst)), Guarded(n // block)
        mxq.slice_scale(repeated(codes, n), repeated(scales, n // block), n, "e4m3", dst, block, oc.view, os_.view)
        torch.cuda.synchronize()
        oc.check()
        os_.check()
        assert torch.equal(oc.view, repeated(packed, oc.nbytes)), units
        assert torch.equal(os_.view, repeated(ws, os_.nbytes)), units


@pytest.mark.parametrize("block", [16, 32, 64])
@pytest.mark.parametrize("dst", ["int7", "int6", "int4", "int3", "int2"])
def test_slice_scale_from_mxint8_on_both_sides_of_its_one_wave_rules(dst, block):
    """Ten CTAs per SM (twelve to four and three bits; to four bits also five, to three also four), and the smallest tensors."""
    codes, scales = codes_and_scales("int8", block, 5 * block)
    wc, ws = orc.slice_scale(codes, scales, "int8", dst, block)
    packed = orc.pack(wc, orc.bits(dst))
    for units in [1, 65, 3 * CTA - 2] + unit_counts(148 * 4) + unit_counts(148 * 5) + unit_counts(148 * 10) + unit_counts(148 * 12):
        n = max(units * 32, block) // block * block
        oc, os_ = Guarded(mxq.codes_bytes(n, dst)), Guarded(n // block)
        mxq.slice_scale(repeated(codes, n), repeated(scales, n // block), n, "int8", dst, block, oc.view, os_.view)
        torch.cuda.synchronize()
        oc.check()
        os_.check()
        assert torch.equal(oc.view, repeated(packed, oc.nbytes)), units
        assert torch.equal(os_.view, repeated(ws, os_.nbytes)), units


@pytest.mark.parametrize("ctas", [148 * 10, 148 * 10 + 1, 148 * 12, 148 * 12 + 1])
@pytest.mark.parametrize("dst", ["int7", "int6", "int3"])
def test_mxint8_sets_on_both_sides_of_the_one_wave_rules(dst, ctas):
    codes, scales = codes_and_scales("int8", 32, 9)
    wc, ws = orc.slice_scale(codes, scales, "int8", dst, 32)
    packed = orc.pack(wc, orc.bits(dst))
    items, outs = [], []
    for units in (1, 2 * CTA - 3, (ctas - 4) * CTA - 64, CTA):        # 1 + 2 + (ctas - 4) + 1 CTAs
        n = units * 32
        oc, os_ = Guarded(mxq.codes_bytes(n, dst)), Guarded(units)
        items.append((repeated(codes, n), repeated(scales, units), n, oc.view, os_.view))
        outs.append((oc, os_))
    mxq.slice_scale_batched(items, "int8", dst)
    torch.cuda.synchronize()
    for oc, os_ in outs:
        oc.check()
        os_.check()
        assert torch.equal(oc.view, repeated(packed, oc.nbytes))
        assert torch.equal(os_.view, repeated(ws, os_.nbytes))


@pytest.mark.parametrize("block", [16, 32, 64, 128])
@pytest.mark.parametrize("fmt", ["int8", "e4m3", "int7", "e2m3", "e2m2", "int4", "e2m1", "int3"])
def test_reconstruction_on_both_sides_of_the_small_launch_rule(fmt, block):
    codes, scales = codes_and_scales(fmt, block, 3 * block)
    want = orc.dequantize(codes, scales, fmt, block, orc.BF16)
    packed = orc.pack(codes, orc.bits(fmt))
    for units in unit_counts(148 * 8 if orc.bits(fmt) > 4 else 148 * 4):
        n = units * 32
        y = Guarded(n * 2, torch.bfloat16)
        mxq.dequantize(repeated(packed, mxq.codes_bytes(n, fmt)), repeated(scales, n // block), n, fmt, block, dst=y.view)
        torch.cuda.synchronize()
        y.check()
        assert torch.equal(y.view.view(torch.int16), repeated(want.view(np.uint16), n).view(torch.int16)), units


@pytest.mark.parametrize("count", [64, 65])
@pytest.mark.parametrize("bf16", [True, False])
def test_sets_on_both_sides_of_the_small_item_table(count, bf16):
    """Every batched operation at the last set of the small item table and the first of the large one; tensors of one
    block, of whole CTA tiles and one block on either side of them."""
    rng = np.random.default_rng(count + bf16)
    edge = 128 if bf16 else 64                                     # blocks of a CTA tile of the fake-quant (the smallest of the tiles)
    nblks = [int(rng.choice([1, 2, edge - 1, edge, edge + 1, 2 * edge, 2 * edge + 1, 255, 256, 257])) for _ in range(count)]
    xs = [rng.standard_normal(32 * nb).astype(np.float32) * np.float32(2.0 ** rng.integers(-8, 8)) for nb in nblks]
    if bf16:
        xs = [inputs.to_bf16_bits(x) for x in xs]
    dev, dt = [to_dev(x) for x in xs], torch.bfloat16 if bf16 else torch.float32

    def u8(sizes):
        return [Guarded(int(b)) for b in sizes]

    n = [32 * nb for nb in nblks]
    codes, scales, y, f = u8(n), u8(nblks), [Guarded(k * dt.itemsize, dt) for k in n], [Guarded(k * dt.itemsize, dt) for k in n]
    c6, s6, c4, s4 = u8(k * 6 // 8 for k in n), u8(nblks), u8(k // 2 for k in n), u8(nblks)
    rows = [1 if nb < 8 else nb // 3 for nb in nblks]              # tiled: matrices of one row, and of three block-columns
    kb = [nb // r for nb, r in zip(nblks, rows)]
    ct, st = u8(r * k * 32 // 2 for r, k in zip(rows, kb)), u8(mxq.tiled_scales_bytes(r, k) for r, k in zip(rows, kb))
    mxq.quantize_batched([(x, c.view, s.view) for x, c, s in zip(dev, codes, scales)], "e4m3")
    mxq.slice_scale_pair_batched([(c.view, s.view, k, a.view, b.view, d.view, e.view)
                                  for c, s, k, a, b, d, e in zip(codes, scales, n, c6, s6, c4, s4)], "e4m3", "e2m3", "e2m1")
    mxq.dequantize_batched([(c.view, s.view, k, d.view) for c, s, k, d in zip(c4, s4, n, y)], "e2m1")
    mxq.fake_quant_batched([(x, d.view) for x, d in zip(dev, f)], "e2m1", 32, mxq.FQ_VIA_ANCHOR)
    mxq.slice_scale_tiled_batched([(c.view, s.view, r, k * 32, a.view, b.view)
                                   for c, s, r, k, a, b in zip(codes, scales, rows, kb, ct, st)], "e4m3", "e2m1")
    torch.cuda.synchronize()
    for k, x in enumerate(xs):
        for g in (codes[k], scales[k], y[k], f[k], c6[k], s6[k], c4[k], s4[k], ct[k], st[k]):
            g.check()
        wc, ws = orc.quantize(x, "e4m3")
        w6, w6s = orc.slice_scale(wc, ws, "e4m3", "e2m3")
        w4, w4s = orc.slice_scale(wc, ws, "e4m3", "e2m1")
        want = orc.dequantize(w4, w4s, "e2m1", 32, orc.BF16 if bf16 else orc.F32)
        m = rows[k] * kb[k]
        for got, exp in ((codes[k], orc.pack(wc, 8)), (scales[k], ws), (c6[k], orc.pack(w6, 6)), (s6[k], w6s),
                         (c4[k], orc.pack(w4, 4)), (s4[k], w4s), (y[k], want), (f[k], want), (ct[k], orc.pack(w4[:m * 32], 4)),
                         (st[k], orc.tile_scales(w4s[:m].reshape(rows[k], kb[k]), rows[k], kb[k]))):
            assert bits_equal(to_host(got.view), exp), (k, nblks[k], first_diff(to_host(got.view), exp))
