"""The conv kernel's forms at the sizes where their choice changes, byte for byte against the
oracle: slabs shared by the taps of a kernel row, the skip forms and their limits, rows of no whole 32-channel groups, column
counts that leave warps idle or let sets of warps take tiles in turn, and accumulators too
large for the common form."""
import numpy as np
import pytest
import torch

import oracle
from paper_2007_06919_gb300 import aqd, synth

from gpu_util import assert_same, conv_pair, to_device, weights

pytestmark = pytest.mark.gpu
I32 = np.iinfo(np.int32)


def tables(rng, cout, std, out_bits):
    return synth.requant_params(rng, 1, cout, calib_std=std, out_bits=out_bits)


# d at and beside the 32-bit rescale's limits: d + k >= 33 with k = 23 (8-bit codes) or 3 (int32); from 40 or 60 on the
# rescaled skip is 0. (2- to 4-bit codes take a table whatever d is, within the limit of the next test.)
@pytest.mark.parametrize("skip_bits,d_lo,d_hi", [(2, 8, 9), (2, 9, 33), (2, 34, 62), (3, 9, 36), (4, 8, 8), (4, 9, 12),
                                                 (4, 30, 40), (8, 9, 10), (8, 10, 12), (8, 30, 62), (32, 29, 33),
                                                 (32, 30, 34), (32, 55, 62)])
@pytest.mark.parametrize("ws", [False, True])
@pytest.mark.parametrize("huge", [False, True])
def test_skip_rescale_forms_bit_exact(skip_bits, d_lo, d_hi, ws, huge):
    rng = np.random.default_rng(100 * skip_bits + d_lo + 7 * ws)
    n, h, w, cin, cout = 2, 9, 21, 64, 96
    x = synth.act_codes(rng, (n, h, w, cin), 4)
    wt = synth.weight_codes(rng, (cout, 3, 3, cin), 4)
    m0, sh, b = tables(rng, cout, 3000.0, 4)
    c = rng.integers(I32.min, I32.max, size=(1, cout), dtype=np.int64, endpoint=True).astype(np.int32)
    c[0, :3] = (I32.min, I32.max, 0)
    d = rng.integers(d_lo, d_hi + 1, size=(1, cout)).astype(np.int8)
    if skip_bits == 32:
        # below 2^28 everywhere, or values beyond it in some rows (those take the general form)
        lim = 1 << 28
        skip = rng.integers(-lim + 1, lim, size=(n, h, w, cout)).astype(np.int32)
        if huge:
            skip[0, 3, 5, 7], skip[1, 8, 20, 95], skip[1, 0, 0, 0] = I32.max, I32.min, lim
    else:
        skip = synth.act_codes(rng, (n, h, w, cout), skip_bits)
        if huge:
            b = np.where(rng.random((1, cout)) < 0.5, 1 << 30, -(1 << 30)).astype(np.int32)  # the bias limit
    got, want, _ = conv_pair(x, 4, wt, 4, out_bits=4, m0=m0, shift=sh, bias=b, skip=skip, skip_bits=skip_bits, skip_c=c,
                             skip_d=d, workspace=ws)
    assert_same(got, want, cout, 4, f"skip {skip_bits} bits, d {d_lo}..{d_hi}")


# 2- to 4-bit skips: a table entry, bias + rescaled skip, at the table's limit of 2^30 and one beyond it, either sign
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("ws", [False, True])
def test_skip_table_at_the_limit_bit_exact(bits, over, sign, ws):
    rng = np.random.default_rng(bits + over)
    n, h, w, cin, cout = 1, 9, 21, 64, 96
    x = synth.act_codes(rng, (n, h, w, cin), 4)
    wt = synth.weight_codes(rng, (cout, 1, 1, cin), 4)
    skip = synth.act_codes(rng, (n, h, w, cout), bits)
    top = (1 << bits) - 1
    skip[0, 0, :3] = top
    c = np.full((1, cout), sign << 20, np.int32)
    b = np.full((1, cout), sign * ((1 << 30) + over - (top << 20)), np.int32)  # bias + top c = +-(2^30 + over)
    got, want, _ = conv_pair(x, 4, wt, 4, pad=0, out_bits=4, m0=np.full((1, cout), I32.max, np.int32),
                             shift=rng.integers(25, 29, size=(1, cout)).astype(np.int8), bias=b, skip=skip, skip_bits=bits,
                             skip_c=c, skip_d=np.zeros((1, cout), np.int8), workspace=ws)
    assert_same(got, want, cout, 4, f"{bits}-bit skip")


# int32 skips at the 32-bit form's limit of 2^28 in magnitude: the one product of the largest multiplier that a shift of
# 60 does not round to 0 is that of -2^28 itself (beside it, and at 59, both forms agree)
@pytest.mark.parametrize("s", [-(1 << 28), -(1 << 28) + 1, (1 << 28) - 1, 1 << 28])
@pytest.mark.parametrize("d", [59, 60])
@pytest.mark.parametrize("ws", [False, True])
def test_int32_skip_at_the_limit_bit_exact(s, d, ws):
    n, h, w, cin, cout = 1, 6, 21, 64, 96
    x, wt = np.zeros((n, h, w, cin), np.int32), np.ones((cout, 1, 1, cin), np.int32)
    skip = np.zeros((n, h, w, cout), np.int32)
    skip[0, 1, 5], skip[0, 4, 20, ::7] = s, s
    full = lambda v, t: np.full((1, cout), v, t)
    # a quarter of bias + rescaled skip: 2 is code 0, 3 is code 1
    got, want, _ = conv_pair(x, 4, wt, 4, pad=0, out_bits=4, m0=full(I32.max, np.int32), shift=full(2, np.int8),
                             bias=full(2, np.int32), skip=skip, skip_bits=32, skip_c=full(I32.min, np.int32),
                             skip_d=full(d, np.int8), workspace=ws)
    assert_same(got, want, cout, 4, f"skip {s}, d {d}")


# the general form: shifts below the 32-bit requant's (R = 0, 1, 31, 32), both skip directions with every d down to 0,
# every skip width, saturating biases, int32 outputs with a skip
# (8-bit operands with a skip run on CUDA cores)
@pytest.mark.parametrize("xb,wb,ws,skip_bits,scale_main",
                         [(4, 4, ws, sb, sm) for ws in (False, True) for sb in (2, 3, 4, 8, 32) for sm in (0, 1)] +
                         [(xb, wb, ws, 0, 0) for xb, wb, ws in ((4, 4, False), (4, 4, True), (8, 8, True), (4, 8, True))])
@pytest.mark.parametrize("out_bits", [2, 3, 4, 8, 32])
def test_general_form_bit_exact(xb, wb, ws, skip_bits, scale_main, out_bits):
    rng = np.random.default_rng(skip_bits + 7 * out_bits + scale_main)
    n, h, w, cin, cout = 2, 7, 19, 128, 96
    x = synth.act_codes(rng, (n, h, w, cin), xb)
    wt = synth.weight_codes(rng, (cout, 1, 1, cin), wb)
    m0 = rng.integers(1, 1 << 31, size=(1, cout), dtype=np.int64).astype(np.int32)
    sh = rng.integers(-31, 13, size=(1, cout)).astype(np.int8)
    sh[0, :4], m0[0, :4] = (-31, -30, 0, 1), (3, -5, I32.max, I32.min)
    m0[0, 4::3] >>= rng.integers(0, 31, size=m0[0, 4::3].shape)
    b = rng.integers(-3000, 3000, size=(1, cout)).astype(np.int32)
    b[0, ::9], b[0, 1::9] = I32.max, I32.min
    kw = {}
    if skip_bits:
        c = rng.integers(I32.min, I32.max, size=(1, cout), dtype=np.int64, endpoint=True).astype(np.int32)
        c[0, 3::4] >>= 24
        skip = rng.integers(I32.min, I32.max, size=(n, h, w, cout), dtype=np.int64, endpoint=True).astype(np.int32)
        skip[:, ::2] >>= 16
        d = rng.integers(0, 63, size=(1, cout)).astype(np.int8)
        skip[0, 2, :, :2], c[0, :2], d[0, :2] = I32.min, I32.min, (0, 62)  # the largest product, 2^62
        kw = dict(skip=skip if skip_bits == 32 else synth.act_codes(rng, (n, h, w, cout), skip_bits), skip_bits=skip_bits,
                  skip_c=c, skip_d=d, scale_main=scale_main)
    got, want, _ = conv_pair(x, xb, wt, wb, pad=0, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                             shift=None if out_bits == 32 else sh, bias=b, workspace=ws, **kw)
    assert_same(got, want, cout, out_bits, f"skip {skip_bits}, out {out_bits}, scale_main {scale_main}")


@pytest.mark.parametrize("out_bits,cout", [(8, 1), (8, 40), (8, 48), (8, 272), (8, 96), (32, 33), (32, 84), (32, 20),
                                           (32, 258)])
@pytest.mark.parametrize("skip", [False, True])
@pytest.mark.parametrize("ws", [False, True])
def test_rows_of_no_whole_groups_bit_exact(out_bits, cout, skip, ws):
    rng = np.random.default_rng(cout)
    n, h, w, cin = 1, 11, 27, 64
    x = synth.act_codes(rng, (n, h, w, cin), 4)
    wt = synth.weight_codes(rng, (cout, 3, 3, cin), 4)
    m0, sh, b = tables(rng, cout, 600.0, min(out_bits, 8))
    kw = {}
    if skip:
        kw = dict(skip=synth.act_codes(rng, (n, h, w, cout), 8), skip_bits=8,
                  skip_c=rng.integers(-(1 << 30), 1 << 30, size=(1, cout)).astype(np.int32),
                  skip_d=rng.integers(10, 30, size=(1, cout)).astype(np.int8))
    got, want, _ = conv_pair(x, 4, wt, 4, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                             shift=None if out_bits == 32 else sh, bias=b, workspace=ws, **kw)
    assert_same(got, want, cout, out_bits, f"cout {cout}")


# several tiles per CTA pair; 1, 2, 3, 4 and 8 column groups, and two N tiles
@pytest.mark.parametrize("cout", [32, 64, 96, 128, 256, 320])
@pytest.mark.parametrize("out_bits", [2, 3, 4])
@pytest.mark.parametrize("skip", [False, True])
def test_column_groups_over_many_tiles_bit_exact(cout, out_bits, skip):
    rng = np.random.default_rng(cout + out_bits)
    n, h, w, cin = 3, 150, 179, 64
    x = synth.act_codes(rng, (n, h, w, cin), 3)
    wt = synth.weight_codes(rng, (cout, 1, 1, cin), 3)
    m0, sh, b = tables(rng, cout, 80.0, out_bits)
    sh = np.maximum(sh, 2).astype(np.int8)  # R >= 33
    kw = {}
    if skip:
        c, d = synth.skip_params(rng, 1, cout, sh)
        kw = dict(skip=synth.act_codes(rng, (n, h, w, cout), out_bits), skip_bits=out_bits, skip_c=c, skip_d=d)
    got, want, _ = conv_pair(x, 3, wt, 3, pad=0, out_bits=out_bits, m0=m0, shift=sh, bias=b, workspace=True, **kw)
    assert_same(got, want, cout, out_bits, f"cout {cout}")


# int32 skips through their staging slots over many tiles per warp: the last step's copies of a tile and the first
# of the next go to the same places; 1, 2, 3 and 8 column groups, a tile's last group beside idle warps, and two N tiles
@pytest.mark.parametrize("cout", [32, 64, 96, 256, 320])
@pytest.mark.parametrize("ws", [False, True])
def test_int32_skips_over_many_tiles_bit_exact(cout, ws):
    rng = np.random.default_rng(cout + ws)
    n, h, w, cin = 3, 150, 179, 64
    x = synth.act_codes(rng, (n, h, w, cin), 3)
    wt = synth.weight_codes(rng, (cout, 1, 1, cin), 3)
    m0, sh, b = tables(rng, cout, 80.0, 4)
    c, d = synth.skip_params_acc(rng, 1, cout)
    skip = rng.integers(-4000, 4000, size=(n, h, w, cout)).astype(np.int32)
    got, want, _ = conv_pair(x, 3, wt, 3, pad=0, out_bits=4, m0=m0, shift=np.maximum(sh, 2).astype(np.int8), bias=b,
                             skip=skip, skip_bits=32, skip_c=c, skip_d=d, workspace=ws)
    assert_same(got, want, cout, 4, f"cout {cout}")


@pytest.mark.parametrize("ws", [False, True])
@pytest.mark.parametrize("out_bits", [4, 32])
def test_accumulators_beyond_the_common_form_bit_exact(ws, out_bits):
    rng = np.random.default_rng(5)
    cin, cout = 2112, 32  # K * 15 * 15 = 4.3e6 > 2^22, and sums up to that size occur
    x = np.full((1, 5, 6, cin), 15, np.int32)
    wt = np.full((cout, 3, 3, cin), 15, np.int32)  # odd grid: 2 * 15 - 15 = 15
    wt[1:] = rng.integers(0, 16, size=(cout - 1, 3, 3, cin))
    m0, sh, b = tables(rng, cout, 1e6, 4)
    got, want, _ = conv_pair(x, 4, wt, 4, w_format=1, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                             shift=None if out_bits == 32 else sh, bias=b, workspace=ws)
    assert_same(got, want, cout, out_bits)


# K below, at and past one exact segment of 512, a ragged last segment, several tiles per CTA pair,
# narrow and no-whole-group rows
@pytest.mark.parametrize("cin,k,cout,out_bits,shape", [(128, 1, 64, 8, (1, 7, 9)), (512, 1, 256, 4, (2, 31, 33)),
                                                       (128, 3, 96, 3, (1, 20, 21)), (256, 3, 84, 32, (1, 13, 21)),
                                                       (384, 3, 40, 8, (1, 9, 10)), (128, 3, 33, 32, (2, 5, 6)),
                                                       (128, 3, 320, 2, (3, 90, 101)), (256, 1, 64, 8, (4, 100, 101))])
@pytest.mark.parametrize("path", [0, 2, 3])
def test_f16_pipe_bit_exact(cin, k, cout, out_bits, shape, path):
    if path == 2 and cin * k * k * cout * np.prod(shape) > 1 << 31:
        pytest.skip("the CUDA-core kernel takes seconds")
    rng = np.random.default_rng(cin + cout)
    x = synth.act_codes(rng, (*shape, cin), 8)
    wt = rng.integers(-128, 128, size=(cout, k, k, cin)).astype(np.int32)
    x[0, 0, :, :], wt[0], wt[1] = 255, -128, 127  # the largest sums of either sign
    m0, sh, b = tables(rng, cout, 255 * 74 * np.sqrt(cin * k * k) / 2, min(out_bits, 8))
    got, want, used = conv_pair(x, 8, wt, 8, pad=k // 2, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                                shift=None if out_bits == 32 else sh, bias=b, workspace=True, path=path)
    assert used == {0: 4, 2: 2, 3: 3}[path]
    assert_same(got, want, cout, out_bits, f"F16 pipe {cin}x{k}x{k} -> {cout}")


# narrow outputs of 2 to 8 segments with four tiles or more per CTA (pair): the sets of epilogue warps that take
# tiles in turn, each tile's segments in the four accumulators in turn
@pytest.mark.parametrize("cin,kh,kw,cout,out_bits", [(1024, 1, 1, 64, 8), (128, 3, 3, 64, 4), (128, 4, 4, 64, 3), (256, 3, 3, 64, 32),
                                                     (256, 3, 3, 36, 32), (384, 3, 3, 36, 8), (640, 1, 1, 32, 2),
                                                     (128, 3, 3, 32, 4), (128, 4, 4, 16, 8), (128, 4, 8, 4, 32)])
@pytest.mark.parametrize("path", [0, 3])
def test_f16_pipe_sets_of_warps_bit_exact(cin, kh, kw, cout, out_bits, path):
    rng = np.random.default_rng(cin + kw + cout)
    x = synth.act_codes(rng, (1, 281, 289, cin), 8)
    wt = rng.integers(-128, 128, size=(cout, kh, kw, cin)).astype(np.int32)
    m0, sh, b = tables(rng, cout, 255 * 74 * np.sqrt(cin * kh * kw) / 2, min(out_bits, 8))
    got, want, used = conv_pair(x, 8, wt, 8, pad=kh // 2, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                                shift=None if out_bits == 32 else sh, bias=b, workspace=True, path=path)
    assert used == {0: 4, 3: 3}[path]
    assert_same(got, want, cout, out_bits, f"F16 pipe {kh}x{kw} {cin}->{cout}")


# the same over three levels of their own tables, which the sets rebuild together
@pytest.mark.parametrize("path", [0, 3])
def test_f16_pipe_sets_of_warps_over_levels_bit_exact(path):
    rng = np.random.default_rng(36)
    cin, cout, lv = 256, 36, [(1, 200, 203), (2, 100, 102), (3, 51, 50)]
    wt = rng.integers(-128, 128, size=(cout, 3, 3, cin)).astype(np.int32)
    b = rng.integers(-(1 << 20), 1 << 20, size=(len(lv), cout)).astype(np.int32)
    W, wp = weights(wt, 8)
    xs = [synth.act_codes(rng, (n, h, w, cin), 8) for n, h, w in lv]
    xt = [oracle.CodeTensor.from_codes(x, 8) for x in xs]
    jobs = [(to_device(x), aqd.DTensor.empty(n, h, w, cout, 32), None, l) for l, (x, (n, h, w)) in enumerate(zip(xt, lv))]
    old = aqd.set_conv_path(path)
    try:
        aqd.conv_int_grouped(jobs, W, 1, 1, rq=aqd.RequantParams.from_numpy(None, None, b),
                             workspace=aqd.workspace_for(jobs, W, 1, 1))
    finally:
        aqd.set_conv_path(old)
    assert aqd.device_status() == 0
    for l, x in enumerate(xt):
        ref = oracle.conv_int(x, wp, 8, 0, 3, 3, 1, 1, cout, level=l, bias=b, levels=len(lv), out_bits=32)
        assert_same(jobs[l][1].data.cpu().numpy().reshape(ref.packed.shape), ref.packed, cout, 32, f"level {l}")


# int32 outputs of the F16 pipe: 16-byte pieces where rows are whole ones and the biases stay within 2^30, else the
# general form (which saturates)
@pytest.mark.parametrize("cout", [4, 36, 64, 70, 256, 300])
@pytest.mark.parametrize("bias", [1 << 30, -(1 << 30), (1 << 30) + 1, I32.max, I32.min])
def test_f16_pipe_int32_outputs_bit_exact(cout, bias):
    rng = np.random.default_rng(cout)
    x = synth.act_codes(rng, (1, 19, 31, 128), 8)
    wt = rng.integers(-128, 128, size=(cout, 3, 3, 128)).astype(np.int32)
    b = rng.integers(-1000, 1000, size=(1, cout)).astype(np.int32)
    b[0, cout // 2] = bias
    got, want, used = conv_pair(x, 8, wt, 8, out_bits=32, bias=b, workspace=True)
    assert used == 4
    assert_same(got, want, cout, 32, f"bias {bias}")


# taps per slab 1, 2, 3, 5, 7 and 16, kernels too wide for one (17); resident weights with one and two
# N tiles and with two planes of an 8-bit image; weights streamed beside half-width tiles
@pytest.mark.parametrize("kh,kw,pad,cin,cout,bits", [(1, 1, 0, 128, 512, 4), (2, 2, 0, 64, 128, 3), (3, 3, 1, 64, 512, 4),
                                                     (3, 3, 1, 128, 64, 8), (3, 3, 1, 256, 256, 2), (5, 5, 2, 64, 96, 4),
                                                     (7, 7, 3, 64, 64, 2), (1, 16, 0, 64, 32, 4), (3, 17, 1, 128, 64, 4),
                                                     (1, 17, 0, 64, 288, 2), (17, 1, 0, 64, 64, 4)])
@pytest.mark.parametrize("path", [0, 3])
def test_slabs_bit_exact(kh, kw, pad, cin, cout, bits, path):
    rng = np.random.default_rng(kh * 31 + kw + cin)
    x = synth.act_codes(rng, (2, 41, 83, cin), bits)
    wb = min(bits, 4)
    wt = synth.weight_codes(rng, (cout, kh, kw, cin), wb)
    m0, sh, b = tables(rng, cout, 3.0 * (1 << bits) * np.sqrt(kh * kw * cin) / 4, 4)
    got, want, used = conv_pair(x, bits, wt, wb, pad=pad, out_bits=4, m0=m0, shift=sh, bias=b, workspace=True, path=path)
    assert used == (6 if bits == 2 and cin == 256 and cout <= 240 else 4 if path == 0 else 3)
    assert_same(got, want, cout, 4, f"{kh}x{kw} {cin}->{cout}")


# the first conv at stride 2: image rows as the operand (more than one tile per SM, strips of 128 output columns full
# enough for the channels): strips and their edges, runs of tiles that cross strips and images, more row pairs than the ring
# holds, images smaller than the kernel, wide padding
@pytest.mark.parametrize("shape,pad,cout,out_bits", [((80, 5, 77), 3, 16, 32), ((200, 1, 80), 3, 16, 32), ((90, 3, 121), 6, 32, 3),
                                                     ((24, 13, 257), 3, 32, 8), ((40, 9, 255), 3, 64, 2), ((21, 30, 307), 6, 64, 4),
                                                     ((3, 211, 399), 0, 96, 8), ((2, 45, 1279), 3, 256, 4),
                                                     ((1, 700, 313), 3, 48, 32), ((90, 7, 193), 2, 128, 4), ((30, 21, 151), 3, 64, 4),
                                                     ((30, 21, 153), 3, 64, 4)])
def test_first_conv_rows_of_many_tiles_bit_exact(shape, pad, cout, out_bits):
    test_first_conv_rows_bit_exact(shape, pad, cout, out_bits)


# the same at the sizes on either side of the line to built tiles, and small maps
@pytest.mark.parametrize("shape,pad,cout,out_bits", [((1, 7, 7), 0, 16, 8), ((1, 1, 1), 3, 64, 4), ((2, 3, 5), 6, 32, 3),
                                                     ((1, 5, 259), 3, 64, 2), ((3, 61, 255), 3, 64, 4), ((1, 9, 257), 3, 96, 32),
                                                     ((2, 211, 262), 0, 48, 8), ((1, 30, 1031), 2, 256, 4),
                                                     ((40, 37, 20), 3, 64, 4), ((2, 1200, 517), 3, 64, 4),
                                                     ((30, 21, 141), 3, 64, 4), ((30, 21, 143), 3, 64, 4)])
def test_first_conv_rows_bit_exact(shape, pad, cout, out_bits):
    rng = np.random.default_rng(shape[1] * 7 + shape[2])
    x = synth.act_codes(rng, (*shape, 3), 8)
    wt = rng.integers(-7, 8, size=(cout, 7, 7, 3)).astype(np.int32)
    m0, sh, b = tables(rng, cout, 255 * 2.6 * 12, min(out_bits, 8))
    got, want, used = conv_pair(x, 8, wt, 8, stride=2, pad=pad, out_bits=out_bits, m0=None if out_bits == 32 else m0,
                                shift=None if out_bits == 32 else sh, bias=b)
    assert used == 5
    assert_same(got, want, cout, out_bits, f"first conv {shape}")


# its int32 outputs: whole sectors or, at an address of 16 bytes, 16-byte pieces; sums or biases beyond the lean form
@pytest.mark.parametrize("stride,cout", [(1, 16), (1, 96), (2, 64), (2, 256)])
@pytest.mark.parametrize("offset", [0, 16])
@pytest.mark.parametrize("wide", ["", "weights", "bias"])
def test_first_conv_int32_outputs_bit_exact(stride, cout, offset, wide):
    rng = np.random.default_rng(stride + cout)
    x = synth.act_codes(rng, (2, 37, 141, 3), 8)
    lim = 128 if wide == "weights" else 8
    wt = rng.integers(-lim, lim, size=(cout, 7, 7, 3)).astype(np.int32)
    x[0, :9, :9], wt[0] = 255, -lim
    b = rng.integers(-1000, 1000, size=(1, cout)).astype(np.int32)
    if wide == "bias":
        b[0, 1], b[0, cout - 1] = I32.max, I32.min
    W, wp = weights(wt, 8)
    xt = oracle.CodeTensor.from_codes(x, 8)
    want = oracle.conv_int(xt, wp, 8, 0, 7, 7, stride, 3, cout, bias=b, out_bits=32)
    buf = torch.full((want.packed.size + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    y = aqd.DTensor(buf[offset:offset + want.packed.size], want.n, want.h, want.w, cout, 32)
    aqd.conv_int(to_device(xt), W, stride, 3, y, rq=aqd.RequantParams.from_numpy(None, None, b))
    assert aqd.last_conv_path() == 5 and aqd.device_status() == 0
    assert_same(y.data.cpu().numpy().reshape(want.packed.shape), want.packed, cout, 32, f"stride {stride}, {wide}")
    assert bool((buf[:offset] == 0xA5).all()) and bool((buf[offset + want.packed.size:] == 0xA5).all())


# the in-kernel unpack's two threads per row: K tails of 1 to 4 groups of 32 (whole and empty second halves), chunks
# that cross taps, chunks of one tap (cin % 128 == 0), fewer and more chunks than are held in flight
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("cin,k,stride,shape", [(32, 1, 1, (1, 9, 15)), (64, 1, 2, (1, 9, 15)), (96, 1, 1, (1, 5, 7)),
                                                (32, 3, 2, (1, 20, 21)), (160, 3, 1, (1, 6, 7)), (96, 5, 2, (1, 11, 13)),
                                                (128, 1, 2, (1, 17, 19)), (128, 3, 2, (2, 13, 15)), (384, 3, 2, (1, 9, 9))])
def test_unpack_halves_bit_exact(cin, k, stride, shape, bits):
    rng = np.random.default_rng(cin * k + bits)
    x = synth.act_codes(rng, (*shape, cin), bits)
    wt = synth.weight_codes(rng, (64, k, k, cin), bits)
    m0, sh, b = tables(rng, 64, 3.0 * (1 << bits) * np.sqrt(k * k * cin) / 4, 4)
    got, want, used = conv_pair(x, bits, wt, bits, stride=stride, pad=k // 2, out_bits=4, m0=m0, shift=sh, bias=b)
    assert used == 1
    assert_same(got, want, 64, 4, f"in-kernel unpack {cin}x{k}x{k}")


# int32 outputs of the in-kernel variant through the staging blocks: whole and partial 16- and 32-column steps, several N
# tiles, a last row group that is not whole; cout % 4 != 0 stays with the general form
@pytest.mark.parametrize("cin,k,cout,shape", [(64, 1, 4, (1, 3, 5)), (64, 1, 36, (1, 20, 21)), (32, 3, 128, (2, 13, 15)),
                                              (128, 1, 260, (1, 9, 31)), (128, 3, 516, (1, 7, 9)), (64, 1, 30, (1, 9, 9))])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_unpack_int32_outputs_bit_exact(cin, k, cout, shape, bits):
    rng = np.random.default_rng(cout + bits)
    x = synth.act_codes(rng, (*shape, cin), bits)
    wt = synth.weight_codes(rng, (cout, k, k, cin), bits)
    b = rng.integers(-(1 << 29), 1 << 29, size=(1, cout)).astype(np.int32)
    got, want, used = conv_pair(x, bits, wt, bits, stride=2, pad=k // 2, out_bits=32, m0=None, shift=None, bias=b)
    assert used == 1
    assert_same(got, want, cout, 32, f"int32 {cin}x{k}x{k} -> {cout}")
