"""The streaming kernels at the edges of their dispatch, against the oracle: packed runs with
ragged ends and odd addresses, skips on another grid through the staged kernel, divisors at and
past the limits of the known-divisor quotient, and batch statistics of odd channel counts."""
import numpy as np
import pytest
import torch

import oracle
from oracle import train as ot
from paper_2007_06919_gb300 import aqd, synth

from gpu_util import assert_same, dev, to_device

pytestmark = pytest.mark.gpu


# rows x c: below one block of 128 codes, ragged blocks, more blocks than one grid pass takes
@pytest.mark.parametrize("bits,rows,c", [(2, 1, 32), (2, 33, 96), (3, 5, 32), (3, 77, 160), (4, 3, 32), (4, 20011, 416),
                                         (8, 1, 1), (8, 3, 5), (8, 1, 130), (8, 7, 127), (8, 1001, 33)])
@pytest.mark.parametrize("offset", [0, 1])
def test_pack_unpack_runs(bits, rows, c, offset):
    rng = np.random.default_rng(rows + c)
    raw = rng.integers(-(1 << 31), 1 << 31, size=(rows, c), dtype=np.int64).astype(np.int32)  # low bits are kept
    codes = raw & ((1 << bits) - 1)
    want = oracle.pack(codes, bits)
    buf = torch.zeros(rows * c + 1, dtype=torch.int32, device="cuda")
    src = buf[offset:offset + rows * c].view(rows, c)  # offset 1: no 16-byte reads
    src.copy_(dev(raw))
    got = aqd.pack_codes(src, bits)
    assert np.array_equal(got.cpu().numpy(), want)
    for signed in (False, True):
        back = aqd.unpack_codes(dev(want), c, bits, signed=signed).cpu().numpy()
        ref = codes - ((codes >> (bits - 1)) << bits) if signed else codes
        assert np.array_equal(back, ref)
    if bits == 8:  # an 8-bit buffer at an odd address, on either side
        out = torch.full((rows * c + 2,), 0xA5, dtype=torch.uint8, device="cuda")
        aqd.pack_codes(src, 8, out=out[1:-1])
        assert np.array_equal(out[1:-1].cpu().numpy(), want.reshape(-1))
        assert out[0] == 0xA5 and out[-1] == 0xA5
        assert np.array_equal(aqd.unpack_codes(out[1:-1].view(rows, c), c, 8).cpu().numpy(), codes)


@pytest.mark.parametrize("c", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("b_bits", [2, 4, 8])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 7, 11), (3, 37, 53)])
@pytest.mark.parametrize("grid,wide", [("up", False), ("larger", False), ("up", True)])
def test_skip_on_another_grid(c, b_bits, shape, grid, wide):
    check_skip_on_another_grid(c, b_bits, shape, grid, wide)


# maps on either side of the sizes from which the staged kernel takes them
@pytest.mark.parametrize("c,shape", [(32, (1, 83, 127)), (32, (3, 97, 131)), (32, (5, 97, 131)), (64, (1, 83, 127)),
                                     (64, (3, 97, 131)), (128, (1, 41, 127)), (128, (1, 83, 127)), (256, (1, 41, 67)),
                                     (256, (1, 83, 127))])
@pytest.mark.parametrize("b_bits", [2, 4, 8])
@pytest.mark.parametrize("grid,wide", [("up", False), ("larger", False), ("up", True)])
def test_skip_on_another_grid_of_larger_maps(c, b_bits, shape, grid, wide):
    check_skip_on_another_grid(c, b_bits, shape, grid, wide)


def check_skip_on_another_grid(c, b_bits, shape, grid, wide):
    n, h, w = shape
    rng = np.random.default_rng(c + b_bits + h)
    up = 2 if grid == "up" else 1
    bh, bw = ((h + 1) // 2 + 1, (w + 1) // 2) if up == 2 else (h + 2, w + 1)
    a = rng.integers(-30000, 30000, size=(n, h, w, c)).astype(np.int32)
    b = synth.act_codes(rng, (n, bh, bw, c), b_bits)
    m0, sh, bias = synth.requant_params(rng, 1, c, calib_std=12000.0, out_bits=4)
    cc, dd = synth.skip_params(rng, 1, c, sh)
    if wide:
        cc, dd = np.full_like(cc, 2 ** 31 - 1), np.zeros_like(dd)  # no 32-bit table: the int64 form
    at, bt = oracle.CodeTensor.from_codes(a, 32), oracle.CodeTensor.from_codes(b, b_bits)
    ref = oracle.residual_add(at, bt, cc, dd, upsample=up, scale_a=0, out_bits=4, m0=m0, shift=sh, bias=bias)
    Y = aqd.DTensor.empty(n, h, w, c, 4)
    Y.data.fill_(0xA5)
    aqd.residual_add_int(to_device(at), to_device(bt), aqd.SkipParams.from_numpy(cc, dd, up), Y,
                         rq=aqd.RequantParams.from_numpy(m0, sh, bias))
    assert_same(Y.data.cpu().numpy().reshape(ref.packed.shape), ref.packed, c, 4, f"{grid} skip")


# both sides of 2^-20 and 2^20, a divisor of all ones, one just above a power of two, and values at
# which a quotient under- or overflows
@pytest.mark.parametrize("nu", [2.0 ** -21, 2.0 ** -20, np.float32(2.0 - 2.0 ** -23), np.float32(1.0 + 2.0 ** -23), 3.0, 0.1,
                                2.0 ** 20, 2.0 ** 21, 1e30])
@pytest.mark.parametrize("weight", [False, True])
def test_fake_quant_divisors(nu, weight):
    rng = np.random.default_rng(3)
    nu = float(np.float32(nu))
    n = 400_001
    x = (rng.normal(0.0 if weight else 0.5, 0.8, size=n) * nu).astype(np.float32)
    # rounding thresholds of 4-bit codes and their neighbours
    t = ((np.arange(16) + 0.5) / 15.0 * (2.0 if weight else 1.0) - (1.0 if weight else 0.0)) * nu
    x[:16] = t.astype(np.float32)
    x[16:32] = np.nextafter(x[:16], np.float32(np.inf))
    x[32:48] = np.nextafter(x[:16], np.float32(-np.inf))
    x[48:60] = [0.0, -0.0, 1e-45, -1e-45, 1e-38, 3e-31, -3e-31, np.inf, -np.inf, 3e38, -3e38, np.nan]
    gy = rng.normal(0.1, 1.0, size=n).astype(np.float32)
    fwd, bwd = (ot.fake_quant_weight, ot.fake_quant_weight_backward) if weight else (ot.fake_quant_act, ot.fake_quant_act_backward)
    with np.errstate(all="ignore"):
        x1 = np.where(np.isnan(x), -np.float32(np.inf), x)  # a NaN counts as the lower side
        want_y, want_c = fwd(x1, nu, 4)
        want_gx, want_gnu = bwd(x1, gy, nu, 4)
    y, codes = aqd.fake_quant(dev(x), nu, 4, weight=weight)
    gx, gnu = aqd.fake_quant_backward(dev(x), dev(gy), nu, 4, weight=weight)
    assert np.array_equal(codes.cpu().numpy(), want_c)
    assert np.array_equal(y.cpu().numpy().view(np.uint32), want_y.view(np.uint32))
    assert np.array_equal(gx.cpu().numpy(), want_gx)
    # float32 over runs of 16 vectors (64 products): 64 * 2^-24 of sum|gy dy/dnu| <= sum|gy|
    assert abs(float(gnu.cpu()[0]) - want_gnu) <= 64 * 2.0 ** -24 * float(np.abs(gy.astype(np.float64)).sum())


@pytest.mark.parametrize("c,offset", [(1, 0), (4, 0), (12, 0), (30, 0), (256, 0), (256, 1), (1028, 0), (1100, 0)])
def test_bn_level_stats_channel_counts(c, offset):
    rng = np.random.default_rng(c)
    mean, sd = rng.normal(0, 1, c), rng.uniform(0.1, 3.0, c)
    pix = [1, 700, 37, 0]
    zs = [(rng.normal(0, 1, (p, c)) * sd + mean).astype(np.float32) for p in pix]
    dz = []
    for z in zs:
        buf = torch.zeros(z.size + 1, dtype=torch.float32, device="cuda")
        v = buf[offset:offset + z.size].view(z.shape)  # offset 1: no 16-byte reads
        v.copy_(dev(z))
        dz.append(v)
    m, v = (t.cpu().numpy() for t in aqd.bn_level_stats(dz))
    for l, z in enumerate(zs):
        z64 = z.astype(np.float64)
        wm = z64.mean(0) if len(z) else np.zeros(c)
        wv = z64.var(0) if len(z) else np.zeros(c)
        # sums of float32 runs of 32 shifted values: the bounds of test_gpu_train
        assert np.all(np.abs(m[l] - wm) <= 1e-6 * (np.abs(wm) + sd))
        assert np.all(np.abs(v[l] - wv) <= 1e-5 * wv + 1e-12)
