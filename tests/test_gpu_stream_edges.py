"""The streaming kernels at the edges of their dispatch, against the oracle."""
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
