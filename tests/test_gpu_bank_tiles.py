"""Bank builds at the edges of their two kernels, every row against the
oracle: bins whose length is no multiple of 16 (cores that start inside a
packed word) in the lane-per-core kernel; q = 6, unaligned references, short
and long bins in the tile-of-cores kernel, with reference ends inside a token,
a core and a tile."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, pack_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("q,bin_len,overlap,n,shift", [
    # lane per core, whole and odd words, 31 rows a warp
    (5, 255, 100, 31 * 255, 0), (5, 255, 100, 31 * 255 + 1, 0), (5, 17, 4, 31 * 17 * 4 + 3, 0),
    (4, 200, 150, 40_003, 0), (3, 31, 200, 9_973, 0), (5, 1023, 300, 70_001, 0), (1, 19, 0, 2_003, 0),
    (2, 33, 70, 5_001, 0),
    # tile of cores: 30 finished rows of 32 (q = 6, 256 + 300)
    (6, 256, 300, 30 * 256, 0), (6, 256, 300, 30 * 256 + 1, 0), (6, 256, 300, 60 * 256 - 5, 0),
    (6, 256, 5, 31 * 256 + 6, 0), (6, 255, 261, 20_001, 0), (6, 16, 256, 3_000, 0), (6, 1, 5, 77, 0),
    (6, 2000, 100, 90_011, 0), (6, 256, 300, 5, 0), (6, 7, 200, 1_001, 0),
    # references that do not start at a 4-byte boundary
    (5, 256, 100, 40_007, 1), (4, 64, 150, 9_001, 2), (1, 64, 30, 70_001, 3), (6, 300, 150, 12_345, 3),
    # overlaps shorter than a token: a core's last starts belong to no bin
    (5, 256, 0, 20_003, 0), (5, 100, 3, 9_999, 0), (6, 256, 0, 20_003, 0), (6, 255, 4, 20_003, 0), (6, 3, 0, 500, 0),
    (5, 3, 0, 500, 0), (4, 64, 2, 9_001, 1),
    # bins longer than the lane kernel's
    (5, 1025, 100, 140_003, 0), (3, 20_000, 150, 70_000, 0), (5, 8, 300, 3_001, 0)])
def test_bank_at_kernel_edges(oracle, q, bin_len, overlap, n, shift):
    codes = synth.ref_iid(n, 31 * q + bin_len)
    packed = synth.pack2bit(codes)
    r2 = dev(np.concatenate([np.zeros(shift, np.uint8), packed]))[shift:]
    bank = grim.grim_build_bank(r2, n, q, bin_len, overlap)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    want = pack_rows(oracle.build_bank(packed, n, q, bin_len, overlap), bank.row_words)
    assert np.array_equal(bank.bits().cpu().numpy().view(np.uint32), want)
    bank.bits().fill_(-1)  # and again over rows that hold something
    grim.grim_build_bank_into(bank, r2)
    assert np.array_equal(bank.bits().cpu().numpy().view(np.uint32), want)
    bank.free()
