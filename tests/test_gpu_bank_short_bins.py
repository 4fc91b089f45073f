"""Bank builds of short bins with long overlaps, on both sides of the lines
between the lane kernel, the tile of cores and the walk of a run's token
starts: runs of exactly as many bins as a CTA holds (128 at q = 5, 32 at q =
6), one more and one fewer, spans that reach past the reference's end, and a
reference that does not start at a 4-byte boundary, against the oracle."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, host, pack_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("q,bin_len,overlap", [
    (5, 8, 30), (5, 8, 250), (5, 12, 30), (5, 12, 60), (5, 1, 10), (5, 2, 20), (5, 15, 100), (5, 17, 30), (5, 17, 250),
    (5, 33, 500), (5, 24, 100), (4, 4, 50), (4, 8, 100), (3, 4, 50), (2, 1, 40), (1, 1, 7), (6, 8, 100), (6, 8, 700),
    (6, 32, 100), (6, 32, 300), (6, 64, 900), (6, 64, 100), (5, 9, 120_000), (6, 30, 200_000)])
@pytest.mark.parametrize("bins,shift", [(127, 0), (128, 0), (129, 1), (33, 3), (32, 0), (1, 0)])
def test_short_bins(oracle, q, bin_len, overlap, bins, shift):
    n = max(1, bins * bin_len - (bins % 3 if bin_len > 3 else 0))
    codes = synth.ref_iid(n, 31 * q + bin_len)
    packed = synth.pack2bit(codes)
    r2 = dev(np.concatenate([np.zeros(shift, np.uint8), packed]))[shift:]
    bank = grim.grim_build_bank(r2, n, q, bin_len, overlap)
    assert bank.n_bins == bins and grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    want = pack_rows(oracle.build_bank(packed, n, q, bin_len, overlap), bank.row_words)
    assert np.array_equal(host(bank.bits(), np.uint32), want)
    bank.bits().fill_(-1)  # and again over rows that hold something
    grim.grim_build_bank_into(bank, r2)
    assert np.array_equal(host(bank.bits(), np.uint32), want)
    bank.free()
