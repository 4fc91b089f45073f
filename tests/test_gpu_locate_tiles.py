"""grim_locate at the edges of its tiles of 16,384 candidates (64 a thread):
counts around them, a pass array that starts off a 16-byte boundary, empty and
full tiles, reads without candidates; against numpy."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("n", [1, 63, 64, 65, 16_383, 16_384, 16_385, 49_200, 100_001])
@pytest.mark.parametrize("shift", [0, 1, 8])
@pytest.mark.parametrize("rate", [0.0, 0.01, 1.0])
def test_locations_at_tile_edges(n, shift, rate):
    rng = np.random.default_rng(n + shift)
    codes = synth.ref_iid(50_000, 3)
    bank = grim.grim_build_bank(dev(synth.pack2bit(codes)), len(codes), 5, 100, 50)
    n_reads = max(1, n // 37)
    co = np.sort(rng.integers(0, n + 1, n_reads + 1)).astype(np.int64)  # some reads have none
    co[0], co[-1] = 0, n
    cb = rng.integers(0, bank.n_bins, n).astype(np.uint32)
    p = (rng.random(n) < rate).astype(np.uint8) * rng.integers(1, 255, n).astype(np.uint8)
    buf = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    buf[shift:shift + n] = dev(p)
    loc = grim.grim_locate(bank, dev(cb), dev(co), buf[shift:shift + n])
    at = np.flatnonzero(p)
    assert loc.n == len(at)
    assert np.array_equal(host(loc.bin, np.uint32), cb[at])
    assert np.array_equal(host(loc.read, np.uint32), np.searchsorted(co, at, side="right") - 1)
    begin = cb[at].astype(np.int64) * 100
    assert np.array_equal(host(loc.begin, np.int64), begin)
    assert np.array_equal(host(loc.end, np.int64), np.minimum(begin + 150, len(codes)))
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    bank.free()
