"""Locations of calls on both sides of the line between 16 and 64 candidates
a thread, and above it of dense tiles (written by warps) beside sparse ones:
pass bytes at offsets from a 16-byte boundary, reads of no candidates and of
thousands, invalid bins, and room for all locations, for some and for one."""
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


@pytest.mark.parametrize("shift", [0, 1, 8, 15])
@pytest.mark.parametrize("rate,tiles", [(0.05, -1), (0.3, 0), (0.08, 1), (0.09, 70_001), (0.3, 16_384 * 9), (0.9, 1)])
def test_dense_tiles(rate, tiles, shift):
    # the line lies at eight CTAs of 4,096 candidates per SM
    n = 8 * 4096 * torch.cuda.get_device_properties(0).multi_processor_count + tiles
    rng = np.random.default_rng(shift + n)
    codes = synth.ref_iid(50_000, 3)
    bank = grim.grim_build_bank(dev(synth.pack2bit(codes)), len(codes), 5, 100, 50)
    sizes = rng.choice([0, 0, 1, 5, 40, 3000], n // 60 + 2)
    co = np.minimum(np.concatenate([[0], np.cumsum(sizes)]), n).astype(np.int64)
    co[-1] = n
    cb = rng.integers(0, bank.n_bins, n).astype(np.uint32)
    tile_rate = np.repeat(rng.choice([rate, rate, 0.002], n // 16_384 + 1), 16_384)[:n]  # dense and sparse tiles
    p = (rng.random(n) < tile_rate).astype(np.uint8) * rng.integers(1, 255, n).astype(np.uint8)
    buf = torch.full((n + 40,), 9, dtype=torch.uint8, device="cuda")  # the neighbours pass
    buf[16 + shift:16 + shift + n] = dev(p)
    at = np.flatnonzero(p)
    begin = cb[at].astype(np.int64) * 100
    reads = np.searchsorted(co, at, side="right") - 1
    for cap in (len(at) + 5, len(at) // 2 + 1, 1):
        loc = grim.grim_locate(bank, dev(cb), dev(co), buf[16 + shift:16 + shift + n], capacity=cap)
        m = min(len(at), cap)
        assert loc.n == len(at)
        assert np.array_equal(host(loc.bin, np.uint32)[:m], cb[at][:m])
        assert np.array_equal(host(loc.read, np.uint32)[:m], reads[:m])
        assert np.array_equal(host(loc.begin, np.int64)[:m], begin[:m])
        assert np.array_equal(host(loc.end, np.int64)[:m], np.minimum(begin + 150, len(codes))[:m])
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    if len(at):
        cb[at[len(at) // 2]] = bank.n_bins
        grim.grim_locate(bank, dev(cb), dev(co), buf[16 + shift:16 + shift + n])
        assert grim.grim_bank_status(bank)[1] == grim.GRIM_FLAG_BAD_BIN
    bank.free()
