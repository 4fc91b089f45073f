"""The full scan at the edges of its read tiles: 192 digit rows a tile, that
is 192, 96, 48 and 24 reads of 1, 2, 4 and 8 base-4 digits, one read fewer and
one more than a tile of each class, against the oracle; and bin windows of
one more and one fewer than a tile of 128 bins."""
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


@pytest.mark.parametrize("counts,window", [
    ((191, 0, 0, 0), 127), ((192, 0, 0, 0), 128), ((193, 0, 0, 0), 129), ((1, 95, 0, 0), 256),
    ((0, 97, 0, 0), 257), ((0, 0, 47, 1), 130), ((0, 0, 49, 0), 300), ((0, 0, 0, 23), 300),
    ((2, 1, 1, 25), 300), ((385, 193, 97, 49), 300)])
def test_scan_tiles_of_every_class(oracle, counts, window):
    rng = np.random.default_rng(sum(counts) + window)
    codes = synth.ref_iid(300 * 64, 29)
    codes[2000:2700] = 0                      # runs that the repetitive reads pass in
    codes[9000:9400] = np.tile([0, 1], 200)
    reads = []
    for cls, n in enumerate(counts):
        for i in range(n):
            if cls == 0:
                s = int(rng.integers(0, len(codes) - 120))
                r = codes[s:s + 100].copy() if s < 1800 or s > 9500 else rng.integers(0, 4, 90).astype(np.uint8)
            else:
                run = [0, 14, 120, 700][cls]  # token counts of 4-15, 16-255 and more
                r = np.concatenate([np.zeros(run, np.uint8) if i % 3 else np.tile([0, 1], run).astype(np.uint8),
                                    rng.integers(0, 4, 20).astype(np.uint8)])
            reads.append(r.astype(np.uint8))
    order = rng.permutation(len(reads))
    reads = [reads[i] for i in order]
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    bases = np.concatenate(reads)
    E = rng.integers(0, 9, len(reads)).astype(np.uint16)
    r2 = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(r2), len(codes), 5, 64, 800)
    res = grim.grim_scan(bank, dev(bases), dev(off), dev(E), 0, window, cap=1 << 18, with_read_pass=True)
    n = res.n_pairs
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    want = oracle.scan(oracle.build_bank(r2, len(codes), 5, 64, 800), 5, bases, off, E, 0, window)
    pr, pb, ps = (host(t[:n], d) for t, d in ((res.pair_read, np.uint32), (res.pair_bin, np.uint32),
                                             (res.pair_sum, np.uint16)))
    o = np.lexsort((pb, pr))
    assert n == len(want[0])
    assert np.array_equal(pr[o], want[0]) and np.array_equal(pb[o], want[1])
    assert np.array_equal(ps[o], want[2].astype(np.uint16))
    bank.free()
