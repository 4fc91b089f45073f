"""grim_verify with the span as the rows of the table: every word count the
kernel is built for and the spans either side of each, reads shorter and
longer than the span, odd bin starts (the 2-bit reference is then read
across word boundaries) and an unaligned reference."""
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


@pytest.mark.parametrize("bin_len,overlap,shift", [
    (1, 8, 0), (31, 0, 0), (200, 56, 0), (201, 56, 0), (256, 64, 1), (256, 65, 0), (255, 129, 0), (256, 129, 0),
    (256, 160, 2), (300, 117, 0), (317, 163, 0), (256, 225, 0), (276, 300, 3), (277, 300, 0), (512, 160, 0),
    (513, 160, 0), (500, 332, 0), (501, 332, 0), (512, 512, 0), (513, 512, 0), (1100, 200, 0)])
def test_spans_around_every_word_count(oracle, bin_len, overlap, shift):
    n = max(6000, 6 * bin_len) + 13
    codes = synth.ref_iid(n, 17 + bin_len)
    n_bins = -(-n // bin_len)
    rng = np.random.default_rng(bin_len + overlap)
    lens = [0, 1, 2, 31, 32, 33, 64, 100, 150, 255, 300, 512]
    reads, lr, lb = [], [], []
    for r in range(2 * len(lens) + 140):  # more locations than one CTA's tile
        L = lens[r % len(lens)] if r < 2 * len(lens) else int(rng.integers(20, 60))
        b = int(rng.integers(0, n_bins))
        start = min(b * bin_len + int(rng.integers(0, bin_len)), max(0, n - L))
        rd = codes[start:start + L].copy()
        rd = np.concatenate([rd, rng.integers(0, 4, L - len(rd)).astype(np.uint8)]).astype(np.uint8)
        for _ in range(int(rng.integers(0, 5)) if L else 0):
            rd[int(rng.integers(0, L))] = rng.integers(0, 5)  # a substitution or a non-base code
        reads.append(rd)
        for bb in (b, n_bins - 1):
            lr.append(r)
            lb.append(bb)
    off = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.int64)
    bases = np.concatenate(reads).astype(np.uint8)
    packed = synth.pack2bit(codes)
    r2 = dev(np.concatenate([np.zeros(shift, np.uint8), packed]))[shift:]
    bank = grim.grim_build_bank(dev(packed), n, 5, bin_len, overlap)
    d = host(grim.grim_verify(bank, r2, dev(bases), dev(off), dev(np.array(lr, np.uint32)),
                              dev(np.array(lb, np.uint32))), np.uint16)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    want = [oracle.sellers(bases[off[r]:off[r + 1]], codes[b * bin_len:min(n, (b + 1) * bin_len + overlap)])
            for r, b in zip(lr, lb)]
    assert d.tolist() == want
    bank.free()
