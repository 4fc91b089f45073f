"""grim_verify where the addition's carry runs through many words: spans that
are one base or a short period for hundreds of rows, broken at, before and
after the words at which the sum passes from one group of words to the next,
for every word count the kernel is built for."""
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


@pytest.mark.parametrize("words", [8, 10, 12, 13, 15, 18, 21, 26, 32])
def test_carries_across_word_groups(oracle, words):
    rng = np.random.default_rng(words)
    span = 32 * words
    bin_len, n_bins = span - 64, 12     # overlap 64: the span fills every word
    n = n_bins * bin_len + 64
    codes = np.zeros(n, np.uint8)
    for b in range(n_bins):
        s = codes[b * bin_len:(b + 1) * bin_len]
        if b % 4 == 1:
            s[:] = np.resize([0, 1], len(s))
        if b % 4 == 2:
            s[:] = np.resize([2, 2, 3], len(s))
        for w in rng.choice(words, 3, replace=False):  # a break near a word's edge
            at = 32 * int(w) + int(rng.integers(-2, 3))
            if 0 <= at < len(s):
                s[at] = 3 if b % 4 != 2 else 0
    reads, lr, lb = [], [], []
    for i in range(30):
        L = int(rng.integers(1, 512)) if i % 3 else min(512, span)
        r = np.resize([[0], [0, 1], [2, 2, 3], [0, 0, 0, 3]][i % 4], L).astype(np.uint8)
        for _ in range(i % 5):
            r[int(rng.integers(0, L))] = rng.integers(0, 5)
        reads.append(r)
        for b in range(n_bins):
            lr.append(i)
            lb.append(b)
    off = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.int64)
    bases = np.concatenate(reads)
    packed = dev(synth.pack2bit(codes))
    bank = grim.grim_build_bank(packed, n, 5, bin_len, 64)
    d = host(grim.grim_verify(bank, packed, dev(bases), dev(off), dev(np.array(lr, np.uint32)),
                              dev(np.array(lb, np.uint32))), np.uint16)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    want = [oracle.sellers(reads[r], codes[b * bin_len:min(n, (b + 1) * bin_len + 64)]) for r, b in zip(lr, lb)]
    assert d.tolist() == want
    bank.free()
