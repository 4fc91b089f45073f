"""Seed candidates at every size of the shared-memory path: the mean votes per
read that choose each group size, reads of more votes than their group takes
(the larger groups, then the sort in scratch), more and fewer seeds than are
looked up ahead, bins of one base (many bins per bitmap cell), tandem repeats
(many votes for one bin) and caps of all sizes, against the oracle."""
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


@pytest.mark.parametrize("n,k,L,bin_len", [
    (30_000, 6, 60, 64), (100_000, 6, 100, 7), (100_000, 5, 40, 256), (100_000, 5, 55, 1), (100_000, 5, 100, 16),
    (100_000, 5, 79, 3), (100_000, 4, 60, 1), (100_000, 4, 100, 30), (200_000, 4, 100, 100), (2_000, 1, 70, 10),
    (3_000, 2, 130, 5), (700, 3, 50, 1)])
@pytest.mark.parametrize("cap", [1, 40, 5000, 100_000])
def test_candidates_of_every_group_size(oracle, n, k, L, bin_len, cap):
    rng = np.random.default_rng(n + 7 * k + L)
    codes = synth.ref_iid(n, 41 + k)
    t = n // 3
    codes[t:t + 200] = np.tile(codes[:4], 50)   # a tandem repeat
    codes[2 * t:2 * t + 200] = codes[t // 2:t // 2 + 200]
    reads = []
    for i in range(40):
        s = int(rng.integers(0, n - L)) if i % 5 else t + int(rng.integers(0, 100))
        m = L if i % 3 else int(rng.integers(0, L + 1))  # uneven lengths, some without a seed
        r = codes[s:s + m].copy()
        if i % 11 == 7 and m:
            r[int(rng.integers(0, m))] = 4
        reads.append(r)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    bases = np.concatenate(reads).astype(np.uint8)
    n_bins = -(-n // bin_len)
    want, want_off = oracle.seed_candidates(codes, k, bases, off, bin_len, n_bins, cap)
    idx = grim.grim_seed_index_build(dev(synth.pack2bit(codes)), n, k)
    cb, co = grim.grim_seed_candidates(idx, dev(bases), dev(off), bin_len, n_bins, cap)
    assert np.array_equal(co.cpu().numpy(), want_off)
    assert np.array_equal(host(cb, np.uint32), want)
    idx.free()
