"""Seed candidates of batches on both sides of every line in the batch's size
and mean votes: the groups' first kernel for each mean, the larger groups and
the sort in scratch for what each leaves, seeds looked up ahead and by the
groups, reads of more seeds than most groups take, with caps that bind and
that do not, against the oracle (176 reads, repeated to the batch's size)."""
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


# reference length, k, length of most reads, lengths of the others, bases per bin
WORKLOADS = [
    (20_000, 5, 20, (75, 400), 7),               # mean votes 100; the longer reads' 400 and 1,600
    (100_000, 6, 60, (300, 1500), 64),           # 340; 1,200 and 6,300
    (100_000, 5, 25, (320, 500, 1000), 16),      # 730; 6,300, 9,800, 22,200
    (100_000, 5, 45, (200, 330, 640), 3),        # 1,050; 4,000, 6,300, 15,500
    (100_000, 5, 75, (250, 400, 1500), 256),     # 1,800; 4,900, 8,200, 31,800
    (200_000, 4, 24, (30, 60, 68), 100),         # 4,800; 5,500, 11,800, 13,800
    (30_000, 6, 500, (380, 390, 2400), 20),      # 740, of 83 seeds; 63, 65 and 400 seeds
    (5_000, 6, 2000, (100, 9300, 19_000), 1),    # 2,900, of 333 seeds; 1,550 and 3,166 seeds
]


@pytest.mark.parametrize("per_sm", [0, 15, 33, 205])
@pytest.mark.parametrize("work", range(len(WORKLOADS)))
@pytest.mark.parametrize("cap", [30, 100_000])
def test_candidates_of_every_batch_size(oracle, per_sm, work, cap):
    n, k, L, longer, bin_len = WORKLOADS[work]
    rng = np.random.default_rng(work)
    codes = synth.ref_iid(n, 60 + work)
    codes[n // 2:n // 2 + 300] = np.tile(codes[:6], 50)  # a tandem repeat: votes that pile up
    reads = []
    for i in range(176):
        m = L if i % 44 != 6 else longer[(i // 44) % len(longer)]
        s = int(rng.integers(0, max(1, n - m))) if i % 7 else n // 2
        r = np.resize(codes[s:s + m], m).copy()
        if i % 9 == 5:
            r[int(rng.integers(0, m))] = 4  # not a base: that seed has no location
        reads.append(r)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    n_bins = -(-n // bin_len)
    want, want_off = oracle.seed_candidates(codes, k, np.concatenate(reads), off, bin_len, n_bins, cap)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = max(1, -(-per_sm * sms // 176))
    lens, kept = np.tile(np.diff(off), copies), np.tile(np.diff(want_off), copies)
    big_off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    idx = grim.grim_seed_index_build(dev(synth.pack2bit(codes)), n, k)
    bases = dev(np.concatenate(reads).astype(np.uint8)).repeat(copies)
    cb, co = grim.grim_seed_candidates(idx, bases, dev(big_off), bin_len, n_bins, cap)
    assert np.array_equal(co.cpu().numpy(), np.concatenate([[0], np.cumsum(kept)]))
    cb = cb.view(copies, len(want))
    assert bool((cb == cb[0]).all()) and np.array_equal(host(cb[0].clone(), np.uint32), want)
    idx.free()
