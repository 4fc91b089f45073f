"""The dispatcher's segment-by-segment gather (banks beyond the L2 whose rows
are scored many times): pass bytes against the one-launch filter for every
kind of candidate list it may meet - ascending, with repeats, unordered, with
invalid bins, empty, across and within segments - and against the oracle for
sampled reads; data flags as the one-launch filter raises them."""
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


def workload(n_bins, n_reads, per_read, seed, bin_len=16):
    rng = np.random.default_rng(seed)
    n = n_bins * bin_len - 3
    codes = synth.ref_iid(n, seed)
    reads, lists = [], []
    for r in range(n_reads):
        L = int(rng.integers(30, 160)) if r % 9 else int(rng.integers(0, 12))
        s = int(rng.integers(0, n - 200))
        x = codes[s:s + L].copy()
        if r % 10 == 3 and L > 40:
            x[20:30] = x[5:15]       # repeated tokens
        if r % 50 == 7:
            x = np.zeros(L, np.uint8)  # one token, many times: more than two planes
        reads.append(x)
        k = per_read if r % 17 else r % 3
        c = np.sort(rng.integers(0, n_bins, k)).astype(np.uint32)
        if k and r % 5 == 0:
            c[k // 2:] = c[k // 2]                           # repeats
        if k and r % 11 == 4:
            c[:] = np.sort(rng.integers(n_bins - 50, n_bins, k))  # all in the last segment
        if k and r % 23 == 8:
            rng.shuffle(c)                                   # unordered
        if k:
            c[np.searchsorted(c, s // bin_len) % k] = s // bin_len if r % 2 else c[0]
            if r % 23 != 8:
                c.sort()
        lists.append(c)
    off = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.int64)
    co = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    E = rng.integers(0, 8, n_reads).astype(np.uint16)
    return codes, np.concatenate(reads), off, np.concatenate(lists), co, E


@pytest.mark.parametrize("n_bins,n_reads,per_read", [
    (2_097_152, 4_200, 16_000), (2_097_153, 33_001, 2_050), (3_000_000, 16_000, 4_400)])
def test_segments_match_the_one_launch_filter(oracle, n_bins, n_reads, per_read):
    codes, bases, off, cb, co, E = workload(n_bins, n_reads, per_read, n_reads)
    packed = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(packed), len(codes), 5, 16, 150)
    assert bank.n_bins == n_bins
    # as the segment form asks: a bank beyond the L2, 8 GB of rows in all
    assert len(cb) * 128 >= 8e9 and n_bins * 128 >= 256e6
    args = (bank, dev(bases), dev(off), dev(cb), dev(co), dev(E))
    want = host(grim.grim_filter(*args), np.uint8)
    got, scanned = grim.grim_filter_auto(*args)
    assert scanned == 0 and np.array_equal(host(got, np.uint8), want)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    for r in np.random.default_rng(1).choice(n_reads, 12, replace=False):
        c = cb[co[r]:co[r + 1]][:200]
        o = np.array([0, off[r + 1] - off[r]], np.int64)
        p, _ = oracle.filter_rows(packed, len(codes), 5, 16, 150, bases[off[r]:off[r + 1]], o, c,
                                  np.array([0, len(c)], np.int64), E[r:r + 1])
        assert np.array_equal(want[co[r]:co[r] + len(c)], p)
    # bad data: the same bytes and the same flags
    bad = cb.copy()
    bad[co[5]:co[5] + 1] = n_bins
    bb = bases.copy()
    bb[off[2]] = 7
    args = (bank, dev(bb), dev(off), dev(bad), dev(co), dev(E))
    want = host(grim.grim_filter(*args), np.uint8)
    flags = grim.grim_bank_status(bank)
    assert flags[1] != 0
    got, _ = grim.grim_filter_auto(*args)
    assert np.array_equal(host(got, np.uint8), want)
    assert grim.grim_bank_status(bank) == flags
    bank.free()
