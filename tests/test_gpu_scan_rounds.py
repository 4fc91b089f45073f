"""The full scan where passing pairs fill both rounds of an epilogue warp: in
every tile of reads some pairs pass in the first round's reads, on lanes that
differ from bin to bin and from read to read, and others in the second
round's, with and without room for all of them, against the oracle."""
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


@pytest.mark.parametrize("digits,per_tile", [(1, 192), (2, 96), (4, 48), (8, 24)])
@pytest.mark.parametrize("cap", [1 << 18, 1000])
def test_passes_in_both_rounds_on_differing_lanes(oracle, digits, per_tile, cap):
    rng = np.random.default_rng(digits)
    n_bins, bin_len = 391, 64           # three whole bin tiles and seven bins
    codes = synth.ref_iid(n_bins * bin_len, 5)
    run = {1: 0, 2: 14, 4: 120, 8: 700}[digits]
    # every read passes in its own few bins and in those that hold what all reads end in
    tail = rng.integers(0, 4, 20).astype(np.uint8)
    for b in rng.choice(n_bins, 60, replace=False):
        at = int(b) * bin_len + int(rng.integers(0, 40))
        codes[at:at + 20] = tail
    reads = []
    for i in range(2 * per_tile + 5):   # two whole read tiles and five reads
        s = int(rng.integers(0, n_bins)) * bin_len + int(rng.integers(0, 30))
        reads.append(np.concatenate([np.zeros(run, np.uint8), codes[s:s + 20] if i % 2 else tail]))
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    bases = np.concatenate(reads).astype(np.uint8)
    # the repeated base's tokens may be missing from a bin: the budget pays for them
    E = np.full(len(reads), (run + 4) // 5 + 1, np.uint16)
    r2 = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(r2), len(codes), 5, bin_len, 30)
    want = oracle.scan(oracle.build_bank(r2, len(codes), 5, bin_len, 30), 5, bases, off, E, 0, n_bins)
    assert len(want[0]) > 50 * per_tile
    res = grim.grim_scan(bank, dev(bases), dev(off), dev(E), cap=cap, with_read_pass=True)
    n = res.n_pairs
    assert n == len(want[0])
    assert np.array_equal(host(res.read_pass, np.uint32), np.bincount(want[0], minlength=len(reads)))
    m = min(n, cap)
    pr, pb, ps = (host(t[:m], d) for t, d in ((res.pair_read, np.uint32), (res.pair_bin, np.uint32),
                                             (res.pair_sum, np.uint16)))
    got = set(zip(pr.tolist(), pb.tolist(), ps.tolist()))
    every = set(zip(want[0].tolist(), want[1].tolist(), want[2].tolist()))
    assert len(got) == m and got <= every
    flags = grim.grim_bank_status(bank)[1]
    assert flags == (0 if m == n else grim.GRIM_FLAG_OVERFLOW)
    bank.free()
