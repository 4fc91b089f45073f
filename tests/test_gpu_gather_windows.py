"""The gather's whole windows of 32 candidates (scored without a test per step)
beside a read's last, partial one: candidate counts at the edges of windows and
of warp steps, reads with and without a folded top plane, ids out of range in
both kinds of window, against the oracle."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu

COUNTS = [1, 7, 8, 9, 31, 32, 33, 40, 63, 64, 65, 95, 96, 97, 128, 255, 256, 257, 1000]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("q", [3, 4, 5, 6])
@pytest.mark.parametrize("repeat", [1, 130])  # the one-read-per-warp kernel; the claiming one
def test_whole_and_partial_windows(oracle, q, repeat):
    rng = np.random.default_rng(q)
    codes = synth.ref_iid(60_000, 7)
    packed = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(packed), len(codes), q, 64, 150)
    k = np.array(COUNTS * repeat)
    reads = []
    for i in range(len(k)):
        L = int(rng.integers(60, 160))
        r = codes[(s := int(rng.integers(0, 59_000))):s + L].copy()
        if i % 5 == 4:
            r[L // 2:] = r[:L - L // 2]  # every token twice: a dense top plane
        reads.append(r)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    co = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
    cb = rng.integers(0, bank.n_bins, int(co[-1])).astype(np.uint32)
    E = rng.integers(0, 10, len(k)).astype(np.uint16)
    sums = torch.empty(len(cb), dtype=torch.int16, device="cuda")
    bases = np.concatenate(reads)
    args = (bank, dev(bases), dev(off), dev(cb), dev(co), dev(E))
    want_p, want_s = oracle.filter(oracle.build_bank(packed, len(codes), q, 64, 150), q, bases, off, cb, co, E)
    p = grim.grim_filter(*args, sums=sums)
    assert np.array_equal(host(p, np.uint8), want_p)
    assert np.array_equal(host(sums, np.uint16), want_s.astype(np.uint16))
    assert np.array_equal(host(grim.grim_filter_batched(*args), np.uint8), want_p)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    # an id out of range: discarded and flagged, the others as before
    bad = cb.copy()
    at = np.concatenate([co[:-1], co[1:] - 1])
    bad[at] = bank.n_bins
    want_p, want_s = want_p.copy(), want_s.copy()
    want_p[at], want_s[at] = 0, 0
    p = grim.grim_filter(*args[:3], dev(bad), *args[4:], sums=sums)
    assert np.array_equal(host(p, np.uint8), want_p)
    assert np.array_equal(host(sums, np.uint16), want_s.astype(np.uint16))
    assert grim.grim_bank_status(bank)[1] != 0
    bank.free()


@pytest.mark.parametrize("q", [1, 4, 5])
def test_long_reads_with_frequent_tokens(oracle, q):
    """Reads around 255 and 1,024 tokens, whose most frequent token occurs up to
    every time: byte counters that just hold, run over, and are not used."""
    rng = np.random.default_rng(40 + q)
    codes = synth.ref_iid(30_000, 9)
    packed = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(packed), len(codes), q, 64, 150)
    reads = []
    for n_tok in [254, 255, 256, 257, 300, 511, 512, 1023, 1024, 1025, 1300]:
        L = n_tok + q - 1
        reads.append(codes[100:100 + L].copy())
        reads.append(np.full(L, n_tok & 3, np.uint8))              # one token
        r = codes[5_000:5_000 + L].copy()
        r[:L // 2] = 3                                             # one token half the time
        reads.append(r)
        reads.append(np.tile(np.array([0, 3], np.uint8), L)[:L])   # two tokens
        r = np.full(L, 3, np.uint8)
        r[-3:] = [0, 1, 2]
        reads.append(r)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    k = np.full(len(reads), 37)
    co = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
    cb = rng.integers(0, bank.n_bins, int(co[-1])).astype(np.uint32)
    E = rng.integers(0, 60, len(reads)).astype(np.uint16)
    bases = np.concatenate(reads)
    sums = torch.empty(len(cb), dtype=torch.int16, device="cuda")
    p = grim.grim_filter(bank, dev(bases), dev(off), dev(cb), dev(co), dev(E), sums=sums)
    want_p, want_s = oracle.filter(oracle.build_bank(packed, len(codes), q, 64, 150), q, bases, off, cb, co, E)
    assert np.array_equal(host(p, np.uint8), want_p)
    assert np.array_equal(host(sums, np.uint16), want_s.astype(np.uint16))
    bank.free()
