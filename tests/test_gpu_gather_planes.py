"""The gather's folded top plane: reads whose repeated tokens do and do not
share bit positions within the words a lane folds together (counts 2-3, 4-7
and 8, one to four planes), at batch sizes of the one-read-per-warp kernel and
of the claiming one, against the oracle."""
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


def reads_with_repeats(rng, n, q):
    out = []
    for i in range(n):
        L = int(rng.integers(q, 200)) if i % 4 else int(rng.integers(250, 420))
        r = rng.integers(0, 4, L).astype(np.uint8)
        for _ in range(i % 7):  # copy q-grams around: tokens of counts 2 and more
            a, b = int(rng.integers(0, L - q + 1)), int(rng.integers(0, L - q + 1))
            r[b:b + q] = r[a:a + q].copy()
        if i % 6 == 5:  # the same low five token bits (bit position), other words
            g = r[:q].copy()
            for k in range(0, L - 2 * q, 2 * q):
                r[k:k + q] = g
                r[k] = (g[0] + k // q) & 3
        if i % 13 == 12:
            r[:] = np.tile(r[:3], L // 3 + 1)[:L]
        out.append(r)
    return out


@pytest.mark.parametrize("q", [4, 5, 6])
@pytest.mark.parametrize("n_reads", [1, 37, 700, 4000])
def test_folded_planes(oracle, q, n_reads):
    rng = np.random.default_rng(100 * q + n_reads)
    codes = synth.ref_with_repeats(120_000, 3 + q, 0.3, n_fam=10, fam_min=100, fam_max=900)
    reads = reads_with_repeats(rng, n_reads, q)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    bases = np.concatenate(reads)
    r2 = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(r2), len(codes), q, 200, 300)
    k = rng.integers(0, 75, n_reads)
    co = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
    cb = rng.integers(0, bank.n_bins, int(co[-1])).astype(np.uint32)
    E = rng.integers(0, 12, n_reads).astype(np.uint16)
    sums = torch.empty(len(cb), dtype=torch.int16, device="cuda")
    args = (bank, dev(bases), dev(off), dev(cb), dev(co), dev(E))
    p = grim.grim_filter(*args, sums=sums)
    want_p, want_s = oracle.filter(oracle.build_bank(r2, len(codes), q, 200, 300), q, bases, off, cb, co, E)
    assert np.array_equal(host(p, np.uint8), want_p)
    assert np.array_equal(host(sums, np.uint16), want_s.astype(np.uint16))
    assert np.array_equal(host(grim.grim_filter_batched(*args), np.uint8), want_p)
    assert np.array_equal(host(grim.grim_filter_auto(*args)[0], np.uint8), want_p)
    assert grim.grim_bank_status(bank) == (grim.GRIM_OK, 0)
    bank.free()
