"""The corners of the dispatcher's segment-by-segment gather: reads of three and
four count planes, more of them than their planes have room for, reads the
form leaves to the direct kernel (five planes, no tokens, over the length
limit, decreasing offsets, codes that are no bases), and more than 2^20 reads,
whose second round reuses the first one's memory.  Every byte and flag against
the one-launch filter, and samples against the oracle."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu

N_BINS, BIN_LEN = 2_097_152, 16


@pytest.fixture(scope="module")
def bank():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    codes = synth.ref_iid(N_BINS * BIN_LEN, 77)
    packed = synth.pack2bit(codes)
    b = grim.grim_build_bank(dev(packed), len(codes), 5, BIN_LEN, 150)
    yield b, codes, packed
    b.free()


def by_segment(args):
    """Whether the call makes the segment form's fourth launch (the other forms make two)."""
    grim.grim_fault_inject(grim.GRIM_FAULT_LAUNCH, 4)
    try:
        grim.grim_filter_auto(*args)
    except grim.GrimError as e:
        assert e.status == grim.GRIM_ECUDA
        return True
    finally:
        grim.grim_fault_inject(grim.GRIM_FAULT_NONE, 0)
    return False


def test_planes_and_reads_of_every_kind(oracle, bank):
    b, codes, packed = bank
    rng = np.random.default_rng(9)
    n, per_read = 16_000, 4_000
    reads = []
    for r in range(n):
        s = int(rng.integers(0, len(codes) - 200))
        kind = r % 8
        if kind in (0, 1):                              # counts 4-7: three planes
            x = np.concatenate([np.full(8 + r % 4, r % 4), codes[s:s + 60]])
        elif kind in (2, 3):                            # 8-15: four
            x = np.concatenate([codes[s:s + 50], np.full(12 + r % 8, (r // 8) % 4)])
        elif kind == 4:
            x = codes[s:s + 100]
        elif kind == 5:
            x = codes[s:s + 6 + r % 4]                  # one plane
        elif kind == 6:
            x = np.full(25 + r % 9, 1) if r % 16 == 6 else codes[s:s + r % 5]  # five planes; no token
        else:
            x = codes[s:s + 150].copy()
            if r % 80 == 7:
                x[r % 150] = 4                          # not a base
        reads.append(x.astype(np.uint8))
    reads[1000] = synth.ref_iid(65_536, 1)
    reads[2001] = synth.ref_iid(65_535, 2)
    off = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.int64)
    for r in (3000, 3004):
        off[r + 1] = off[r] - 20                        # decreasing: the next read is longer for it
    cb = np.sort(rng.integers(0, N_BINS, (n, per_read), dtype=np.uint32), axis=1).reshape(-1)
    cb[5 * per_read + 17] = N_BINS + 5                  # no bin
    co = np.arange(n + 1, dtype=np.int64) * per_read
    E = rng.integers(0, 6, n).astype(np.uint16)
    bases = np.concatenate(reads)
    args = (b, dev(bases), dev(off), dev(cb), dev(co), dev(E))
    want = grim.grim_filter(*args)
    flags = grim.grim_bank_status(b)
    assert flags[1] == (grim.GRIM_FLAG_BAD_BASE | grim.GRIM_FLAG_BAD_BIN | grim.GRIM_FLAG_BAD_OFFSETS |
                        grim.GRIM_FLAG_LONG_READ)
    got, scanned = grim.grim_filter_auto(*args)
    assert scanned == 0 and torch.equal(got, want)
    assert grim.grim_bank_status(b) == flags
    assert by_segment(args)
    torch.cuda.synchronize()
    grim.grim_bank_status(b)
    p = host(want, np.uint8)
    for r in list(range(16, 32)) + [2001]:
        c = cb[co[r]:co[r] + 60]
        o = np.array([0, off[r + 1] - off[r]], np.int64)
        o_p, _ = oracle.filter_rows(packed, len(codes), 5, BIN_LEN, 150, bases[off[r]:off[r + 1]], o, c,
                                    np.array([0, len(c)], np.int64), E[r:r + 1])
        assert np.array_equal(p[co[r]:co[r] + 60], o_p), r


def test_two_rounds_of_reads(bank):
    b, codes, _ = bank
    n, per_read = (1 << 20) + 7, 80
    rng = np.random.default_rng(4)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    lens = rng.integers(20, 60, n)
    starts = rng.integers(0, len(codes) - 60, n)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    at = np.repeat(starts - off[:-1], lens) + np.arange(off[-1])
    bases = codes[at].astype(np.uint8)
    for r in range(0, n, 11):                            # three planes and more, in both rounds
        bases[off[r]:off[r] + 9 + r % 12] = 2
    cb = torch.randint(0, N_BINS, (n, per_read), dtype=torch.int32, device="cuda", generator=g).sort(1).values.view(-1)
    true = torch.from_numpy(np.clip(starts // BIN_LEN, 0, N_BINS - 1).astype(np.int32)).cuda()
    cb.view(n, per_read)[:, 40] = true                   # near enough ascending; some pass
    co = torch.arange(n + 1, dtype=torch.int64, device="cuda") * per_read
    E = torch.full((n,), 1, dtype=torch.int16, device="cuda")
    args = (b, dev(bases), dev(off), cb, co, E)
    want = grim.grim_filter(*args)
    got, scanned = grim.grim_filter_auto(*args)
    assert scanned == 0 and torch.equal(got, want)
    assert int(want.sum()) > n // 2
    assert grim.grim_bank_status(b) == (grim.GRIM_OK, 0)
    assert by_segment(args)
    torch.cuda.synchronize()
