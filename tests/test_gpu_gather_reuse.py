"""The gather where every warp takes several reads one after another (more
than 16 reads per SM): reads whose counts leave every part of the warp's plane
area behind - bytes, bytes that ran over, carry chains of many planes, one
plane, none, invalid ones - in front of each other, with lists of every length
around a window and around the line of the short lists at q = 6; and the work
counter between the launches of a captured and replayed graph."""
import numpy as np
import pytest
import torch

import paper_1711_01177_gb300 as grim
import synth
from gpu_util import dev, host

pytestmark = pytest.mark.gpu

KINDS = 13


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grim.build()
    grim.load()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def read_of(kind, rng, codes, q):
    s = int(rng.integers(0, len(codes) - 6000))
    if kind == 0:
        return codes[s:s + 40]
    if kind in (1, 2):
        return np.zeros((300, 262)[kind - 1], np.uint8)             # one token, more than 255 times
    if kind in (3, 4, 5):
        return codes[s:s + (900, 1500, 5000)[kind - 3]]              # to and beyond the counted lengths
    if kind == 6:
        return np.zeros(4000, np.uint8)                              # 12 planes
    if kind == 7:
        return codes[s:s + q - 1]                                    # no token
    if kind == 8:
        return np.concatenate([codes[s:s + 150], codes[s + 20:s + 60]])
    if kind == 9:
        return np.concatenate([codes[s:s + 30]] * 5)                 # three planes
    if kind == 10:
        return np.concatenate([codes[s:s + 700], np.zeros(290, np.uint8)])
    if kind == 11:
        r = codes[s:s + 400].copy()
        r[int(rng.integers(0, 400))] = 4 + int(rng.integers(0, 4))   # not a base
        return r
    return codes[s:s + int(rng.integers(q, 60))]


def workload(q, seed):
    """Every kind of read after every other, twice (the second time in another order)."""
    rng = np.random.default_rng(seed)
    codes = synth.ref_with_repeats(60_000, 3 + q, 0.3, n_fam=10, fam_min=100, fam_max=900)
    kinds = [k for a in range(KINDS) for b in range(KINDS) for k in (a, b)]
    kinds += list(rng.permutation(kinds))
    reads = [np.asarray(read_of(k, rng, codes, q), np.uint8) for k in kinds]
    sizes = rng.permutation(np.resize([0, 1, 7, 31, 32, 33, 63, 64, 65, 95, 96, 97, 128, 161], len(reads)))
    return codes, kinds, reads, sizes, rng


def tiled(x, copies):
    return np.concatenate([[0], np.cumsum(np.tile(np.diff(x), copies))]).astype(np.int64)


@pytest.mark.parametrize("q", [3, 4, 5, 6])
def test_reads_of_every_kind_after_each_other(oracle, q):
    codes, kinds, reads, sizes, rng = workload(q, q)
    n = len(reads)
    off = np.concatenate([[0], np.cumsum([len(r) for r in reads])]).astype(np.int64)
    co = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    bases = np.concatenate(reads)
    r2 = synth.pack2bit(codes)
    bank = grim.grim_build_bank(dev(r2), len(codes), q, 200, 300)
    cb = rng.integers(0, bank.n_bins, int(co[-1])).astype(np.uint32)
    E = rng.integers(0, 12, n).astype(np.uint16)
    want, sums = oracle.filter(oracle.build_bank(r2, len(codes), q, 200, 300), q, np.where(bases > 3, 0, bases), off,
                               cb, co, E)
    rejected = np.repeat(np.array([(r > 3).any() for r in reads]), sizes)
    want, sums = np.where(rejected, 0, want).astype(np.uint8), np.where(rejected, 0, sums).astype(np.uint16)
    # as many copies as give each of the GPU's warps (at most 32 an SM) several reads
    copies = -(-100 * torch.cuda.get_device_properties(0).multi_processor_count // n)
    big = (bank, dev(bases).repeat(copies), dev(tiled(off, copies)), dev(cb).repeat(copies),
           dev(tiled(co, copies)), dev(E).repeat(copies))
    got_s = torch.full((copies * len(cb),), -1, dtype=torch.int16, device="cuda")
    p = grim.grim_filter(*big, sums=got_s)
    assert np.array_equal(host(p, np.uint8).reshape(copies, -1), np.tile(want, (copies, 1)))
    assert np.array_equal(host(got_s, np.uint16).reshape(copies, -1), np.tile(sums, (copies, 1)))
    assert grim.grim_bank_status(bank)[1] == grim.GRIM_FLAG_BAD_BASE
    stream = torch.cuda.Stream()
    for shape in (dict(), dict(warps_per_cta=4, reads_per_claim=16), dict(batch_reads=n * (copies // 3) + 5, use_graph=1)):
        t = grim.GrimTune()
        for k, v in shape.items():
            setattr(t, k, v)
        out = torch.full_like(p, 7)
        for _ in range(3):  # a graph: first captured, then replayed
            out.fill_(7)
            stream.wait_stream(torch.cuda.current_stream())
            grim.grim_filter_batched(*big, pass_out=out, tune=t, stream=stream)
            stream.synchronize()
            assert torch.equal(out, p), shape
    assert grim.grim_bank_status(bank, stream)[1] == grim.GRIM_FLAG_BAD_BASE
    bank.free()


def test_replayed_graph_of_counted_batches_reads_current_inputs(oracle):
    w = synth.batched_varlen(ref_len=300_000, n_reads=500, q=5, k_max=60)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    copies = -(-70 * sms // 500)
    bank = grim.grim_build_bank(dev(w.ref2bit), w.ref_len, w.q, w.bin_len, w.overlap)
    ob = oracle.build_bank(w.ref2bit, w.ref_len, w.q, w.bin_len, w.overlap)
    args = [dev(w.bases).repeat(copies), dev(tiled(w.read_offsets, copies)), dev(w.cand_bins).repeat(copies),
            dev(tiled(w.cand_offsets, copies)), dev(w.E).repeat(copies)]
    out = torch.empty(copies * w.n_checks, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    t = grim.GrimTune()
    t.use_graph, t.batch_reads = 1, 20 * sms + 3  # every batch above 16 reads per SM, but for the last
    for step in range(4):
        E = (w.E + step).astype(np.uint16)
        args[4].copy_(dev(E).repeat(copies))  # the same buffer: the replayed graph must see it
        torch.cuda.synchronize()
        grim.grim_filter_batched(bank, *args, pass_out=out, tune=t, stream=stream)
        stream.synchronize()
        want, _ = oracle.filter(ob, w.q, w.bases, w.read_offsets, w.cand_bins, w.cand_offsets, E)
        assert np.array_equal(host(out, np.uint8).reshape(copies, -1), np.tile(want, (copies, 1))), step
    assert grim.grim_bank_status(bank, stream) == (grim.GRIM_OK, 0)
    bank.free()
