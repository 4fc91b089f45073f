"""What the performance of this library is measured on.

Every case is one call (or one short chain of calls) that a read mapper built
on the library makes, with inputs drawn on the GPU from a seed:

- references are i.i.d. ACGT with planted repeat families (300-6,000 bases
  long, copies diverged by 5-20%), 2-bit packed;
- reads start at uniform positions and carry substitutions and single-base
  insertions and deletions;
- candidate lists ascend, as a seed table yields them: either the bins of the
  reads' exact 12-mer hits, or the true bin among uniform ones.
"""
import ctypes
import math

import torch

import paper_1711_01177_gb300 as grim

SEED_K = 12      # the mapper's seed length
SLOT = 6144      # at most one repeat copy per slot of this many bases
N_FAM = 200
FAM_MIN, FAM_MAX = 300, 6000
SCAN_CAP = 1 << 22  # passing pairs a scan has room for


def listed():
    """The cases, named by what they are."""
    return [
        # A mapper's smallest call: a thousand short reads against a bacterial-size
        # reference, 32 candidates each.  Launch and latency count.
        dict(name="filter_small", kind="filter", entry="filter", ref_len=1_000_000, repeats=0.0, q=5, bin_len=256,
             overlap=100, n_reads=1_000, lmin=100, lmax=100, cands="random", k_fixed=32, k_max=0),
        # The ordinary call: a million 150-base reads with the bins of their seed hits,
        # the bank in the L2.
        dict(name="filter_reads", kind="filter", entry="filter", ref_len=100_000_000, repeats=0.3, q=5, bin_len=256,
             overlap=150, n_reads=1_000_000, lmin=150, lmax=150, cands="seeds", cap=1_000),
        # Reads of mixed length with very uneven candidate lists, finer tokens (a bank
        # larger than the L2), in batches.
        dict(name="batched_q6", kind="filter", entry="batched", ref_len=100_000_000, repeats=0.3, q=6, bin_len=256,
             overlap=300, n_reads=500_000, lmin=50, lmax=300, cands="random", k_fixed=0, k_max=5_000),
        # The ordinary call from page-locked host buffers, answers back on the host.
        dict(name="filter_host", kind="filter", entry="host", ref_len=100_000_000, repeats=0.3, q=5, bin_len=256,
             overlap=150, n_reads=400_000, lmin=150, lmax=150, cands="seeds", cap=1_000),
        # Human-genome scale through the dispatcher: about 1,700 candidates per read
        # against a 1.55 GB bank.
        dict(name="auto_genome", kind="filter", entry="auto", ref_len=3_100_000_000, repeats=0.4, q=5, bin_len=256,
             overlap=100, n_reads=1_000_000, lmin=100, lmax=100, cands="seeds", cap=10_000),
        # A batch of reads against every bin of a human-size reference.
        dict(name="scan_genome", kind="scan", ref_len=3_100_000_000, repeats=0.3, q=5, bin_len=256, overlap=100,
             n_reads=16_384, lmin=100, lmax=100, window=0),
        # A small batch of uneven reads against one window of bins.
        dict(name="scan_window", kind="scan", ref_len=100_000_000, repeats=0.3, q=5, bin_len=256, overlap=150,
             n_reads=3_001, lmin=50, lmax=150, window=65_536),
        # The bank of a human-size reference.
        dict(name="bank_genome", kind="bank", ref_len=3_100_000_000, repeats=0.4, q=5, bin_len=256, overlap=100),
        # The bank of finer tokens for reads of up to 300 bases.
        dict(name="bank_q6", kind="bank", ref_len=100_000_000, repeats=0.3, q=6, bin_len=256, overlap=300),
        # The candidate lists of a batch of reads at human-genome scale.
        dict(name="seeds_genome", kind="seeds", ref_len=3_100_000_000, repeats=0.4, bin_len=256, n_reads=500_000,
             lmin=100, lmax=100, cap=10_000),
        # The aligner's check of passing locations, reads of mixed length.
        dict(name="verify_mixed", kind="verify", ref_len=100_000_000, repeats=0.3, bin_len=256, overlap=300,
             n_reads=250_000, lmin=50, lmax=300, per_read=4),
        # The whole mapper path at human-genome scale, in batches: candidates, filter,
        # locations, edit distances.
        dict(name="map_genome", kind="map", ref_len=3_100_000_000, repeats=0.4, q=5, bin_len=256, overlap=100,
             n_reads=300_000, lmin=100, lmax=100, cap=10_000, batch_reads=131_072),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["filter", "filter", "filter", "scan", "bank", "seeds", "verify", "map"])
    ref_len = _log(rng, 1_000_000, 3_100_000_000)
    bin_len = rng.choice([128, 200, 255, 256, 256, 256, 512])
    lmin = rng.choice([50, 75, 100, 100, 150, 150])
    lmax = rng.choice([lmin, lmin, max(lmin, 151), 300])
    c = dict(kind=kind, ref_len=ref_len, repeats=rng.choice([0.0, 0.3, 0.4]), bin_len=bin_len)
    overlap = rng.choice([lmax, lmax, lmax + 15])
    if kind == "bank":
        c.update(q=rng.choice([4, 5, 5, 6]), overlap=overlap)
        if c["q"] == 6:
            c["ref_len"] = min(ref_len, 1_000_000_000)
        return c
    c.update(lmin=lmin, lmax=lmax)
    per_read = _seed_cands(ref_len, (lmin + lmax) / 2)
    if kind == "filter":
        entry = rng.choice(["filter", "batched", "host", "auto"])
        c.update(entry=entry, q=rng.choice([4, 5, 5, 6]), overlap=overlap, cands=rng.choice(["random", "seeds"]))
        if c["q"] == 6:
            c["ref_len"] = ref_len = min(ref_len, 1_000_000_000)
        if c["cands"] == "random":
            c.update(k_fixed=rng.choice([0, 16, 32, 100]), k_max=5_000)
            per_read = c["k_fixed"] or 5_000 / math.log(5_000)
        else:
            c.update(cap=rng.choice([100, 1_000, 10_000]))
            per_read = min(_seed_cands(ref_len, (lmin + lmax) / 2), c["cap"])
        most = 150_000_000 if c["q"] == 6 or entry == "host" else 800_000_000
        c.update(n_reads=_log(rng, 500, max(1_000, min(1_000_000, most / per_read))))
    elif kind == "scan":
        bins = ref_len // bin_len
        window = rng.choice([0, min(bins, 4_096), min(bins, 65_536)])
        # (finer than 5 is refused; coarser, or longer bins, would let nearly every bin pass)
        c.update(q=5, bin_len=min(bin_len, 256), overlap=overlap, window=window,
                 n_reads=_log(rng, 500, max(1_000, min(65_536, 150_000_000_000 / (window or bins)))))
    elif kind == "seeds":
        c.update(cap=rng.choice([100, 1_000, 10_000]), n_reads=_log(rng, 500, max(1_000, min(1_000_000, 600_000_000 / per_read))))
    elif kind == "verify":
        c.update(overlap=overlap, per_read=rng.choice([1, 4, 10]), n_reads=_log(rng, 500, 200_000))
    else:
        n = _log(rng, 500, max(1_000, min(300_000, 400_000_000 / per_read)))
        c.update(q=5, overlap=overlap, cap=rng.choice([1_000, 10_000]), n_reads=n,
                 batch_reads=rng.choice([0, 131_072, max(500, n // 3)]))
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1_000_003 + stream)
    return g


def _u8(shape, hi, g):
    return torch.randint(0, hi, shape, dtype=torch.uint8, device="cuda", generator=g)


def _reference(length, repeats, seed):
    """Base codes (u8) of a reference whose share `repeats` is copies of repeat families."""
    g = _gen(seed, 1)
    codes = torch.empty(length, dtype=torch.uint8, device="cuda")
    table = _u8((N_FAM, FAM_MAX), 4, g)
    fam_len = torch.randint(FAM_MIN, FAM_MAX + 1, (N_FAM,), device="cuda", generator=g)
    p_copy = repeats * SLOT / ((FAM_MIN + FAM_MAX) / 2)
    j = torch.arange(SLOT, device="cuda", dtype=torch.int32)
    step = 16_384 * SLOT
    for p0 in range(0, length, step):
        n = min(step, length - p0)
        slots = -(-n // SLOT)
        base = _u8((slots, SLOT), 4, g)
        if repeats > 0:
            fam = torch.randint(0, N_FAM, (slots,), device="cuda", generator=g)
            has = torch.rand(slots, device="cuda", generator=g) < p_copy
            ln = torch.where(has, fam_len[fam], torch.zeros_like(fam)).to(torch.int32)
            off = (torch.rand(slots, device="cuda", generator=g) * (SLOT - ln)).to(torch.int32)
            div = torch.randint(13, 52, (slots,), device="cuda", generator=g).to(torch.uint8)  # of 256: 5-20%
            src = j[None, :] - off[:, None]
            keep = (src >= 0) & (src < ln[:, None]) & (_u8((slots, SLOT), 256, g) >= div[:, None])
            src = src.clamp_(0, FAM_MAX - 1).add_((fam * FAM_MAX).to(torch.int32)[:, None])
            base = torch.where(keep, torch.take(table, src.to(torch.int64)), base)
            del src, keep
        codes[p0:p0 + n] = base.view(-1)[:n]
    return codes


def _pack(codes):
    n = codes.numel()
    out = torch.empty((n + 3) // 4, dtype=torch.uint8, device="cuda")
    m = n // 4 * 4
    for i in range(0, m, 1 << 28):
        c = codes[i:min(m, i + (1 << 28))].view(-1, 4)
        out[i // 4:i // 4 + c.shape[0]] = c[:, 0] | (c[:, 1] << 2) | (c[:, 2] << 4) | (c[:, 3] << 6)
    if m < n:
        out[-1] = sum(int(b) << (2 * k) for k, b in enumerate(codes[m:].tolist()))
    return out


def _reads(codes, n, lmin, lmax, seed, sub=0.03, indel=0.01):
    """(bases, read_offsets, starts): a walk along the reference from a uniform start, read by read."""
    g = _gen(seed, 2)
    lens = torch.randint(lmin, lmax + 1, (n,), device="cuda", generator=g)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    starts = (torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * (codes.numel() - 2 * lmax)).long()
    bases = torch.empty(int(off[-1]), dtype=torch.uint8, device="cuda")
    col = torch.arange(lmax, device="cuda")
    for r0 in range(0, n, 131_072):
        r1 = min(n, r0 + 131_072)
        u = torch.rand((r1 - r0, lmax), device="cuda", generator=g)
        step = torch.ones((r1 - r0, lmax), dtype=torch.int32, device="cuda")
        ins, dele = u < indel / 2, (u >= indel / 2) & (u < indel)
        step[ins], step[dele] = 0, 2
        src = starts[r0:r1, None] + (torch.cumsum(step, 1) - 1).clamp_(min=0)
        b = torch.take(codes, src)
        rnd = _u8((r1 - r0, lmax), 3, g)
        changed = ins | ((u >= indel) & (u < indel + sub))
        b = torch.where(changed, (b + 1 + rnd) & 3, b)
        bases[int(off[r0]):int(off[r1])] = b[col[None, :] < lens[r0:r1, None]]
    return bases, off, starts


def _random_cands(starts, bin_len, n_bins, k_fixed, k_max, seed):
    """The true bin and uniform others, distinct and ascending: k_fixed, or a log-uniform number up to k_max, per read."""
    g = _gen(seed, 3)
    n = starts.numel()
    if k_fixed:
        k = torch.full((n,), k_fixed, dtype=torch.int64, device="cuda")
    else:
        k = torch.exp(torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * math.log(k_max)).long().clamp_(min=1)
    bins, counts = [], []
    r0 = 0
    ends = torch.cumsum(k, 0).tolist()
    while r0 < n:  # blocks of reads of about 100M candidates
        r1 = r0 + 1
        before = ends[r0 - 1] if r0 else 0
        lo, hi = r1, n
        while lo < hi:
            mid = (lo + hi + 1) // 2
            lo, hi = (mid, hi) if ends[mid - 1] - before <= 100_000_000 else (lo, mid - 1)
        r1 = lo
        kk = k[r0:r1]
        read = torch.repeat_interleave(torch.arange(r1 - r0, device="cuda"), kk)
        b = (torch.rand(read.numel(), dtype=torch.float64, device="cuda", generator=g) * n_bins).long()
        first = torch.cumsum(kk, 0) - kk
        b[first] = (starts[r0:r1] // bin_len).clamp_(max=n_bins - 1)
        key = torch.unique_consecutive(torch.sort(read * (1 << 32) + b)[0])
        bins.append((key & 0xFFFFFFFF).to(torch.int32))
        counts.append(torch.bincount(key >> 32, minlength=r1 - r0))
        r0 = r1
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.cat(counts), 0, out=off[1:])
    return torch.cat(bins), off


def _n_bins(c):
    return -(-c["ref_len"] // c["bin_len"])


def _seed_candidates(c, ref2bit, bases, off):
    idx = grim.grim_seed_index_build(ref2bit, c["ref_len"], SEED_K)
    cb, co = grim.grim_seed_candidates(idx, bases, off, c["bin_len"], _n_bins(c), c["cap"])
    idx.free()
    return cb.clone() if 8 * cb.numel() < cb.untyped_storage().nbytes() else cb, co


def _capacity(c):
    """Room for the candidates of any such batch of reads, by the case alone."""
    n = c["n_reads"]
    if c.get("cands") == "random":
        if c["k_fixed"]:
            return n * c["k_fixed"]
        k = c["k_max"]
        return min(n * k, int(n * k / math.log(k) + 8 * k * math.sqrt(n / math.log(k))))
    return n * min(c["cap"], int(2 * _seed_cands(c["ref_len"], (c["lmin"] + c["lmax"]) / 2)) + 64)


def _budgets(off):
    return ((off[1:] - off[:-1]) * 5 // 100).to(torch.int16)


def prepare(case, seed):
    """The inputs a mapper holds before the call, and the bank or seed table it keeps."""
    c = case
    codes = _reference(c["ref_len"], c["repeats"], seed)
    s = dict(case=c, ref2bit=_pack(codes))
    if c["kind"] in ("filter", "scan", "bank", "map", "verify"):
        s["bank"] = grim.grim_build_bank(s["ref2bit"], c["ref_len"], c.get("q", 5), c["bin_len"], c["overlap"])
    if c["kind"] == "bank":
        return s
    s["reads"], s["off"], starts = _reads(codes, c["n_reads"], c["lmin"], c["lmax"], seed)
    del codes
    s["E"] = _budgets(s["off"])
    if c["kind"] == "filter":
        if c["cands"] == "seeds":
            s["cb"], s["co"] = _seed_candidates(c, s["ref2bit"], s["reads"], s["off"])
        else:
            s["cb"], s["co"] = _random_cands(starts, c["bin_len"], _n_bins(c), c["k_fixed"], c["k_max"], seed)
        # one answer buffer, large enough for any such batch
        s["pass"] = torch.zeros(_capacity(c), dtype=torch.uint8, device="cuda")
        if c["entry"] == "host":
            for k in ("reads", "off", "E", "cb", "co", "pass"):
                t = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=True)
                t.copy_(s[k])
                s[k] = t
    elif c["kind"] in ("seeds", "map"):
        s["idx"] = grim.grim_seed_index_build(s["ref2bit"], c["ref_len"], SEED_K)
        n = c["n_reads"]
        if c["kind"] == "seeds":
            s["cb"] = torch.zeros(_capacity(c), dtype=torch.int32, device="cuda")
            s["co"] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        else:  # room for the locations of any such batch
            s["loc_read"], s["loc_bin"] = (torch.zeros(64 * n, dtype=torch.int32, device="cuda") for _ in "rb")
            s["dist"] = torch.zeros(64 * n, dtype=torch.int16, device="cuda")
    elif c["kind"] == "scan":
        s["out"] = grim.ScanResult(*(torch.zeros(SCAN_CAP, dtype=t, device="cuda")
                                     for t in (torch.int32, torch.int32, torch.int16)),
                                   torch.zeros(1, dtype=torch.int64, device="cuda"),
                                   torch.zeros(c["n_reads"], dtype=torch.int32, device="cuda"))
        s["pairs"] = torch.zeros(SCAN_CAP, dtype=torch.int64, device="cuda")
        s["sums"] = torch.zeros(SCAN_CAP, dtype=torch.int16, device="cuda")
    elif c["kind"] == "verify":
        s["loc_read"] = torch.arange(c["n_reads"], device="cuda").repeat_interleave(c["per_read"]).to(torch.int32)
        g = _gen(seed, 4)
        b = (torch.rand(s["loc_read"].numel(), dtype=torch.float64, device="cuda", generator=g) * _n_bins(c)).long()
        b[::c["per_read"]] = (starts // c["bin_len"]).clamp_(max=_n_bins(c) - 1)
        s["loc_bin"] = b.to(torch.int32)
        s["dist"] = torch.empty(b.numel(), dtype=torch.int16, device="cuda")
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------ the calls

def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _ok(status):
    if status != grim.GRIM_OK:
        raise grim.GrimError(status, "perf case")


def run(state):
    """One pass of the case through the public entry points."""
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "filter":
        args = (s["bank"], s["reads"], s["off"], s["cb"], s["co"], s["E"], s["pass"])
        if c["entry"] == "filter":
            return grim.grim_filter(*args)
        if c["entry"] == "batched":
            return grim.grim_filter_batched(*args)
        if c["entry"] == "host":
            return grim.grim_filter_host(*args)
        return grim.grim_filter_auto(*args)[0]
    if kind == "scan":
        r = grim.grim_scan(s["bank"], s["reads"], s["off"], s["E"], 0, c["window"] or None, out=s["out"])
        # the pairs come in no particular order: put in (read, bin) order, as a mapper takes them
        n = min(r.n_pairs, SCAN_CAP)
        key, order = torch.sort(r.pair_read[:n].long() << 32 | r.pair_bin[:n].long())
        s["pairs"][:n] = key
        s["sums"][:n] = r.pair_sum[:n][order]
        return dict(n_pairs=n, pairs=s["pairs"], sums=s["sums"], read_pass=r.read_pass)
    if kind == "bank":
        grim.grim_build_bank_into(s["bank"], s["ref2bit"])
        rows = s["bank"].bits()  # a view of the bank's own memory
        rows.bank = s["bank"]    # which lives as long as the view
        return rows
    if kind == "verify":
        return grim.grim_verify(s["bank"], s["ref2bit"], s["reads"], s["off"], s["loc_read"], s["loc_bin"], s["dist"])
    # the C entry points fill the caller's own buffers
    n = ctypes.c_int64()
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "seeds":
        _ok(grim.load().grim_seed_candidates(s["idx"].handle, _p(s["reads"]), _p(s["off"]), c["n_reads"], c["bin_len"],
                                             _n_bins(c), c["cap"], _p(s["cb"]), s["cb"].numel(), _p(s["co"]),
                                             ctypes.byref(n), stream))
        return dict(n_cands=n.value, cand_bins=s["cb"], cand_offsets=s["co"])
    _ok(grim.load().grim_map(s["bank"].handle, s["idx"].handle, _p(s["ref2bit"]), _p(s["reads"]), _p(s["off"]),
                             c["n_reads"], _p(s["E"]), c["cap"], c["batch_reads"], _p(s["loc_read"]),
                             _p(s["loc_bin"]), _p(s["dist"]), s["dist"].numel(), ctypes.byref(n), stream, None))
    return dict(n_loc=n.value, loc_read=s["loc_read"], loc_bin=s["loc_bin"], loc_dist=s["dist"])


# ------------------------------------------------------------------ what a pass cannot do without

def _seed_cands(ref_len, L):
    """About how many distinct bins the exact 12-mer hits of a read of L bases fall into."""
    return 1 + (L // SEED_K) * 1.08 * ref_len / 4 ** SEED_K


def _row_bytes(q):
    return max(16, 4 ** q // 8)


def work(case):
    c = case
    n_bins = _n_bins(c)
    packed = (c["ref_len"] + 3) // 4
    if c["kind"] == "bank":
        return {"bytes": packed + n_bins * _row_bytes(c["q"]), "flops": 0}
    n, L = c["n_reads"], (c["lmin"] + c["lmax"]) / 2
    reads = n * (L + 8)
    if c["kind"] == "scan":
        bins = c["window"] or n_bins
        return {"bytes": reads + bins * _row_bytes(c["q"]), "flops": 2.0 * 4 ** c["q"] * n * bins}
    if c["kind"] == "verify":
        loc = n * c["per_read"]
        return {"bytes": reads + loc * 10 + min(packed, loc * (c["bin_len"] + c["overlap"]) / 4), "flops": 0}
    if c["kind"] == "filter" and c["cands"] == "random":
        per_read = c["k_fixed"] or c["k_max"] / math.log(c["k_max"])
    else:
        per_read = min(_seed_cands(c["ref_len"], L), c["cap"])
    cands = n * per_read
    if c["kind"] == "filter":
        rows = min(n_bins, cands) * _row_bytes(c["q"])
        return {"bytes": reads + 10 * n + rows + 5 * cands, "flops": 0}
    votes = n * (L // SEED_K) * c["ref_len"] / 4 ** SEED_K
    table = min(4.0 * c["ref_len"], 4 * votes)
    if c["kind"] == "seeds":
        return {"bytes": reads + table + 4 * cands + 8 * n, "flops": 0}
    return {"bytes": reads + table + min(n_bins, cands) * _row_bytes(c["q"]) + 4 * n * 10, "flops": 0}


# ------------------------------------------------------------------ the same numbers in plain torch

def _tokens(codes, q):
    t = torch.zeros(codes.numel() - q + 1, dtype=torch.int64, device=codes.device)
    for k in range(q):
        t = t * 4 + codes[k:codes.numel() - q + 1 + k].long()
    return t


def _bits(codes, c):
    """Existence table (n_bins, 4^q) of bool."""
    n_bins, q = _n_bins(c), c["q"]
    table = torch.zeros(n_bins * 4 ** q, dtype=torch.bool, device=codes.device)
    tok = _tokens(codes, q)
    pos = torch.arange(tok.numel(), device=codes.device)
    home = pos // c["bin_len"]
    for back in range(c["overlap"] // c["bin_len"] + 2):
        b = home - back
        ok = (b >= 0) & (pos + q <= b * c["bin_len"] + c["bin_len"] + c["overlap"])
        table[b[ok] * 4 ** q + tok[ok]] = True
    return table.view(n_bins, -1)


def exact(case, seed):
    """The outputs of the small filter and bank calls in plain torch integers; None where that would take long."""
    c = case
    if c["ref_len"] > 20_000_000 or c["kind"] not in ("filter", "bank"):
        return None
    if c["kind"] == "filter" and (c["cands"] != "random" or c["n_reads"] * c["lmax"] * (c["k_fixed"] or 600) > 10 ** 9):
        return None
    codes = _reference(c["ref_len"], c["repeats"], seed)
    table = _bits(codes, c)
    if c["kind"] == "bank":
        n_bins, bits = table.shape
        words = torch.zeros((n_bins, max(128, bits)), dtype=torch.int64, device=codes.device)
        words[:, :bits] = table
        words = words.view(n_bins, -1, 32)
        v = (words << torch.arange(32, device=codes.device)).sum(-1)
        return torch.where(v >= 1 << 31, v - (1 << 32), v).to(torch.int32)
    bases, off, starts = _reads(codes, c["n_reads"], c["lmin"], c["lmax"], seed)
    cb, co = _random_cands(starts, c["bin_len"], _n_bins(c), c["k_fixed"], c["k_max"], seed)
    E = _budgets(off).long()
    q, out = c["q"], torch.zeros(_capacity(c), dtype=torch.uint8, device=codes.device)
    o, cl = off.tolist(), co.tolist()
    for r in range(c["n_reads"]):
        if cl[r] == cl[r + 1]:
            continue
        tok = _tokens(bases[o[r]:o[r + 1]], q)
        rows = table[cb[cl[r]:cl[r + 1]].long() & 0xFFFFFFFF]
        sums = rows[:, tok].sum(1)
        out[cl[r]:cl[r + 1]] = (sums >= tok.numel() - q * E[r]).to(torch.uint8)
    return out.cpu() if c["entry"] == "host" else out
