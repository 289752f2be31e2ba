"""Seeding workloads of this library, each through the calls a program makes, with seeded inputs.

A case names a `kind` (the entry points it goes through), a reference (bases, the share of it that
is repeats, k of the k-mer table, whether the full suffix array was dropped after the build) and a
batch.  References are drawn once per case shape and kept with their index, as a mapper keeps its
genome; reads are drawn from the seed of each preparation.  The shapes follow the workloads of the
benchmark and the tests: 1 Mbp uniform, 100 Mbp with 8% repeats, 1 Gbp with 45% repeats; 2x150 bp
pairs, single reads of 100 bp - 10 kb, bisulfite pairs, mate-rescue pairs, served requests.
"""
import collections
import ctypes
import math

import numpy as np
import torch

import paper_2606_15357_gb300 as mb

DEV = "cuda"
BENCH = dict(block_size=512, prefetch_depth=2, flags=mb.MB_BATCHED | mb.MB_LOCATE_JOIN)   # the 1 Gbp step
MIXED = dict(block_size=128, smem_burst=8, smem_wait=16, prefetch_depth=4, flags=mb.MB_BATCHED)


def _case(name, kind, ref, repeat, reads, lo=150, hi=150, k=10, drop=False, c=1):
    d = dict(kind=kind, ref=ref, repeat=repeat, reads=reads, len_lo=lo, len_hi=hi, kmer_k=k, drop_sa=drop, min_occ=c)
    return dict(d, name=name) if name else d


def listed():
    return [
        # an interactive query: a few reads against a small genome, the latency of the two calls
        _case("call_64", "device", 1_000_000, 0.0, 64),
        # a small batch of a program that keeps a plan and replays its graph
        _case("graph_10k", "graph", 1_000_000, 0.0, 10_000),
        # convenience call on host arrays, ragged reads, at least two occurrences asked for
        _case("host_call_20k", "seed", 100_000_000, 0.08, 20_000, 36, 301, c=2),
        # one batch of 2x150 bp pairs in device memory, default options
        _case("batch_2m", "device", 100_000_000, 0.08, 2_000_000),
        # the headline step: 20M reads, 1 Gbp repeat-rich genome, one graph launch
        _case("graph_20m", "graph_bench", 1_000_000_000, 0.45, 20_000_000, k=14, drop=True),
        # a mapper's stream: reads and results in pinned host memory, one call per batch
        _case("pinned_4m", "pinned", 1_000_000_000, 0.45, 4_000_000, k=14, drop=True),
        # long and short reads mixed, the shape the autotuner picks for them
        _case("mixed_200k", "graph_mixed", 100_000_000, 0.08, 200_000, 100, 10_000),
        # bisulfite pairs: seeding and locate on the 3-base index, strand rule, T-to-C split
        _case("bisulfite_500k", "bisulfite", 100_000_000, 0.45, 500_000),
        # the second seeding round on the records of the first
        _case("reseed_1m", "reseed", 100_000_000, 0.08, 1_000_000),
        # mate-rescue prefilter: reads against 600 bp windows, ragged read lengths
        _case("rescue_1m", "rescue", 100_000_000, 0.0, 1_000_000, 100, 150),
        # indexing a genome
        _case("index_100m", "index", 100_000_000, 0.08, 0),
        # 30 requests of different sizes to a running server, from submit to the last result
        _case("serve_30", "serve", 100_000_000, 0.08, 30),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["device", "device", "graph", "graph_bench", "pinned", "graph_mixed", "bisulfite", "reseed",
                       "rescue", "seed", "index", "serve"])
    ref = _log(rng, 1_000_000, 200_000_000)
    repeat = rng.choice([0.0, 0.08, 0.45])
    k = rng.choice([10, 10, 12, 14])
    drop = rng.random() < 0.5
    if kind == "index":
        return _case(None, kind, _log(rng, 500_000, 100_000_000), repeat, 0, k=rng.choice([10, 12]))
    if kind == "serve":
        return _case(None, kind, ref, repeat, rng.randint(3, 30), k=k, drop=drop)
    if kind == "rescue":
        return _case(None, kind, ref, 0.0, _log(rng, 1_000, 1_000_000), rng.randint(60, 140), rng.randint(140, 251))
    if kind == "graph_mixed":
        return _case(None, kind, ref, repeat, _log(rng, 2_000, 200_000), 100, rng.randint(2_000, 10_000), k=k, drop=drop)
    if kind == "seed":
        return _case(None, kind, ref, repeat, _log(rng, 10, 40_000), rng.randint(20, 100), rng.randint(100, 400), k=k,
                     drop=drop, c=rng.choice([1, 2, 3]))
    if kind in ("graph_bench", "pinned") and rng.random() < 0.3:
        ref = _log(rng, 200_000_000, 1_000_000_000)
    lo = rng.choice([76, 100, 150, 250])
    hi = lo if rng.random() < 0.5 else lo + rng.randint(1, 60)
    top = {"device": 4_000_000, "graph": 1_000_000, "graph_bench": 10_000_000, "pinned": 2_000_000,
           "bisulfite": 500_000, "reseed": 500_000}[kind]
    return _case(None, kind, ref, repeat, 2 * _log(rng, 16, top // 2), lo, hi, k=k, drop=drop)


# ---------------------------------------------------------------------------- inputs
def _rng(seed):
    return torch.Generator(DEV).manual_seed(int(seed))


def _reference(length, repeat, seed):
    """Uniform bases; tandem : segmental : satellite repeats 5 : 2 : 1 over `repeat` of it; 0.5% N."""
    g, r = _rng(seed), np.random.default_rng(seed)
    ref = torch.randint(0, 4, (length,), dtype=torch.uint8, device=DEV, generator=g)
    spans = []
    for what, share in (("tandem", 5 / 8), ("dup", 2 / 8), ("satellite", 1 / 8)):
        left = repeat * share * length
        while left > 0:
            period = int(r.integers(1, 201)) if what == "tandem" else 171
            n = int(r.integers(1_000, 50_000)) if what == "dup" else period * int(r.integers(2, 501))
            n = min(n, length // 8, int(left) + 400)
            spans.append((what, period, n))
            left -= n
    left = 0.005 * length if repeat else 0
    while left > 0:
        spans.append(("n", 0, int(r.integers(100, min(10_000, length // 20)))))
        left -= spans[-1][2]
    r.shuffle(spans)
    free = length - sum(int(n) for _, _, n in spans)
    gaps = np.sort(r.integers(0, max(free, 1), len(spans)))
    at = 0
    for i, (what, period, n) in enumerate(spans):
        period, n = int(period), int(n)
        at += int(gaps[i] - (gaps[i - 1] if i else 0))
        span = ref[at:at + n]
        if what == "n":
            span.fill_(4)
        else:
            if what == "dup":
                s = int(r.integers(0, length - n))
                new = ref[s:s + n].clone()
                if r.random() < 0.5:
                    new = torch.where(new < 4, 3 - new, new).flip(0)
                rate = r.uniform(0.01, 0.05)
            else:
                s = int(r.integers(0, 4)) * 1000 if what == "satellite" else int(r.integers(0, length - period))
                new = ref[s:s + period].repeat(n // period + 1)[:n]
                rate = 0.02 if what == "satellite" else r.uniform(0, 0.03)
            hit = torch.rand(n, device=DEV, generator=g) < rate
            other = torch.randint(0, 4, (n,), dtype=torch.uint8, device=DEV, generator=g)
            span.copy_(torch.where(hit & (new < 4), other, new))
        at += n
    return ref


def _lengths(case, n, r):
    lo, hi = case["len_lo"], case["len_hi"]
    if lo == hi:
        return np.full(n, lo, np.int64)
    if hi > 8 * lo:
        return np.exp(r.uniform(math.log(lo), math.log(hi), n)).astype(np.int64)
    return r.integers(lo, hi + 1, n).astype(np.int64)


def _reads(ref, lens, seed, pairs, bisulfite=False, sub=(0.001, 0.01), indel=1e-4):
    """(seq uint8, off int64, mate uint8) on the device: pairs with an insert of N(400, 50), or single
    reads; substitutions ramping along the read, one 1-3 bp indel in some, a few N."""
    g, r, n, L = _rng(seed), np.random.default_rng(seed), len(lens), ref.numel()
    start = r.integers(0, L - int(lens.max()) - 8, n)
    rc = r.integers(0, 2, n)
    if pairs:   # the mate lies an insert away on the other strand
        ins = np.maximum(r.normal(400, 50, n // 2).astype(np.int64), lens[1::2])
        start[1::2] = np.clip(np.where(rc[0::2] == 0, start[0::2] + ins - lens[1::2],
                                       start[0::2] + lens[0::2] - ins), 0, L - lens[1::2] - 8)
        rc[1::2] = 1 - rc[0::2]
    gap = np.where(r.random(n) < indel * lens, r.integers(-3, 4, n), 0)
    cut = (r.random(n) * lens).astype(np.int64)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    per = torch.from_numpy(np.stack([lens, start, rc, gap, cut])).to(DEV)
    doff = torch.from_numpy(off).to(DEV)
    seq = torch.empty(int(off[-1]), dtype=torch.uint8, device=DEV)
    mate = torch.zeros(n, dtype=torch.uint8, device=DEV)
    if pairs:
        mate[0::2], mate[1::2] = 1, 2
    a = 0
    while a < n:
        b = max(a + 1, int(np.searchsorted(off, off[a] + (1 << 26), side="right")) - 1)
        o, tot = doff[a:b] - off[a], int(off[b] - off[a])
        rid = torch.repeat_interleave(torch.arange(a, b, device=DEV), per[0, a:b], output_size=tot)
        ln, st, flip, gp, ct = (x[rid] for x in per)
        j = torch.arange(tot, device=DEV) - o[rid - a]
        t = j + torch.where(j >= ct, gp, 0)
        x = (st + torch.where(flip == 1, ln - 1 - t, t)).clamp_(0, L - 1)
        v = ref[x]
        v = torch.where((flip == 1) & (v < 4), 3 - v, v)
        if bisulfite:
            m = mate[rid]
            cpg = ((m == 1) & (v.roll(-1) == 2)) | ((m == 2) & (v.roll(1) == 1))
            conv = torch.rand(tot, device=DEV, generator=g) < torch.where(cpg, 0.30, 0.98)
            v = torch.where(conv & (m == 1) & (v == 1), 3, torch.where(conv & (m == 2) & (v == 2), 0, v)).to(torch.uint8)
        u = torch.rand(tot, device=DEV, generator=g)
        hit = (u < sub[0] + (sub[1] - sub[0]) * j / ln) & (v < 4)
        v = torch.where(hit, (v + 1 + torch.randint(0, 3, (tot,), dtype=torch.uint8, device=DEV, generator=g)) % 4, v)
        seq[off[a]:off[b]] = torch.where(u > 1 - 1e-5, 4, v)
        a = b
    return seq, doff, mate


class _Kept:
    """A few indexes (and servers on them), the least recently used given up first."""

    def __init__(self, most):
        self.most, self.kept = most, collections.OrderedDict()

    def get(self, key, make):
        if key not in self.kept:
            while len(self.kept) >= self.most:
                self.kept.popitem(last=False)
            self.kept[key] = make()
        self.kept.move_to_end(key)
        return self.kept[key]


_genomes, _servers = _Kept(2), _Kept(1)


def _genome(case):
    """(reference on the device, its index), the same for every seed."""
    bs = case["kind"] == "bisulfite"
    key = (case["ref"], case["repeat"], case["kmer_k"], case["drop_sa"], bs)

    def make():
        ref = _reference(case["ref"], case["repeat"], 0x6D6200)
        idx = mb.mb_index_build(ref, opts=dict(kmer_k=case["kmer_k"], flags=mb.MB_BS3 if bs else 0))
        if case["drop_sa"]:
            idx.drop_sa()
        return ref, idx

    return key, _genomes.get(key, make)


_rooms = {}


def _room(case, idx, ref):
    """Records and hits that a program leaves room for, from a sample of such reads: 30% above it."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _rooms:
        n, r = case["reads"], np.random.default_rng(5)
        ns = min(n, 20_000)
        seq, off, mate = _batch(case, ref, ns, 5, r)
        cap = 4 * ns + seq.numel() // 16 + 1024
        _, m, nh = mb.mb_seed_batch(idx, seq, off, mate if case["kind"] == "bisulfite" else None, opts=_opts(case),
                                    cap=cap, out=torch.empty(cap * 48, dtype=torch.uint8, device=DEV))
        _rooms[key] = int(1.3 * m * n / ns) + 4096, int(1.3 * nh * n / ns) + (1 << 20)
    return _rooms[key]


def _opts(case):
    o = dict(min_occ=case["min_occ"], max_occ=500)
    o.update({"graph_bench": BENCH, "pinned": BENCH, "graph_mixed": MIXED}.get(case["kind"], {}))
    if case["kind"] == "bisulfite":
        o.update(flags=mb.MB_BS3)
    return mb.Opts(**o)


def _batch(case, ref, n, seed, r):
    long = case["kind"] == "graph_mixed"
    pairs = not long and case["kind"] != "seed" and n % 2 == 0
    return _reads(ref, _lengths(case, n, r), seed, pairs, bisulfite=case["kind"] == "bisulfite",
                  sub=(0.001, 0.001) if long else (0.001, 0.01), indel=2e-4 if long else 1e-4)


def prepare(case, seed):
    kind, n = case["kind"], case["reads"]
    s = dict(kind=kind)
    if kind == "index":
        return dict(s, ref=_reference(case["ref"], case["repeat"], seed), opts=dict(kmer_k=case["kmer_k"]))
    r = np.random.default_rng(seed + 1)
    if kind == "rescue":
        ref = _reference(case["ref"], 0.0, seed)
        return dict(s, **_rescue_pairs(case, ref, r, seed))
    key, (ref, s["idx"]) = _genome(case)
    if kind == "serve":
        s["server"] = _servers.get(key, lambda: mb.Server(s["idx"], hbm_budget=8 << 30))
        s["requests"], s["smem"], s["hits"] = [], np.zeros((1 << 19, 6), np.int64), np.zeros(1 << 24, np.int32)
        r = np.random.default_rng(n)   # the same request sizes for every seed
        for q in range(n):   # four of five are short pairs, one is long single reads
            long = r.random() < 0.2
            k = int(math.exp(r.uniform(0, math.log(2048))))
            lens = np.exp(r.uniform(math.log(1000), math.log(10_000), max(1, k // 4))).astype(np.int64) if long \
                else np.full(2 * k, 150, np.int64)
            seq, off, _ = _reads(ref, lens, seed * 64 + q, pairs=not long)
            s["requests"].append((seq.cpu().numpy(), off.cpu().numpy().view(np.uint64)))
        return s
    s["seq"], s["off"], s["mate"] = _batch(case, ref, n, seed, r)
    s.update(ref=ref, opts=_opts(case))
    s["cap"], s["hits_cap"] = _room(case, s["idx"], ref)
    where = dict(pin_memory=True) if kind == "pinned" else dict() if kind == "seed" else dict(device=DEV)
    s["out"] = torch.zeros((s["cap"], 6), dtype=torch.int64, **where)
    s["hits"] = torch.zeros(s["hits_cap"], dtype=torch.int32, **where)
    if kind.startswith("graph"):
        s["plan"] = mb.Plan(s["idx"], n, s["seq"].numel(), s["cap"], s["hits_cap"], opts=s["opts"])
        s["plan"].capture(s["seq"], s["off"])
    if kind in ("pinned", "seed"):
        for k in ("seq", "off"):
            s[k] = torch.empty(s[k].shape, dtype=s[k].dtype, pin_memory=kind == "pinned").copy_(s[k])
    if kind == "reseed":
        s["first"] = torch.empty_like(s["out"])
        _, s["n_first"], _ = mb.mb_seed_batch(s["idx"], s["seq"], s["off"], opts=s["opts"], out=s["first"], cap=s["cap"])
    if kind == "bisulfite":
        s["keep"] = torch.zeros(s["hits_cap"], dtype=torch.uint8, device=DEV)
        s["pieces"] = torch.zeros((s["hits_cap"], 3), dtype=torch.int64, device=DEV)
    torch.cuda.synchronize()
    return s


def _rescue_pairs(case, ref, r, seed, win=600):
    """Windows at uniform places; half of the reads come from their window, half from elsewhere."""
    n, L = case["reads"], ref.numel()
    lens = _lengths(case, n, r)
    w0 = r.integers(0, L - win, n)
    inside = w0 + (r.random(n) * (win - lens)).astype(np.int64)
    st = np.where(r.random(n) < 0.5, inside, r.integers(0, L - win, n))
    roff = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=roff[1:])
    g, dst, dl = _rng(seed), torch.from_numpy(st).to(DEV), torch.from_numpy(lens).to(DEV)
    off = torch.from_numpy(roff).to(DEV)
    rid = torch.repeat_interleave(torch.arange(n, device=DEV), dl, output_size=int(roff[-1]))
    v = ref[dst[rid] + torch.arange(int(roff[-1]), device=DEV) - off[rid]]
    hit = torch.rand(v.numel(), device=DEV, generator=g) < 0.01
    v = torch.where(hit, (v + 1 + torch.randint(0, 3, v.shape, dtype=torch.uint8, device=DEV, generator=g)) % 4, v)
    wins = torch.empty(n * win, dtype=torch.uint8, device=DEV)
    for a in range(0, n, 1 << 17):
        w = torch.from_numpy(w0[a:a + (1 << 17)]).to(DEV)
        wins[a * win:(a + w.numel()) * win] = ref[(w[:, None] + torch.arange(win, device=DEV))].reshape(-1)
    return dict(reads=v, roff=off, wins=wins, woff=torch.arange(n + 1, device=DEV) * win,
                best=torch.empty(n, dtype=torch.int32, device=DEV))


# ---------------------------------------------------------------------------- one pass
class _DevArray:
    """`n` items at a device pointer of the library, for torch; `owner` (the plan that holds them) lives
    as long as a tensor made from it."""

    def __init__(self, owner, ptr, n, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=(n,), typestr=typestr, data=(ptr, False), version=3)


def _device(owner, ptr, n, typestr, dtype):
    return torch.as_tensor(_DevArray(owner, ptr, n, typestr), device=DEV) if n else torch.empty(0, dtype=dtype, device=DEV)


def _call(name, *args):
    """One call of the C interface with the current stream, arrays given by their addresses."""
    at = [ctypes.c_void_p(a.data_ptr()) if isinstance(a, torch.Tensor) else a for a in args]
    rc = getattr(mb.lib(), name)(*at)
    if rc:
        raise mb.MbError(rc, name)


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def run(s):
    kind = s["kind"]
    if kind.startswith("graph"):   # the plan's results are its own until its next run: kept by a copy
        s["plan"].replay()
        sp, m, hp, nh = s["plan"].result_ptrs()
        s["out"][:m].copy_(_device(s["plan"], sp, 6 * m, "<i8", torch.int64).view(-1, 6))
        s["hits"][:nh].copy_(_device(s["plan"], hp, nh, "<i4", torch.int32))
        return dict(smem=s["out"], hits=s["hits"], n=[m, nh])
    if kind == "pinned":
        m, nh = mb.seed_locate(s["idx"], s["seq"], s["off"], opts=s["opts"], out=s["out"], cap=s["cap"],
                               hits=s["hits"], hits_cap=s["hits_cap"])
        return dict(smem=s["out"], hits=s["hits"], n=[m, nh])
    if kind == "reseed":
        m, nh = ctypes.c_uint64(), ctypes.c_uint64()
        _call("mb_reseed", s["idx"].handle, s["seq"], s["off"], s["off"].numel() - 1, None, s["first"], s["n_first"],
              ctypes.byref(s["opts"]), _stream(), s["out"], s["cap"], ctypes.byref(m), ctypes.byref(nh))
        return dict(smem=s["out"], n=[m.value, nh.value])
    if kind == "rescue":
        return mb.mb_rescue_prefilter(s["reads"], s["roff"], s["wins"], s["woff"], best=s["best"])
    if kind == "index":
        idx = mb.mb_index_build(s["ref"], opts=s["opts"])
        arrays = idx.export(ssa=True, occ=True, kmer=True, kmer_k=s["opts"]["kmer_k"])
        return {name: a.view(np.int32 if a.itemsize == 4 else np.int64) for name, a in arrays.items()}
    if kind == "serve":   # every request's results in one array of the program's own
        m = nh = 0
        tickets = [s["server"].submit(seq, off) for seq, off in s["requests"]]
        for t in tickets:
            sm, hits, _ = s["server"].wait(t)
            s["smem"][m:m + len(sm)] = sm.view(np.int64).reshape(-1, 6)
            s["hits"][nh:nh + len(hits)] = hits.view(np.int32)
            m, nh = m + len(sm), nh + len(hits)
        return dict(smem=s["smem"], hits=s["hits"], n=[m, nh])
    mate = s["mate"] if kind == "bisulfite" else None
    _, m, nh = mb.mb_seed_batch(s["idx"], s["seq"], s["off"], mate, opts=s["opts"], out=s["out"], cap=s["cap"])
    mb.mb_locate(s["idx"], s["out"], m, opts=s["opts"], hits=s["hits"], cap=s["hits_cap"])
    got = dict(smem=s["out"], hits=s["hits"], n=[m, nh])
    if kind == "bisulfite":
        mb.mb_bs_filter(s["idx"], s["out"], m, mate, s["hits"], nh, keep=s["keep"])
        np_ = ctypes.c_uint64()
        _call("mb_bs_split", s["idx"].handle, s["ref"], s["seq"], s["off"], s["off"].numel() - 1, mate, s["out"], m,
              s["hits"], s["keep"], nh, ctypes.byref(s["opts"]), _stream(), s["pieces"], s["hits_cap"],
              ctypes.byref(np_))
        got.update(keep=s["keep"], pieces=s["pieces"], n=[m, nh, np_.value])
    return got


def work(case):
    """Inputs read once, outputs written once; record and hit counts are those usual for the shape."""
    n, mean = case["reads"], (case["len_lo"] + case["len_hi"]) / 2
    if case["kind"] == "index":   # bases in; blocks, sampled suffix array and k-mer table out
        return dict(bytes=case["ref"] * (1 + 1 + 0.25) + 12 * 4 ** case["kmer_k"], flops=0)
    if case["kind"] == "rescue":
        return dict(bytes=n * (mean + 600 + 20), flops=0)
    if case["kind"] == "serve":   # requests average about 270 reads of 150, or 70 of 4 kb
        n, mean = n * 220, 300
    elif case["len_hi"] > 8 * case["len_lo"]:
        mean = (case["len_hi"] - case["len_lo"]) / math.log(case["len_hi"] / case["len_lo"])
    per = 1.2 + mean / 400
    return dict(bytes=n * (mean + 8 + per * 48 + per * 4 * (8 if case["repeat"] > 0.1 else 2)), flops=0)


def exact(case, seed):
    """Every output is a whole number, compared for equality: there is no rounding to measure."""
    return None
