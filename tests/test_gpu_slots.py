"""The SMEM kernel's slot form at its edges, against the CPU oracle: reads cut into items (long reads
inside tandem repeats), records past a read's slots (the pool, and the pass that recomputes a read
when the pool is full), windows of read bases at every alignment, N, reads shorter than l."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mb():
    import paper_2606_15357_gb300 as m
    return m


@pytest.fixture(scope="module")
def tandem(mb):
    """A reference that is 70% tandem repeats; 60 reads of 100-6,000 bases, then reads of 0-330 bases
    with N, some periodic."""
    ref = synth.reference(60_000, 5, tandem=0.7)
    long = synth.reads(ref, 60, 9, mode=2, len_lo=100, len_hi=6000, sub_lo=0.002)
    r = np.random.default_rng(3)
    reads = [long.read(i) for i in range(long.n)]
    for t in range(300):
        n, s = int(r.integers(0, 331)), int(r.integers(0, len(ref) - 400))
        x = ref[s:s + n].copy()
        x[r.random(n) < 0.01] = 4
        if t % 5 == 0 and n > 3:
            x = np.tile(x[:3], n // 3 + 1)[:n]
        reads.append(x)
    off = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.uint64)
    return ref, np.concatenate(reads).astype(np.uint8), off, mb.mb_index_build(ref), oracle.Index(ref)


@pytest.mark.parametrize("l,c,shift,slots", [(19, 1, 0, 0), (19, 1, 7, 3), (12, 2, 1, 0), (5, 3, 15, 0), (1, 3, 0, 0),
                                             (100, 1, 3, 1)])
def test_slots_match_oracle(mb, tandem, l, c, shift, slots):
    ref, seq, off, G, X = tandem
    buf = torch.zeros(len(seq) + shift, dtype=torch.uint8, device="cuda")
    buf[shift:] = torch.from_numpy(seq).cuda()
    o = dict(min_len=l, min_occ=c, smem_reads_per_warp=slots)
    sm, m, nh = mb.mb_seed_batch(G, buf[shift:], torch.from_numpy(off.view(np.int64)).cuda(), opts=o)
    osm, over, hoff, _ = X.seed(seq, off, l, c, 500)
    assert m == len(osm)
    for f in ("read", "qbeg", "qend", "k", "kr", "s"):
        assert np.array_equal(sm[f].astype(np.uint64), osm[f]), f
    assert np.array_equal(sm["flags"] & 1, over.astype(np.uint32))
    # the plan form keeps the positions found while seeding: its hits are the located ones
    P = mb.Plan(G, len(off) - 1, len(seq), m + 1, nh + 1, opts=o)
    P.run(buf[shift:], torch.from_numpy(off.view(np.int64)).cuda())
    psm, phits = P.result()
    assert psm.tobytes() == sm.tobytes()
    hits, _ = mb.mb_locate(G, sm, m, opts=o, cap=nh)
    assert np.array_equal(phits, hits)


def test_long_reads_without_room_to_cut(mb, tandem):
    """The no-allocation call has no items: long reads, meant to be cut at once, run whole in slots that
    held other reads before."""
    ref, seq, off, G, X = tandem
    reps = 8
    big = np.tile(seq, reps)
    boff = np.concatenate([off[:-1] + i * off[-1] for i in range(reps)] + [[reps * off[-1]]]).astype(np.uint64)
    n = len(boff) - 1
    dseq, doff = torch.from_numpy(big).cuda(), torch.from_numpy(boff.view(np.int64)).cuda()
    want, m, _ = mb.mb_seed_batch(G, big, boff)
    out = torch.empty(m * 48, dtype=torch.uint8, device="cuda")
    for slots in (1, 5, 0):
        no, nh = ctypes.c_uint64(), ctypes.c_uint64()
        o = mb.Opts(smem_reads_per_warp=slots)
        rc = mb.lib().mb_seed_batch_noalloc(G.handle, ctypes.c_void_p(dseq.data_ptr()),
                                            ctypes.c_void_p(doff.data_ptr()), n, None, ctypes.byref(o), None,
                                            ctypes.c_void_p(out.data_ptr()), m, ctypes.byref(no), ctypes.byref(nh))
        assert rc == 0 and no.value == m and out.cpu().numpy().tobytes() == want.tobytes()
    osm = X.seed(seq, off, 19, 1, 500)[0]
    assert m == reps * len(osm) and np.array_equal(want["qbeg"][:len(osm)], osm["qbeg"])


def test_profile_counts_the_items_of_cut_reads(mb, tandem):
    """A small batch with cut reads runs the SMEM kernel twice, for the reads and for the items: both are timed;
    a batch without cut reads runs it once."""
    ref, seq, off, G, X = tandem
    short = synth.reads(ref, 50, 3, mode=1, read_len=100)
    for s, o, launches in ((seq, off, 2), (short.seq, short.off, 1)):
        mb.profile_reset()
        mb.profile_enable(True)
        mb.mb_seed_batch(G, s, o)
        mb.profile_enable(False)
        ms, n = mb.profile_get("smem")
        assert n == launches and ms > 0


def test_batch_of_long_reads_has_slots_for_its_records(mb):
    """6,000 reads of 10 kb, all cut before their first step, with a record per 100 bases: more than the pool
    holds (a record per 256 bases).  The records are those of the one-loop form, which cuts nothing, and
    the call takes little more than the same bases in reads of 150 (1.1 and 0.8 ms; 21 ms when reads were
    recomputed one per thread)."""
    ref = np.random.default_rng(12).integers(0, 4, 5_000_000).astype(np.uint8)
    G = mb.mb_index_build(ref)
    G.drop_sa()
    n, length = 6000, 10_000
    rd = synth.reads(ref, n, 13, mode=0, read_len=length, sub_lo=0.01)
    seq, off = torch.from_numpy(rd.seq).cuda(), torch.from_numpy(rd.off.view(np.int64)).cuda()
    short = torch.arange(0, n * length + 1, 150, device="cuda")
    cap = 2 * n * length // 100
    out = torch.zeros(cap * 48, dtype=torch.uint8, device="cuda")
    ms, recs = {}, {}
    for name, o, opts in (("long", off, {}), ("short", short, {}), ("one loop", off, dict(flags=mb.MB_SMEM_ONE_LOOP))):
        t = []
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            _, m, nh = mb.mb_seed_batch(G, seq, o, opts=opts, out=out, cap=cap)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ms[name], recs[name] = min(t), (m, nh, out[:48 * m].cpu().numpy().tobytes())
    assert recs["long"] == recs["one loop"]
    assert recs["long"][0] > n // 2 + n * length // 256 + 16384
    assert ms["long"] < 4 * ms["short"], ms
    P = mb.Plan(G, n, n * length, recs["long"][0] + 1, recs["long"][1] + 1)
    P.run(seq, off)
    psm, phits = P.result()
    assert psm.tobytes() == recs["long"][2]
    hits, _ = mb.mb_locate(G, psm, len(psm), cap=len(phits))
    assert np.array_equal(hits, phits)
