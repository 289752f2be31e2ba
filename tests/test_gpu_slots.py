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
