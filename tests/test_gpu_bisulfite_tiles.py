"""Strand rule and T-to-C split over tiles of hits, against the oracle: seeds longer than the marks of a
record reach (256 bases), records with hundreds of hits that cross tiles, records without hits, reads
that are not converted, small and large minimum lengths."""
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


@pytest.mark.parametrize("max_occ,min_len", [(500, 19), (40, 1), (3, 30)])
def test_tiles(mb, max_occ, min_len):
    ref = synth.reference(40_000, 81, tandem=0.4)
    rds = [synth.reads(ref, 40, 82, mode=1, read_len=600, bisulfite=True, sub_lo=0.0005),
           synth.reads(ref, 300, 83, mode=1, read_len=100, bisulfite=True, sub_lo=0.01, sub_hi=0.03)]
    seq = np.concatenate([r.seq for r in rds])
    off = np.concatenate([rds[0].off, rds[1].off[1:] + rds[0].off[-1]])
    mate = np.concatenate([r.mate for r in rds])
    mate[::7] = 0
    G = mb.mb_index_build(ref, opts=dict(flags=mb.MB_BS3))
    o = dict(flags=mb.MB_BS3, max_occ=max_occ)
    sm, m, nh = mb.mb_seed_batch(G, seq, off, mate=mate, opts=o)
    hits, _ = mb.mb_locate(G, sm, m, opts=o, cap=nh)
    length = sm["qend"].astype(np.int64) - sm["qbeg"]
    cnt = np.where(sm["flags"] & 1, 0, sm["s"]).astype(np.int64)
    assert length.max() > 256 and (nh > 512 or max_occ == 3) and (max_occ == 500 or (cnt == 0).any())
    keep = mb.mb_bs_filter(G, sm, m, mate, hits, nh)
    own = np.repeat(np.arange(m), cnt)
    assert np.array_equal(keep, oracle.bs_keep(hits.astype(np.int64), length[own], mate[sm["read"][own]], len(ref)))
    for kp in (keep, None):
        inside = kp is not None or ((hits.astype(np.int64) + length[own] - 1) // len(ref) == hits // len(ref))
        k = kp if kp is not None else inside.astype(np.uint8)   # the oracle splits hits inside one copy
        got = mb.mb_bs_split(G, ref, seq, off, mate, sm, m, hits, nh, keep=kp, opts=dict(min_len=min_len))
        want = oracle.bs_split(ref, seq, off, mate, sm, hits, k, min_len=min_len)
        assert got.tobytes() == want.astype(mb.PIECE_DTYPE).tobytes()


def test_tile_sizes(mb):
    """Numbers of hits on both sides of the lines between tiles of 32, 64, 128 and 256 hits (152 x 32 tiles of
    each), and few: the strand rule against the oracle, the pieces against those of the whole set, whose
    tiles hold 256."""
    r = np.random.default_rng(91)
    ref = np.concatenate([r.integers(0, 4, 15_000), np.tile(r.integers(0, 4, 331), 200), r.integers(0, 4, 15_000)]).astype(np.uint8)
    rd = synth.reads(ref, 8000, 92, mode=1, read_len=150, bisulfite=True, sub_lo=0.002)
    G = mb.mb_index_build(ref, opts=dict(flags=mb.MB_BS3))
    o = dict(flags=mb.MB_BS3, max_occ=2000)
    sm, m, nh = mb.mb_seed_batch(G, rd.seq, rd.off, mate=rd.mate, opts=o)
    hits, _ = mb.mb_locate(G, sm, m, opts=o, cap=nh)
    line = 32 * 152 * 32
    assert nh > 4 * line
    cnt = np.where(sm["flags"] & 1, 0, sm["s"]).astype(np.int64)
    own = np.repeat(np.arange(m), cnt)
    length = (sm["qend"].astype(np.int64) - sm["qbeg"])[own]
    want = oracle.bs_keep(hits.astype(np.int64), length, rd.mate[sm["read"][own]], len(ref)).astype(np.uint8)
    whole = mb.mb_bs_split(G, ref, rd.seq, rd.off, rd.mate, sm, m, hits, nh, keep=want)
    assert len(whole) > 0
    for h in (1, 31, 32, 33, 1000, line, line + 1, 2 * line, 2 * line + 1, 4 * line, 4 * line + 1, nh):
        keep = mb.mb_bs_filter(G, sm, m, rd.mate, hits[:h].copy(), h)
        assert np.array_equal(keep, want[:h]), h
        got = mb.mb_bs_split(G, ref, rd.seq, rd.off, rd.mate, sm, m, hits[:h].copy(), h, keep=keep)
        assert got.tobytes() == whole[whole["hit"] < h].tobytes(), h
