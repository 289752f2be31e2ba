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
