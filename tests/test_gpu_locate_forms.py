"""Every way locate finds positions, against the oracle's full suffix array: the kept full array, walks
to the rate-4 samples after it was dropped (also by a graph captured before), indexes without those
samples (shared walks, plain and joining), other sample rates; records whose hits fill several
pieces, and records that share places in the output."""
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
def small():
    ref, rd, _ = synth.workload(2, scale=0.005)
    X = oracle.Index(ref)
    return ref, rd, X.sa().astype(np.int64)


def records(mb, n, sizes, seed):
    """Records with random places in the text for the given interval sizes, hits one after the other."""
    r = np.random.default_rng(seed)
    sm = np.zeros(len(sizes), dtype=mb.SMEM_DTYPE)
    sm["s"] = sizes
    sm["k"] = [int(r.integers(0, n - s + 1)) for s in sizes]
    sm["flags"][r.random(len(sizes)) < 0.05] = mb.MB_SMEM_OVER_MAX_OCC
    sm["flags"][-1] = 0
    cnt = np.where(sm["flags"] & mb.MB_SMEM_OVER_MAX_OCC, 0, sm["s"]).astype(np.int64)
    sm["hit_off"] = np.concatenate([[0], np.cumsum(cnt)[:-1]])
    rows = np.concatenate([np.arange(int(k), int(k) + int(c)) for k, c in zip(sm["k"], cnt)])
    return sm, rows


@pytest.mark.parametrize("rate,aux,drop", [(32, True, False), (32, True, True), (32, False, True), (1, False, True),
                                           (2, True, True), (4, False, True), (5, True, True), (5, False, True)])
def test_every_index_form(mb, small, rate, aux, drop):
    ref, rd, S = small
    G = mb.mb_index_build(ref, opts=dict(sa_rate=rate, flags=0 if aux else mb.MB_NO_AUX))
    if drop:
        G.drop_sa()
    r = np.random.default_rng(rate)
    sizes = np.concatenate([r.integers(0, 4, 500), r.integers(1, 500, 200), [1, 255, 256, 257, 8192, 8193, 300_000, 1]])
    sm, rows = records(mb, G.n, r.permutation(sizes), 7)
    for flags in (0, mb.MB_LOCATE_JOIN, mb.MB_LOCATE_AUX, mb.MB_CHECKED):
        for depth in (1, 8):
            hits, nh = mb.mb_locate(G, sm, len(sm), opts=dict(flags=flags, prefetch_depth=depth), cap=len(rows))
            assert nh == len(rows) and np.array_equal(hits, S[rows]), (flags, depth)


def test_graph_captured_before_the_array_was_dropped(mb, small):
    ref, rd, S = small
    G = mb.mb_index_build(ref)
    sm, hits = mb.seed(G, rd.seq, rd.off)
    seq, off = torch.from_numpy(rd.seq).cuda(), torch.from_numpy(rd.off.view(np.int64)).cuda()
    P = mb.Plan(G, rd.n, len(rd.seq), len(sm) + 8, len(hits) + 8)
    P.capture(seq, off)
    for drop in (False, True):
        if drop:
            G.drop_sa()
        P.replay()
        psm, phits = P.result()
        assert psm.tobytes() == sm.tobytes() and np.array_equal(phits, hits)


@pytest.mark.parametrize("drop", [False, True])
def test_records_that_share_places(mb, small, drop):
    """2,000 records of one interval, all with the same hit_off: far more hits than output places."""
    ref, rd, S = small
    G = mb.mb_index_build(ref)
    if drop:
        G.drop_sa()
    sm = np.zeros(2000, dtype=mb.SMEM_DTYPE)
    sm["k"], sm["s"] = 12345, 3000
    hits, nh = mb.mb_locate(G, sm, len(sm), cap=3000)
    assert nh == 3000 and np.array_equal(hits, S[12345:15345])


def test_many_hits_share_their_walks(mb, small):
    """More than 2^25 hits on a dropped array: each distinct row walked once, to the rate-4 samples."""
    ref, rd, S = small
    G = mb.mb_index_build(ref)
    G.drop_sa()
    sm, rows = records(mb, G.n, np.full(90, 400_000), 3)
    assert len(rows) > 1 << 25
    dsm = torch.from_numpy(sm.view(np.uint8)).cuda()
    out = torch.empty(len(rows), dtype=torch.int32, device="cuda")
    want = torch.from_numpy(S.astype(np.int32)).cuda()[torch.from_numpy(rows).cuda()]
    for flags in (0, mb.MB_LOCATE_JOIN):
        out.zero_()
        mb.mb_locate(G, dsm, len(sm), opts=dict(flags=flags), hits=out, cap=len(rows))
        assert torch.equal(out, want)


@pytest.mark.parametrize("rate", [1, 2, 3, 4, 5, 6, 7, 12, 33])
@pytest.mark.parametrize("aux", [True, False])
def test_every_rate_dropped_and_loaded(mb, small, tmp_path, rate, aux):
    """Sample rates on both sides of the rate-4 samples, powers of two and not, without the full array:
    after it was dropped, and on an index read back from its file (which never has it); mb_locate, a plan
    and the pipelined call."""
    ref, rd, S = small
    G = mb.mb_index_build(ref, opts=dict(sa_rate=rate, flags=0 if aux else mb.MB_NO_AUX))
    G.save(str(tmp_path / "i.mbi"))
    G.drop_sa()
    r = np.random.default_rng(rate)
    sm, rows = records(mb, G.n, np.concatenate([r.integers(0, 40, 400), [5000, 1]]), rate)
    want_sm, _, _ = mb.mb_seed_batch(G, rd.seq, rd.off)
    cnt = np.where(want_sm["flags"] & mb.MB_SMEM_OVER_MAX_OCC, 0, want_sm["s"]).astype(np.int64)
    want = S[np.concatenate([np.arange(int(k), int(k) + int(c)) for k, c in zip(want_sm["k"], cnt)])]
    seq, off = torch.from_numpy(rd.seq).cuda(), torch.from_numpy(rd.off.view(np.int64)).cuda()
    for X in (G, mb.mb_index_load(str(tmp_path / "i.mbi"))):
        hits, nh = mb.mb_locate(X, sm, len(sm), cap=len(rows))
        assert nh == len(rows) and np.array_equal(hits, S[rows])
        P = mb.Plan(X, rd.n, len(rd.seq), len(want_sm) + 8, len(want) + 8)
        P.run(seq, off)
        psm, phits = P.result()
        assert psm.tobytes() == want_sm.tobytes() and np.array_equal(phits, want)
        lsm, lhits = mb.seed_locate(X, rd.seq, rd.off)
        assert lsm.tobytes() == want_sm.tobytes() and np.array_equal(lhits, want)


@pytest.mark.parametrize("rate", [1, 2, 3, 4])
def test_many_hits_at_dense_rates(mb, small, rate):
    """More than 2^25 hits without the full array where the index's own samples are as dense as the rate-4
    ones or denser, or not a power of two apart."""
    ref, rd, S = small
    G = mb.mb_index_build(ref, opts=dict(sa_rate=rate))
    G.drop_sa()
    sm, rows = records(mb, G.n, np.full(110, 400_000), rate)
    assert len(rows) > 1 << 25
    dsm = torch.from_numpy(sm.view(np.uint8)).cuda()
    out = torch.empty(len(rows), dtype=torch.int32, device="cuda")
    want = torch.from_numpy(S.astype(np.int32)).cuda()[torch.from_numpy(rows).cuda()]
    for flags in (0, mb.MB_LOCATE_AUX, mb.MB_LOCATE_JOIN, mb.MB_CHECKED, mb.MB_COUNT, mb.MB_COUNT | mb.MB_LOCATE_AUX):
        out.zero_()
        mb.mb_locate(G, dsm, len(sm), opts=dict(flags=flags), hits=out, cap=len(rows))
        assert torch.equal(out, want), flags


def test_dense_own_samples_end_the_walks(mb):
    """36M distinct rows without the full array: with every row sampled no walk takes a step (0.15 ms; 0.96 ms
    to the rate-4 samples), so the walks take well under those of an index that has only the latter."""
    ref = np.random.default_rng(2).integers(0, 4, 40_000_000).astype(np.uint8)
    sm = np.zeros(400_000, dtype=mb.SMEM_DTYPE)
    sm["s"], sm["k"], sm["hit_off"] = 90, np.arange(400_000) * 199, np.arange(400_000) * 90
    dsm = torch.from_numpy(sm.view(np.uint8)).cuda()
    out = torch.empty(36_000_000, dtype=torch.int32, device="cuda")
    ms = {}
    for rate in (1, 32):
        G = mb.mb_index_build(ref, opts=dict(sa_rate=rate))
        G.drop_sa()
        for _ in range(6):
            mb.profile_reset()
            mb.profile_enable(True)
            mb.mb_locate(G, dsm, len(sm), hits=out, cap=out.numel())
            mb.profile_enable(False)
            ms[rate] = min(ms.get(rate, 1e9), mb.profile_get("locate")[0])
        G.free()
    assert ms[1] < 0.5 * ms[32], ms


def test_hits_up_to_the_walk_queue_limit(mb, small):
    """4,292M hits, under what one walk per lane can queue (2^32 less a chunk per warp), on a dropped array:
    4,292 records of the same 1M rows, walked once."""
    free, _ = torch.cuda.mem_get_info()
    if free < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    ref, rd, S = small
    G = mb.mb_index_build(ref)
    G.drop_sa()
    n = G.n
    m = 4_292_300_000 // n
    sm = np.zeros(m, dtype=mb.SMEM_DTYPE)
    sm["s"], sm["hit_off"] = n, np.arange(m) * n
    out = torch.zeros(m * n, dtype=torch.int32, device="cuda")
    hits, nh = mb.mb_locate(G, torch.from_numpy(sm.view(np.uint8)).cuda(), m, hits=out, cap=m * n)
    want = torch.from_numpy(S.astype(np.int32)).cuda()
    assert nh == m * n and all(torch.equal(out[t * n:(t + 1) * n], want) for t in range(m))
