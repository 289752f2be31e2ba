"""Mate-rescue prefilter (Section 2.7) on the GPU against the oracle's definition: max over
diagonals t of the number of q-mer matches (i, j) with j - i = t, per (read, window) pair."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_15357_gb300 as m
    m.lib()
    return m


def dev(a):
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a.view(np.int64) if a.dtype == np.uint64 else a).cuda()


def test_mate_rescue_shaped_pairs(mb):
    ref = synth.repeat_rich_reference(300_000, 95, 0.2)
    r, ro, w, wo = synth.rescue_pairs(ref, 3000, 96)
    want = oracle.qmer_diag_max_batch(r, ro, w, wo)
    assert 0.3 < (want >= 10).mean() < 0.7
    assert np.array_equal(mb.mb_rescue_prefilter(r, ro, w, wo), want)
    got = torch.empty(len(want), dtype=torch.int32, device="cuda")
    mb.mb_rescue_prefilter(dev(r), dev(ro), dev(w), dev(wo), best=got)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("q", [1, 4, 7, 11, 15])
def test_lengths_ns_and_q(mb, q):
    """Reads of 0-300 bases, windows of 0-2,000 (shorter than q included), N bases, any q."""
    rng = np.random.default_rng(q)
    reads, wins = [], []
    for t in range(600):
        W = rng.integers(0, 4, int(rng.integers(0, 2000))).astype(np.uint8)
        if t % 3 == 0 and len(W) > 300:
            s = int(rng.integers(0, len(W) - 300))
            P = W[s:s + int(rng.integers(0, 300))].copy()
        else:
            P = rng.integers(0, 4, int(rng.integers(0, 300))).astype(np.uint8)
        for x in (P, W):
            if len(x):
                k = int(rng.integers(0, 4))
                x[rng.integers(0, len(x), k)] = 4
        reads.append(P)
        wins.append(W)
    ro = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.uint64)
    wo = np.concatenate([[0], np.cumsum([len(x) for x in wins])]).astype(np.uint64)
    r, w = np.concatenate(reads).astype(np.uint8), np.concatenate(wins).astype(np.uint8)
    want = oracle.qmer_diag_max_batch(r, ro, w, wo, q)
    assert np.array_equal(mb.mb_rescue_prefilter(r, ro, w, wo, q=q), want)


def test_periodic_pairs_and_empty_batch(mb):
    P = np.tile(np.array([0, 1], np.uint8), 100)
    W = np.tile(np.array([0, 1], np.uint8), 400)
    got = mb.mb_rescue_prefilter(P, np.array([0, 200], np.uint64), W, np.array([0, 800], np.uint64))
    assert got.tolist() == [200 - 7 + 1]
    e = mb.mb_rescue_prefilter(P, np.array([0], np.uint64), W, np.array([0], np.uint64))
    assert len(e) == 0
    with pytest.raises(mb.MbError):
        mb.mb_rescue_prefilter(P, np.array([0, 200], np.uint64), W, np.array([0, 800], np.uint64), q=16)


@pytest.mark.parametrize("m", [6, 31, 32, 33, 64, 96, 97, 128, 160, 161, 256, 257])
def test_word_edges(mb, m):
    """Read and window lengths around the 32-base words of the register form (reads up to 256 bases) and
    past it, unaligned in memory, q at and off 7, matches up to both ends of the window."""
    rng = np.random.default_rng(m)
    reads, wins = [rng.integers(0, 4, 1).astype(np.uint8)], [rng.integers(0, 4, 3).astype(np.uint8)]
    for w in (m, m + 1, 31, 32, 33, 63, 64, 65, 600, 1023, 1025):
        for at in (0, 1):
            W = rng.integers(0, 2, w).astype(np.uint8)
            P = np.resize(W[:m] if at == 0 else W[max(0, w - m):], m) if w else W
            P = np.where(rng.random(m) < 0.02, 4, P).astype(np.uint8)
            reads.append(P)
            wins.append(W)
    ro = np.concatenate([[0], np.cumsum([len(x) for x in reads])]).astype(np.uint64)
    wo = np.concatenate([[0], np.cumsum([len(x) for x in wins])]).astype(np.uint64)
    r, w = np.concatenate(reads), np.concatenate(wins)
    for q in (7, 8, 15, 1):
        want = oracle.qmer_diag_max_batch(r, ro, w, wo, q)
        got = torch.empty(len(want), dtype=torch.int32, device="cuda")
        mb.mb_rescue_prefilter(dev(r), dev(ro), dev(w), dev(wo), q=q, best=got)
        assert np.array_equal(got.cpu().numpy().view(np.uint32), want), q
        assert np.array_equal(mb.mb_rescue_prefilter(r, ro, w, wo, q=q), want), q


def test_decreasing_offsets_are_refused(mb):
    r, w = np.zeros(300, np.uint8), np.zeros(900, np.uint8)
    good, bad = np.array([0, 100, 200, 300], np.uint64), np.array([0, 100, 90, 300], np.uint64)
    wo = np.array([0, 300, 600, 900], np.uint64)
    for ro, wins in ((bad, wo), (good, np.array([0, 300, 900, 600], np.uint64))):
        for f in (lambda a: a, dev):
            with pytest.raises(mb.MbError) as e:
                mb.mb_rescue_prefilter(f(r), f(ro), f(w), f(wins))
            assert e.value.code == -1 and b"decrease" in mb.lib().mb_last_error()


def test_host_offsets_that_the_stream_still_writes(mb):
    """Pinned offsets that hold a small batch's values until earlier work of the call's stream replaces them:
    the sizes of the launch are those of the new values."""
    rng = np.random.default_rng(8)
    lens, wlens = rng.integers(100, 251, 400), rng.integers(300, 3000, 400)
    ro, wo = (np.concatenate([[0], np.cumsum(x)]) for x in (lens, wlens))
    r, w = rng.integers(0, 4, ro[-1]).astype(np.uint8), rng.integers(0, 4, wo[-1]).astype(np.uint8)
    for p in range(0, 400, 2):   # half of the reads come from their window
        r[ro[p]:ro[p + 1]] = w[wo[p] + 20:wo[p] + 20 + lens[p]]
    want = oracle.qmer_diag_max_batch(r, ro.astype(np.uint64), w, wo.astype(np.uint64), 7)
    new = [torch.from_numpy(x).cuda() for x in (ro, wo)]
    pinned = [torch.from_numpy(np.arange(401) * k).pin_memory() for k in (8, 16)]
    dr, dw = dev(r), dev(w)
    best = torch.empty(400, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(100_000_000)   # about 50 ms before the new offsets arrive
        for a, b in zip(pinned, new):
            a.copy_(b, non_blocking=True)
        mb.mb_rescue_prefilter(dr, pinned[0], dw, pinned[1], best=best, stream=st.cuda_stream)
    assert np.array_equal(best.cpu().numpy().view(np.uint32), want)


@pytest.mark.parametrize("m", [100, 300])
def test_calls_of_several_threads(mb, m):
    """Threads whose windows need 60 to 210 kB of shared memory per block, each on its own stream (reads in the
    register form, and past it)."""
    import threading
    rng = np.random.default_rng(m)
    work, errors = [], []
    for w in (18_000, 30_000, 42_000, 55_000):
        ro, wo = np.arange(9, dtype=np.uint64) * m, np.arange(9, dtype=np.uint64) * w
        r, x = rng.integers(0, 4, 8 * m).astype(np.uint8), rng.integers(0, 4, 8 * w).astype(np.uint8)
        want = torch.from_numpy(oracle.qmer_diag_max_batch(r, ro, x, wo, 7).view(np.int32)).cuda()
        work.append((dev(r), dev(ro), dev(x), dev(wo), want, torch.cuda.Stream()))
    torch.cuda.synchronize()

    def calls(r, ro, x, wo, want, st):
        try:
            best = torch.empty(8, dtype=torch.int32, device="cuda")
            for _ in range(150):
                mb.mb_rescue_prefilter(r, ro, x, wo, best=best, stream=st.cuda_stream)
                st.synchronize()
            with torch.cuda.stream(st):
                assert torch.equal(best, want)
        except Exception as e:   # noqa: BLE001 - reported by the test
            errors.append(e)

    threads = [threading.Thread(target=calls, args=a) for a in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
