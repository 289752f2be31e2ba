"""Calls on a nearly full device: an allocation that is refused gives its error (or, for the optional
deeper k-mer table, none), and nothing of it is left for the next call to find."""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
MB = 1 << 20


@pytest.fixture(scope="module")
def mb():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_15357_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def tiny(mb):
    """A small index with one record and its hits on the device."""
    ref, _, _ = synth.workload(1, scale=0.01)
    sm = np.zeros(1, dtype=mb.SMEM_DTYPE)
    sm["qend"], sm["s"] = 20, 100
    return dict(ref=ref, G=mb.mb_index_build(ref), sm=torch.from_numpy(sm.view(np.uint8)).cuda(),
                hits=torch.zeros(100, dtype=torch.int32, device="cuda"),
                keep=torch.zeros(100, dtype=torch.uint8, device="cuda"))


def next_call(mb, t):
    """The call that follows: one kernel, no allocation, and nothing that would drop an earlier error."""
    return mb.lib().mb_bs_filter(t["G"].handle, mb._ptr(t["sm"]), 1, None, mb._ptr(t["hits"]), 100, None,
                                 mb._ptr(t["keep"]))


def leave(mb, tiny, room):
    """The rest of the device taken but for `room` bytes; the library's pool given back first."""
    mb.mb_index_build(tiny["ref"][:1000], opts=dict(kmer_k=4))   # a build ends by trimming the pool
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - room, dtype=torch.uint8, device="cuda")


def test_a_refused_call_leaves_no_error_behind(mb, tiny):
    sm = np.zeros(1, dtype=mb.SMEM_DTYPE)
    sm["s"] = 1 << 38   # a terabyte of hits, staged on the device for a host array
    hits, nh, o = np.zeros(4, np.uint32), ctypes.c_uint64(), mb.Opts(max_occ=1)
    rc = mb.lib().mb_locate(tiny["G"].handle, mb._ptr(sm), 1, ctypes.byref(o), None, mb._ptr(hits), 1 << 40, ctypes.byref(nh))
    after = next_call(mb, tiny)
    assert rc == -2 and nh.value == 1 << 38 and after == 0 and bool(tiny["keep"].all())


def test_load_with_little_room(mb, tiny, tmp_path):
    """20 Mbp at k = 4: 115 MB of index, a deeper table of 201 MB and 63 MB to make it with.  At every room
    the load succeeds from the index's own size on, and calls after it (or after its refusal) work."""
    ref = np.random.default_rng(3).integers(0, 4, 20_000_000).astype(np.uint8)
    G = mb.mb_index_build(ref, opts=dict(kmer_k=4))
    G.save(str(tmp_path / "i.mbi"))
    G.free()
    loaded = []
    for room in range(64 * MB, 480 * MB, 24 * MB):
        rest = leave(mb, tiny, room)
        try:
            X, rc = mb.mb_index_load(str(tmp_path / "i.mbi")), 0
        except mb.MbError as e:
            X, rc = None, e.code
        after = next_call(mb, tiny)
        assert rc in (0, -2) and after == 0, (room, rc, after)
        if X is not None:
            X.free()
        del rest
        torch.cuda.empty_cache()
        loaded.append(rc == 0)
    assert loaded[-1] and not loaded[0] and loaded == sorted(loaded)


def test_more_room_never_builds_less(mb, tiny):
    """The optional table takes no array's room: from the smallest room in which a build succeeds on, every
    larger one does too."""
    ref = np.random.default_rng(4).integers(0, 4, 20_000_000).astype(np.uint8)
    built = []
    for room in range(1000 * MB, 1660 * MB, 60 * MB):
        rest = leave(mb, tiny, room)
        try:
            mb.mb_index_build(ref, opts=dict(kmer_k=4)).free()
            rc = 0
        except mb.MbError as e:
            rc = e.code
        assert next_call(mb, tiny) == 0 and rc in (0, -2)
        del rest
        torch.cuda.empty_cache()
        built.append(rc == 0)
    assert built[-1] and not built[0] and built == sorted(built)


def test_the_deeper_table_can_be_declined(mb, tiny, tmp_path):
    """MB_NO_KMER at the build: 201 MB less at 20 Mbp and k = 4, also after a load; the same records."""
    ref = np.random.default_rng(5).integers(0, 4, 20_000_000).astype(np.uint8)
    rd = synth.reads(ref, 2000, 6, mode=1, read_len=150, sub_lo=0.001, sub_hi=0.01, indel=0.0001)
    used, recs = [], []
    for flags in (0, mb.MB_NO_KMER):
        for load in (False, True):
            torch.cuda.empty_cache()
            before = torch.cuda.mem_get_info()[0]
            if load:
                G = mb.mb_index_load(str(tmp_path / f"{flags}.mbi"))
            else:
                G = mb.mb_index_build(ref, opts=dict(kmer_k=4, flags=flags))
                G.save(str(tmp_path / f"{flags}.mbi"))
                G.drop_sa()
            mb.mb_index_build(tiny["ref"][:1000], opts=dict(kmer_k=4)).free()   # trims the pool
            used.append(before - torch.cuda.mem_get_info()[0])
            recs.append(mb.mb_seed_batch(G, rd.seq, rd.off)[0].tobytes())
            G.free()
            mb.mb_index_build(tiny["ref"][:1000], opts=dict(kmer_k=4)).free()
    table = 12 * 4 ** 12
    assert abs(used[0] - used[2] - table) < 8 * MB and abs(used[1] - used[3] - table) < 8 * MB
    assert len(set(recs)) == 1
