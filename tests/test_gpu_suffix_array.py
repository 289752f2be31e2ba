"""The suffix array builder where its first sort and its rank writes have edges: texts shorter and longer
than the 20 symbols of a sort key, with suffixes that end within a key tied to others, and text sizes on
both sides of the line from which ranks are written in order of place."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mb():
    import paper_2606_15357_gb300 as m
    return m


def text(ref):
    return np.concatenate([ref.astype(np.int64) + 1, 4 - ref[::-1].astype(np.int64), [0]])   # $ = 0, A..T = 1..4


@pytest.mark.parametrize("unit", [(0,), (3,), (0, 3), (0, 0, 1), (1, 2), (2, 0, 1, 3, 3)])
def test_short_and_periodic_texts(mb, unit):
    for m in [1, 2, 9, 10, 11, 19, 20, 21, 22, 40, 41, 63, 64, 200]:
        ref = np.tile(np.array(unit, np.uint8), m)[:m].copy()
        t = text(ref).tolist()
        want = sorted(range(len(t)), key=lambda p: t[p:])
        assert mb.mb_index_build(ref, opts=dict(kmer_k=4)).export(sa=True)["sa"].tolist() == want, m


@pytest.mark.parametrize("m", [(1 << 23) - 1, 1 << 23, (1 << 23) + 2049])
def test_order_of_neighbours(mb, m):
    """S is sorted iff (T[S(x)], row of the suffix at S(x) + 1) increases with x."""
    ref, _, _ = synth.workload(2, scale=0.1)
    ref = np.resize(ref[ref < 4], m).astype(np.uint8)
    sa = mb.mb_index_build(ref).export(sa=True)["sa"].astype(np.int64)
    t = text(ref)
    rank = np.full(len(t) + 1, -1, np.int64)
    rank[sa] = np.arange(len(t))
    assert (rank[:-1] >= 0).all() and sa[0] == len(t) - 1
    key = t[sa] * (len(t) + 1) + rank[sa + 1] + 1
    assert (key[1:] > key[:-1]).all()
