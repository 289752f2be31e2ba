"""The L2 access-policy window lies over the k-mer table that seeding reads."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_window_covers_the_table_in_use():
    """1 Mbp at k = 4: the index keeps a table of k = 10 for seeding (12.6 MB) beside the 3 kB one; without it
    (MB_NO_KMER) the window is the 3 kB."""
    import paper_2606_15357_gb300 as mb
    ref = np.random.default_rng(1).integers(0, 4, 1_050_000).astype(np.uint8)
    for flags, k in ((0, 10), (mb.MB_NO_KMER, 4)):
        G = mb.mb_index_build(ref, opts=dict(kmer_k=4, flags=flags))
        st = torch.cuda.Stream()
        try:
            assert G.l2_persist(1 << 40, stream=st.cuda_stream) == 12 * 4 ** k
            assert G.l2_persist(1000, stream=st.cuda_stream) == 1000
        finally:
            assert G.l2_persist(0, stream=st.cuda_stream) == 0
