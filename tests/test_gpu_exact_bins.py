"""The exact path verifies the recorded pairs in batches of whole histogram
bins.  All dimensions constant over a stretch: 101475 pairs lie at distance 0,
and with w = 100 and d = 3 the first edge is 5% of the largest distance, 3, so
that 0 is exactly the lower edge of a bin, whose pairs alone fill a batch.
The three motifs are the first pairs of the stretch that do not overlap."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_pairs_on_the_edge_of_a_bin_are_verified():
    from paper_2502_14446_gb300 import build_ext, momenti
    build_ext.build()
    rng = np.random.default_rng(3)
    T = np.cumsum(rng.standard_normal((4, 30_000)), axis=1)
    T[:, 20010:20110] = T[:, 1010:1110] + 0.01 * rng.standard_normal((4, 100))
    T[:, 3000:3600] = T[:, 3000:3001]
    with momenti.Momenti(w=100, d=3, k=3, delta=0.05, L=1) as h:
        h.hash_all(T.astype(np.float32))
        got = h.topk_exact()
    assert [(m["a"], m["b"], m["dist_d"]) for m in got] == [(3000, 3051, 0.0), (3102, 3153, 0.0), (3204, 3255, 0.0)]
