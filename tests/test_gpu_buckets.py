"""Bucket lists and candidate tiles on indexes whose segments start at every
byte alignment and end inside a 32-rank word or a 1024-rank warp, against
brute force on the keys.  With one repetition every pair with W >= d at
prefix length 1 is a candidate of the tile form exactly once (at the longest
prefix where W >= d); the bucket form finds all of them (some twice), so
the verified pairs, and with them the motifs of the traversal, agree."""
import numpy as np
import pytest

from oracle import momenti_oracle as O
from paper_2502_14446_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mom():
    from paper_2502_14446_gb300 import build_ext
    build_ext.build()
    from paper_2502_14446_gb300 import momenti
    return momenti


@pytest.mark.parametrize("D,n", [(3, 60), (4, 1055), (5, 1056), (7, 1057), (8, 2079), (9, 1100), (11, 1301), (16, 1090)])
@pytest.mark.parametrize("r", [1.0, 8.0, 60.0])
def test_candidates_against_brute_force(mom, D, n, r):
    # r from narrow (buckets of a few windows) to wide (one bucket holds most)
    wl = synth.tiny(100 + D, n=n, D=D, w=24, d=2, k=2, n_motifs=0)
    top = []
    for flags in (0, mom.FLAG_TILES_ONLY):
        with mom.Momenti(w=wl.w, d=wl.d, k=wl.k, delta=1e-12, K=4, L=1, r=r,
                         flags=flags | mom.FLAG_NO_COST_SWITCH) as h:
            h.hash_all(wl.series)
            h.search_begin()
            while not h.search_step(1):
                pass
            now, _ = h.search_current()
            top.append([(m["a"], m["b"], m["dist_d"]) for m in now[wl.d]])
            _, st = h.search_finish()
            keys, M = h.keys(0), h.info()["M"]
            pairs = {tuple(p) for p in h.collide(2, 0)}
        a, b = np.triu_indices(M, k=O.exclusion_zone(wl.w) + 1)
        w1 = ((keys[a] >> np.uint64(56)) == (keys[b] >> np.uint64(56))).sum(axis=1)
        n1 = int((w1 >= wl.d).sum())
        assert st["n_candidates"] == n1 if flags else st["n_candidates"] >= n1
        ok = ((keys[a] >> np.uint64(48)) == (keys[b] >> np.uint64(48))).sum(axis=1) >= wl.d
        assert pairs == set(zip(a[ok].tolist(), b[ok].tolist()))
    assert top[0] == top[1]
