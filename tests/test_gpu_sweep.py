"""The recording sweep of the exact path at the sizes where its layout can
go wrong: every number of dimension groups per diagonal (1 to 64
dimensions), both element types, lengths that leave partial 64-window
blocks, 8-row groups and diagonal blocks, series shorter than one block,
exclusion zones from 0 to nearly all pairs.  The exact top-k must be the
oracle's: pairs and dimension sets identical, distances 1e-9 relative (they
are re-verified in float64)."""
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


def check(mom, wl, **kw):
    with mom.Momenti(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta, L=1, **kw) as h:
        h.hash_all(wl.series)
        got = h.topk_exact()
    ref = O.exact_topk(wl.series, wl.w, wl.d, wl.k, kw.get("excl"))
    if ref is None:                       # fewer than k non-trivial motifs: the oracle's top-m, and no (m + 1)-th
        m = len(got)
        assert 0 < m < wl.k and O.exact_topk(wl.series, wl.w, wl.d, m + 1, kw.get("excl")) is None
        ref = O.exact_topk(wl.series, wl.w, wl.d, m, kw.get("excl"))
    assert [(m["a"], m["b"]) for m in got] == [(m[1], m[2]) for m in ref]
    for g, r in zip(got, ref):
        assert g["dist_d"] == pytest.approx(r[0], rel=1e-9, abs=1e-9)
        assert g["dims"] == tuple(r[3])


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 17, 21, 25, 31, 33, 49, 64])
def test_every_group_count(mom, D, dtype):
    wl = synth.tiny(60 + D, n=1171 + 7 * D, D=D, w=29, d=max(1, D // 3), k=3, n_motifs=2, dtype=dtype)
    check(mom, wl)


@pytest.mark.parametrize("n", [40, 64, 71, 129, 513, 1000])
def test_short_series(mom, n):
    wl = synth.tiny(80 + n, n=n, D=3, w=12, d=2, k=2, n_motifs=0, dtype=np.float32)
    check(mom, wl)


@pytest.mark.parametrize("excl", [0, 7, 8, 700])
def test_exclusion_zones(mom, excl):
    wl = synth.tiny(90, n=900, D=5, w=40, d=2, k=2, n_motifs=0, dtype=np.float32)
    check(mom, wl, excl=excl)


def test_several_segments_and_tails(mom):
    # several row blocks and diagonal blocks, staged rows, ragged tails
    wl = synth.tiny(92, n=6007, D=2, w=33, d=1, k=3, n_motifs=2, dtype=np.float32)
    check(mom, wl)
