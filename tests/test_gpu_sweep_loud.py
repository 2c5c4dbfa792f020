"""Series whose loudness changes: the recording sweep's running sums carry
what was rounded away in a loud stretch into the quiet rows after it.  What a
sweep records is held against the distances in float64, for every pair:
every pair whose exact distance x has 1.01 x + 0.01 below the edge is recorded,
at most that far out, and none nearer than the table's allowance lets it be
(2 kappa <= 2e-3 in the correlation of each dimension: at most sqrt(4e-3 w)
per dimension).  Bursts, level steps, constant stretches and walks; pairs planted on the
lag of two bursts, a few hundred to two thousand rows after them; every form
of the launch."""
import numpy as np
import pytest

from oracle import momenti_oracle as O
from paper_2502_14446_gb300 import synth

pytestmark = pytest.mark.gpu

N, LAG, B0, BLEN = 6000, 3000, 600, 500
GAPS = (300, 700, 1100, 1700)


def series(kind, ratio, D, w, dtype, seed=5):
    rng = np.random.default_rng(seed)
    T = rng.standard_normal((D, N))
    if kind == "walk":
        T = np.cumsum(T, axis=1)
    for gap in GAPS:                                # the planted pairs
        a = B0 + BLEN + gap
        T[:, a + LAG:a + LAG + w] = T[:, a:a + w] + 0.01 * rng.standard_normal((D, w))
    for b in (B0, B0 + LAG):
        if kind == "burst":
            T[:, b:b + BLEN] *= ratio
        elif kind == "level":
            T[:, b:b + BLEN] += ratio
        elif kind == "spike":
            T[0, b:b + BLEN:23] += ratio
    if kind == "flat":
        T[0, B0:B0 + BLEN] = 3.5
        T[D - 1, B0 + LAG + 40:B0 + LAG + BLEN] = -1.25
    return np.ascontiguousarray(T, dtype=dtype)


def exact_distances(T, w, d, excl):
    """dist_d of every non-trivial pair (a < b), float64, as (M, M) with inf elsewhere."""
    T = T.astype(np.float64)
    M = T.shape[1] - w + 1
    Z, n2 = [], []
    for x in T:
        W = np.lib.stride_tricks.sliding_window_view(x, w)
        mu = W.mean(axis=1)
        c = W - mu[:, None]
        sd = np.sqrt((c * c).mean(axis=1))
        flat = sd <= 1e-8 * (1 + np.abs(mu))
        Z.append(np.where(flat[:, None], 0.0, c / np.where(flat, 1.0, sd)[:, None]))
        n2.append(np.where(flat, 0.0, float(w)))
    out = np.full((M, M), np.inf)
    for r in range(0, M, 500):
        per = np.stack([np.sqrt(np.maximum(n[r:r + 500, None] + n[None, :] - 2.0 * (z[r:r + 500] @ z.T), 0.0))
                        for z, n in zip(Z, n2)])
        out[r:r + 500] = (np.partition(per, d - 1, axis=0)[:d] if d < len(per) else per).sum(axis=0)
    a, b = np.indices((M, M), sparse=True)
    return np.where(b - a > excl, out, np.inf)


KINDS = [("burst", 300.0), ("burst", 3000.0), ("burst", 30.0), ("level", 1000.0), ("spike", 3000.0), ("flat", 0.0),
         ("walk", 0.0)]
CASES = ([(*k, 2, 2, 2048, np.float32) for k in KINDS] + [(*k, 1, 1, 2048, np.float32) for k in KINDS[:2]] +
         [(*k, 2, 1, 0, np.float32) for k in KINDS[3:]] + [(*k, 2, 2, 1, np.float64) for k in KINDS[1:6:2]] +
         [(*k, 5, 3, 512, np.float64) for k in KINDS[:6:2]] + [(*k, 5, 2, 0, np.float32) for k in KINDS[3:6:2]] +
         [(*k, 8, 3, 2048, np.float32) for k in KINDS[1::5]] + [("burst", 3000.0, 28, 6, 2048, np.float32)])


@pytest.mark.parametrize("kind,ratio,D,d,form,dtype", CASES)
def test_every_near_pair_is_recorded(kind, ratio, D, d, form, dtype):
    from sweep_client import sweep
    w = 48
    T = series(kind, ratio, D, w, dtype)
    x = exact_distances(T, w, d, w // 2)
    hi = float(np.quantile(x[np.isfinite(x)][::7], 2e-3))
    hi = max(hi, 0.5 * d)
    pairs, dist = sweep(T, w, d, -1.0, hi, form=form)
    a, b = (pairs >> 32).astype(np.int64), (pairs & 0xffffffff).astype(np.int64)
    rec = np.full(x.shape, np.inf)
    rec[a, b] = dist
    assert len(np.unique(pairs)) == len(pairs)
    assert np.isfinite(x[a, b]).all()
    bound = 1.01 * x + 0.01
    need = bound <= hi
    assert need.sum() > 500
    far = need & ~(rec <= bound)
    assert far.sum() == 0, (int(far.sum()), np.argwhere(far)[:4].tolist(), x[far][:4], rec[far][:4])
    near = dist < x[a, b] - d * np.sqrt(4e-3 * w) - 1e-3
    assert near.sum() == 0, (int(near.sum()), a[near][:4], b[near][:4], x[a, b][near][:4], dist[near][:4])


@pytest.mark.parametrize("kind,ratio", [("burst", 3000.0), ("level", 1000.0)])
def test_exact_search_after_a_loud_stretch(kind, ratio):
    from paper_2502_14446_gb300 import momenti
    w, d, k = 48, 2, 12
    T = series(kind, ratio, 3, w, np.float32)
    with momenti.Momenti(w=w, d=d, k=k, delta=0.05, L=1) as h:
        h.hash_all(T)
        got = h.topk_exact()
    ref = O.exact_topk(T, w, d, k)
    assert [(m["a"], m["b"]) for m in got] == [(m[1], m[2]) for m in ref]
    for g, r in zip(got, ref):
        assert g["dist_d"] == pytest.approx(r[0], rel=1e-9, abs=1e-9)
