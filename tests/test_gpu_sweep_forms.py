"""Every form of the recording sweep records the same pairs: the plain launch
(lane groups as a constant, 1 or 2 pairs of dimensions per lane), the batching
form's and blocks of 32 to 2048 rows (lane groups at run time).  The forms'
sums are rounded differently: correlations differ by at most 2 kappa, which is
below 1e-4 on these walks (kappa = 4 e^2 / 2^24, e below 14 over 2000 windows
of w = 64 points of noise), so a dimension's distance by at most
sqrt(2e-4 w) = 0.12, and a pair that one form leaves out lies within d times
that of the edge."""
import numpy as np
import pytest

from paper_2502_14446_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,d", [(1, 1), (2, 2), (4, 2), (5, 3), (8, 3), (16, 4), (27, 5), (40, 8)])
def test_forms_record_the_same_pairs(D, d):
    from sweep_client import sweep
    w, n = 64, 5003
    rng = np.random.default_rng(D)
    T = rng.standard_normal((D, n))
    for a, b in ((100, 3000), (1200, 4111)):
        T[:, b:b + 2 * w] = T[:, a:a + 2 * w] + 0.05 * rng.standard_normal((D, 2 * w))
    T = T.astype(np.float32)
    lo, hi = 0.0, 2.0 * np.sqrt(w) * d
    while hi - lo > 0.01 * d:                     # an edge with some 20000 pairs
        mid = 0.5 * (lo + hi)
        if len(sweep_or_many(sweep, T, w, d, mid)) > 20000:
            hi = mid
        else:
            lo = mid
    forms = {f: dict(zip(*map(np.ndarray.tolist, sweep(T, w, d, -1.0, lo, form=f)))) for f in (0, 1, 32, 256, 2048)}
    tol = d * np.sqrt(2e-4 * w)
    assert len(forms[0]) > 100
    for f, got in forms.items():
        for p in forms[0].keys() ^ got.keys():
            assert (forms[0].get(p) or got.get(p)) > lo - tol, (f, p)
        assert max(abs(forms[0][p] - got[p]) for p in forms[0].keys() & got.keys()) <= tol


def sweep_or_many(sweep, T, w, d, thr):
    try:
        return sweep(T, w, d, -1.0, thr, cap=1 << 18)[0]
    except AssertionError:                        # more than the buffer holds
        return range(1 << 18)
