"""Window statistics on both sides of the longest window whose starts are
summed from groups of points (16384): means and deviations against numpy's
two-pass float64 values.  A mean's rounding is some 2^-53 of the largest
point, a variance's some 2^-53 of the mean square about the run's first point
(within a factor 100 of the variance here): 1e-12 covers both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("w", [16368, 16384, 16385, 20011])
def test_statistics_of_long_windows(w, dtype):
    from paper_2502_14446_gb300 import build_ext, momenti
    build_ext.build()
    rng = np.random.default_rng(w)
    T = (rng.standard_normal((2, w + 203)) + np.array([[0.0], [5.0]])).astype(dtype)
    T[1, 40] += 30.0
    with momenti.Momenti(w=w, d=1, k=1, delta=0.1, L=1) as h:
        h.hash_all(T)
        mu, sd = h.window_stats()
    W = np.lib.stride_tricks.sliding_window_view(T.astype(np.float64), w, axis=1)
    np.testing.assert_allclose(mu, W.mean(axis=2), rtol=0, atol=1e-12 * np.abs(T).max())
    np.testing.assert_allclose(sd, W.std(axis=2), rtol=1e-12)
