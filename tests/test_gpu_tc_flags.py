"""The tensor-core form's keys where the lanes of a warp flag different numbers
of values: half of the offsets are 0 and r is 2^11 standard deviations of a
projection, so about two in three of those values lie within 2^-11 of a bucket
boundary.  The keys must be the FP32 form's, bit for bit."""
import numpy as np
import pytest

from paper_2502_14446_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,K", [(16, 8), (37, 5)])
def test_keys_with_many_flagged_values(L, K):
    from paper_2502_14446_gb300 import build_ext, momenti
    build_ext.build()
    wl = synth.tiny(41, n=260, D=2, w=64, d=2, k=2, n_motifs=1)
    A, U = synth.hash_draws(wl.D, L, K, wl.w, 11)
    U[:, :, ::2] = 0.0
    r = 2048.0 * np.sqrt(wl.w)
    keys = {}
    for precision in (momenti.PREC_FP32, momenti.PREC_F16X2):
        with momenti.Momenti(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta, K=K, L=L, r=r, precision=precision) as h:
            h.set_hash_params(A, U)
            h.hash_all(wl.series)
            _, st = h.topk()
            assert st["precision_used"] == precision
            keys[precision] = [h.keys(j) for j in range(L)]
    assert st["n_rehashed"] > 0.2 * (wl.n - wl.w + 1) * wl.D * L * K
    for j in range(L):
        np.testing.assert_array_equal(keys[momenti.PREC_F16X2][j], keys[momenti.PREC_FP32][j])
