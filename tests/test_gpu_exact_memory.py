"""An exact search that fails gives everything back: a constant series, whose
1.1e9 pairs all lie at distance 0, overflows the record buffers' largest size
(2^30 pairs) and the search returns an error.  Nothing of its buffers may stay
behind in the library's pool once the handle is gone (a pool block is 2 MB)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_a_failed_exact_search_leaves_nothing_behind():
    import torch
    from paper_2502_14446_gb300 import build_ext, momenti
    build_ext.build()

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def search(T, fails):
        with momenti.Momenti(w=16, d=1, k=3, delta=0.05, L=1) as h:
            h.hash_all(T)
            if not fails:
                return h.topk_exact()
            with pytest.raises(momenti.MomentiError):
                h.topk_exact()

    rng = np.random.default_rng(3)
    torch.zeros(1, device="cuda")
    search(rng.standard_normal((1, 48_000)).astype(np.float32), False)
    before = free()
    for _ in range(3):
        search(np.ones((1, 48_000), np.float32), True)
    assert abs(before - free()) < 1 << 20
