"""The exact path's table of a wide series (800 bytes a window at D = 40, more
than the record buffers here) lies inside the memory that the handle planned
and reports, not beside it: what the device holds beyond device_bytes while
the exact path has run is its record buffers (2^24 pairs of 8 + 4 bytes, an
8-byte selection of those found) and small change, 64 MB."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,dtype", [(40, np.float32), (33, np.float64)])
def test_exact_path_stays_inside_the_planned_memory(D, dtype):
    import torch
    from paper_2502_14446_gb300 import build_ext, momenti
    build_ext.build()
    n, w = 400_000, 32
    rng = np.random.default_rng(7)
    T = np.cumsum(rng.standard_normal((D, n)), axis=1).astype(dtype)
    T[:, n - w:] = T[:, :w] + 1e-3 * rng.standard_normal((D, w))
    limit = 12 << 30
    torch.zeros(1, device="cuda")
    with momenti.Momenti(w=w, d=D, k=1, delta=0.05, L=1, mem_limit=limit) as h:
        free0 = torch.cuda.mem_get_info()[0]
        h.hash_all(T)
        torch.cuda.synchronize()
        free1 = torch.cuda.mem_get_info()[0]
        got = h.topk_exact()
        torch.cuda.synchronize()
        free2 = torch.cuda.mem_get_info()[0]
        assert free0 - free1 <= limit
        assert free1 - free2 <= (1 << 24) * 20 + (64 << 20), (free1 - free2) >> 20
    assert (got[0]["a"], got[0]["b"]) == (0, n - w)
