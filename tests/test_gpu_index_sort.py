"""The index sort's branches on keys made for them, against a host stable
sort: bins of one entry, crowded bins (the network), chunks in order already,
buckets above and below a chunk's size, equal keys, short keys, ragged sizes."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mom():
    from paper_2502_14446_gb300 import build_ext
    build_ext.build()
    from paper_2502_14446_gb300 import momenti
    return momenti


def make_keys(kind, m, K):
    g = np.random.default_rng(m * 8 + K)
    b = g.integers(0, 256, size=(m, 8))
    if kind == "normal":                      # rounded normals, as hash values are
        b = np.clip(np.rint(g.standard_normal((m, 8)) * 25 + 128), 0, 255).astype(int)
    elif kind == "few":                       # many equal keys among few distinct ones
        b = g.integers(0, 3, size=(m, 8)) + 126
    elif kind == "equal":
        b[:] = 77
    elif kind == "first":                     # only the first value differs
        b[:, 1:] = 9
    elif kind == "last":                      # only the last of K values differs
        b[:, :K - 1] = 200
    elif kind == "tail":                      # alike in the leading values, distinct below
        b[:, :3] = g.integers(0, 2, size=(m, 3))
    b[:, K:] = 0
    key = np.zeros(m, dtype=np.uint64)
    for q in range(8):
        key |= b[:, q].astype(np.uint64) << np.uint64(56 - 8 * q)
    return key


@pytest.mark.parametrize("kind", ["random", "normal", "few", "equal", "first", "last", "tail"])
@pytest.mark.parametrize("m,K", [(1, 8), (2, 8), (33, 1), (2047, 8), (2048, 3), (2049, 8), (4097, 2), (70001, 8)])
def test_order_and_prefixes(mom, kind, m, K):
    import torch
    key = make_keys(kind, m, K)
    kt = torch.from_numpy(key.view(np.int64)).cuda()
    order = torch.full((m,), -1, dtype=torch.int32, device="cuda")
    lcp = torch.full((m,), 255, dtype=torch.uint8, device="cuda")
    rc = mom.lib.momenti_index_sort_noalloc(C.c_void_p(kt.data_ptr()), m, K, C.c_void_p(order.data_ptr()),
                                            C.c_void_p(lcp.data_ptr()),
                                            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == mom.OK
    torch.cuda.synchronize()
    ref = np.argsort(key, kind="stable")
    s = key[ref]
    pre = np.zeros(m, dtype=np.uint8)
    same = np.full(max(m - 1, 0), K, dtype=np.uint8)
    x = s[1:] ^ s[:-1]
    for q in range(K - 1, -1, -1):
        same[(x >> np.uint64(56 - 8 * q)) & np.uint64(255) != 0] = q
    pre[1:] = same
    np.testing.assert_array_equal(order.cpu().numpy(), ref.astype(np.int32))
    np.testing.assert_array_equal(lcp.cpu().numpy(), pre)
