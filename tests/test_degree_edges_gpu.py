"""Synchronous parity at the degrees where the local-moving kernels change hands."""
import numpy as np
import pytest

from engine_util import assert_sync_parity

pytestmark = pytest.mark.gpu


class _Csr:
    def __init__(self, n, u, v, w):
        key = np.concatenate([u * n + v, v * n + u])
        o = np.argsort(key, kind="stable")
        self.n = n
        self.off = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int64)
        self.col = (key[o] % n).astype(np.int32)
        self.w = np.concatenate([w, w])[o].astype(np.int32)
        self.nnz = len(self.col)


def _stars(degrees, wmax, seed):
    """One vertex of each degree, joined to random others of a pool of small random communities."""
    rng = np.random.default_rng(seed)
    k, pool = len(degrees), max(degrees) + 64
    u, v = [], []
    for i, d in enumerate(degrees):
        leaf = rng.choice(pool, d, replace=False)
        u.append(np.full(d, i))
        v.append(k + leaf)
    for _ in range(2):
        a = rng.integers(0, pool, pool)
        b = (a // 16 * 16 + rng.integers(0, 16, pool)) % pool
        u.append(k + a[a != b])
        v.append(k + b[a != b])
    u, v = np.concatenate(u), np.concatenate(v)
    n = k + pool
    pair = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    return _Csr(n, pair // n, pair % n, rng.integers(1, wmax + 1, len(pair)))


EDGES = [[1, 8, 9, 31, 32, 33, 64, 127, 128, 129], [256, 1000, 1024, 1025, 2048, 4095, 4096],
         [4097, 6144, 6145, 8191, 12287], [12288, 12289, 16384, 16385]]


@pytest.mark.parametrize("wmax", [1, 8, 200000, 1 << 30])   # 128-bit gains: of some vertices, of all
@pytest.mark.parametrize("degrees", EDGES, ids=["-%d" % max(d) for d in EDGES])
def test_degrees_at_bucket_edges(degrees, wmax):
    assert_sync_parity(_stars(degrees, wmax, 11), prune=1, max_iterations=6, max_passes=3)
