"""Synchronous parity at the kernels' edges on graphs large enough, or of the weights, that reach each kernel."""
import numpy as np
import pytest

from engine_util import assert_sync_parity, engine_run
from test_degree_edges_gpu import _Csr
from test_pull_activity_gpu import _Stars

pytestmark = pytest.mark.gpu


def _edges(degrees, copies, wmax, pool=9000, seed=7):
    """`copies` vertices of each degree, joined to a pool of 9,000 vertices in groups of 12: more vertices than a
    block takes."""
    rng = np.random.default_rng(seed)
    d = np.repeat(degrees, copies)
    u = np.repeat(np.arange(len(d)), d)
    v = np.concatenate([rng.integers(0, pool - x) + np.arange(x) for x in d])   # neighbours next to each other
    a = rng.integers(0, pool, 2 * pool)
    b = np.minimum(a // 12 * 12 + rng.integers(0, 12, len(a)), pool - 1)
    k, n = len(d), len(d) + pool
    u, v = np.concatenate([u, k + a[a != b]]), np.concatenate([k + v, k + b[a != b]])
    pair = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    g = _Csr(n, pair // n, pair % n, rng.integers(1, wmax + 1, len(pair)))
    assert np.array_equal(np.diff(g.off)[:k], d)
    return g


LOW = [1, 2, 4, 5, 7, 8, 9, 16, 31, 32, 33, 64, 65, 127, 128]


@pytest.mark.parametrize("wmax", [1, 100_000, 1 << 30])   # M below 2^31; above, 64-bit gains; 128-bit gains
@pytest.mark.parametrize("degrees", [LOW, LOW + [129]], ids=["one-launch-classes", "launch-per-bucket"])
@pytest.mark.parametrize("opt", [{}, {"prune": 1, "subrounds": 3}], ids=["plain", "pruned"])
def test_low_degrees(degrees, wmax, opt):
    assert_sync_parity(_edges(degrees, 37, wmax), max_iterations=5, max_passes=2, **opt)


@pytest.mark.parametrize("classes", [1, 3])
@pytest.mark.parametrize("wmax", [3, 1 << 29])
def test_flags_at_low_degrees(wmax, classes):
    # stars of every low degree, settled early, beside moving rings; one row above 128 keeps the pass on the
    # kernels that read the flags
    g = _Stars([5, 8, 9, 16, 32, 33] * 40 + [200], 30000, wmax, 5)
    assert_sync_parity(g, prune=1, max_passes=1, max_iterations=8, subrounds=classes)
    opt = dict(mode=0, prune=1, max_passes=1, max_iterations=4, tolerance=0.0, subrounds=classes)
    got, ref = engine_run(g, **opt), engine_run(g, stop_rule=1, **opt)   # stop rule 1 keeps the stamps
    assert len(ref["iters"]) == 4 and ref["iters"] == got["iters"]
    for f in ("lm_vertices", "lm_edges", "lm_bytes"):
        assert getattr(ref["stats"], f) == getattr(got["stats"], f), f


def _spokes(n, degrees, pairs, wlo, whi, seed=3):
    rng = np.random.default_rng(seed)
    k = len(degrees)
    u = [np.full(d, i) for i, d in enumerate(degrees)] + [k + 2 * np.arange(pairs)]
    v = [k + rng.choice(n - k, d, replace=False) for d in degrees] + [k + 1 + 2 * np.arange(pairs)]
    u, v = np.concatenate(u), np.concatenate(v)
    pair = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    return _Csr(n, pair // n, pair % n, rng.integers(wlo, whi + 1, len(pair)))


@pytest.mark.parametrize("classes", [1, 2, 8])
@pytest.mark.parametrize("prune", [0, 1])
@pytest.mark.parametrize("n,degrees", [(1025, [129, 500]), (3000, [129, 130, 256, 1000]), (8192, [2000])], ids=str)
def test_one_block_with_long_rows(n, degrees, prune, classes):
    assert_sync_parity(_spokes(n, degrees, 500, 1, 9), prune=prune, subrounds=classes)


@pytest.mark.parametrize("n", [900, 2000])
def test_one_block_with_large_totals(n):
    # M above 2^31, every degree suited to 64-bit gains and 32-bit sums
    rng = np.random.default_rng(n)
    u = np.arange(n)
    g = _Csr(n, np.concatenate([u[:-1], u[:-7:3]]), np.concatenate([u[1:], u[7::3]])[:n - 1 + len(u[:-7:3])],
             rng.integers(1, 6_000_000, n - 1 + len(u[:-7:3])))
    K = np.add.reduceat(g.w.astype(np.int64), g.off[:-1])
    assert int(K.sum()) > 1 << 32 and int(K.max()) <= (1 << 61) // int(K.sum())
    for opt in ({}, {"prune": 1, "subrounds": 4}, {"colour_classes": 1}):
        assert_sync_parity(g, **opt)


@pytest.mark.parametrize("hubs", [6, 30])   # insert chunks of 1,024 entries; from 16 hubs of one class on, of 4,096
@pytest.mark.parametrize("wmax", [3, 1 << 29])
@pytest.mark.parametrize("opt", [{"prune": 0}, {"prune": 1}, {"prune": 1, "subrounds": 3}], ids=str)
def test_hub_chunks(hubs, wmax, opt):
    # degrees at the ends of both chunk lengths
    degrees = np.resize([12289, 13312, 13313, 16383, 16384, 16385], hubs)
    assert_sync_parity(_edges(degrees, 1, wmax, pool=20000), max_iterations=4, max_passes=2, **opt)
