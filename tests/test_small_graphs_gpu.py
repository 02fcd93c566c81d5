"""Graphs whose local-moving phase one block runs: sizes, degrees and weights around its limits."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from engine_util import assert_sync_parity
from paper_2301_12390_gb300 import ASYNC, SYNC, Louvain
from test_degree_edges_gpu import _Csr, _stars

pytestmark = pytest.mark.gpu


def _path(n, wmax):
    """A path with a chord every third vertex: two entries and more per vertex, few in all."""
    rng = np.random.default_rng(n)
    u = np.concatenate([np.arange(n - 1), np.arange(0, n - 7, 3)])
    v = np.concatenate([np.arange(1, n), np.arange(7, n, 3)])[: len(u)]
    return _Csr(n, u, v, rng.integers(1, wmax + 1, len(u)))


@pytest.mark.parametrize("n", [8, 1024, 1025, 6000])
@pytest.mark.parametrize("wmax", [1, 1 << 30])   # 2^30: the totals leave 32 bits, then 64-bit gains
@pytest.mark.parametrize("opt", [{}, {"prune": 1}, {"prune": 1, "subrounds": 4},
                                 {"colour_classes": 1, "singleton_guard": 0}], ids=str)
def test_sync_parity_by_size(n, wmax, opt):
    assert_sync_parity(_path(n, wmax), **opt)


@pytest.mark.parametrize("classes", [1, 8])
@pytest.mark.parametrize("degrees", [[1, 7, 8, 9, 31, 33], [64, 127, 128, 129], [129, 300, 900]], ids=str)
def test_sync_parity_by_degree(degrees, classes):
    assert_sync_parity(_stars(degrees, 8, 3), prune=1, subrounds=classes)


def test_sync_parity_at_the_entry_limit():
    # 20,480 entries is the limit of one class: graphs just below and above it
    for n in (4090, 4099):
        rng = np.random.default_rng(5)
        u = np.concatenate([np.arange(n), rng.integers(0, n, 3 * n // 2)])
        v = np.concatenate([(np.arange(n) + 1) % n, rng.integers(0, n, 3 * n // 2)])
        pair = np.unique(np.minimum(u, v)[u != v] * n + np.maximum(u, v)[u != v])
        assert_sync_parity(_Csr(n, pair // n, pair % n, np.ones(len(pair), np.int64)), prune=1)


@pytest.mark.parametrize("mode", [SYNC, ASYNC])
def test_batch_of_small_and_large_graphs(mode):
    """Graphs that fit a block next to ones that do not: each as if alone."""
    graphs = [gg.sbm(7, 200, 4, 0.2, 0.01), gg.rmat(3, 14, 8, wmin=1, wmax=8), gg.sbm(8, 3000, 24, 0.2, 0.001),
              gg.sbm(9, 1024, 2, 0.5, 0.01), _path(5000, 3), gg.sbm(10, 9000, 64, 0.1, 0.0005)]
    with Louvain(device=0, mode=mode, prune=1) as lv:
        lv.load_parts([(g.off, g.col, g.w) for g in graphs])
        lv.run()
        memb, (q, num, M) = lv.membership(), lv.batch_modularity()
        iters = [lv.batch_iterations(k) for k in range(len(graphs))]
        total = lv.iterations()
    at = 0
    for k, g in enumerate(graphs):
        n = len(g.off) - 1
        if mode == SYNC:
            ref = oracle.louvain(g.off, g.col, g.w, mode=oracle.SYNC, prune=1)
            assert np.array_equal(memb[at:at + n], ref.top), k
            assert (num[k], int(M[k])) == (ref.q_num, ref.M) and iters[k] == list(ref.iterations), k
        else:
            ref = oracle.louvain(g.off, g.col, g.w, mode=oracle.ASYNC)
            assert q[k] >= ref.Q - 0.03, k
        at += n
    # the batch's own record sums the graphs', iteration by iteration
    want = {}
    for rows in iters:
        seen = {}
        for p, mv, S in rows:
            t = seen.get(p, 0)
            seen[p] = t + 1
            a = want.setdefault((p, t), [0, 0])
            a[0] += mv
            a[1] += S
    assert total == [(p, want[p, t][0], want[p, t][1]) for p, t in sorted(want)]
