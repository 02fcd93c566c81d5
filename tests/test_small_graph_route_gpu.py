"""Which kernels a graph or a batch takes depends on it alone, not on what its context held before."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from engine_util import assert_sync_parity
from paper_2301_12390_gb300 import ASYNC, SYNC, Louvain
from test_degree_edges_gpu import _Csr

pytestmark = pytest.mark.gpu


def _path(n):
    return _Csr(n, np.arange(n - 1), np.arange(1, n), np.ones(n - 1, np.int64))


def _results(lv):
    q, num, M = lv.batch_modularity()
    return lv.membership().tolist(), q.tolist(), num, lv.stats().kernel_launches, lv.iterations()


@pytest.mark.parametrize("mode", [SYNC, ASYNC])
@pytest.mark.parametrize("sizes", [[1], [2], [8], [8] * 300, [1, 2, 3, 40] * 20, [30] * 40], ids=lambda s: "%dx%d" % (len(s), s[0]))
def test_fresh_and_used_contexts(sizes, mode):
    graphs = [_path(n) for n in sizes]
    big = gg.rmat(1, 14, 8)
    got = []
    for used in (False, True):
        with Louvain(device=0, mode=mode, prune=1) as lv:
            if used:
                lv.load_csr(big.off, big.col, big.w)
                lv.run()
            lv.load_parts([(g.off, g.col, g.w) for g in graphs])
            lv.run()
            got.append(_results(lv))
    assert got[0] == got[1]


@pytest.mark.parametrize("n", [1, 2, 3, 9])
def test_sync_parity_of_the_smallest_graphs(n):
    assert_sync_parity(_path(n), prune=1)
    assert_sync_parity(_path(n), subrounds=4)


def test_more_iterations_than_the_first_fetch():
    # a graph whose vertices go on swapping: as many iterations as allowed
    g = gg.sbm(3, 100, 4, 0.3, 0.05)
    for cap in (1, 7, 8, 9, 20, 32):
        assert_sync_parity(g, singleton_guard=0, tolerance=0.0, max_iterations=cap)


def _repeated(graphs, times):
    """The graphs, each `times` times, side by side."""
    n = np.concatenate([np.diff(g.off) for g in graphs] * times)
    off = np.concatenate([[0], np.cumsum(n)])
    vo = np.concatenate([[0], np.cumsum([g.n for g in graphs] * times)])
    col = np.concatenate([np.concatenate([g.col for g in graphs])] * times).astype(np.int64)
    col += np.repeat(vo[:-1], [g.nnz for g in graphs] * times)
    return vo, off, col.astype(np.int32), np.concatenate([g.w for g in graphs] * times)


@pytest.mark.parametrize("times", [4600, 4800])   # 32 classes each: just below 1.5M classes in all, and above
def test_sync_parity_of_many_graphs(times):
    graphs = [gg.sbm(s, 33 + s, 3, 0.4, 0.05) for s in range(10)]
    want = [oracle.louvain(g.off, g.col, g.w, mode=oracle.SYNC, prune=1, subrounds=32) for g in graphs]
    with Louvain(device=0, mode=SYNC, prune=1, subrounds=32) as lv:
        lv.load_batch(*_repeated(graphs, times))
        lv.run()
        memb = lv.membership().reshape(times, -1)
        assert np.array_equal(memb, np.tile(np.concatenate([r.top for r in want]), (times, 1)))
        assert lv.batch_modularity()[0].tolist() == [r.Q for r in want] * times


def test_launches_for_more_graphs_than_fill_the_chip():
    # 100,000 asynchronous graphs of about 60 vertices took a block each 1.4 times as long; a mapping other than
    # the default one always takes the launches
    graphs = [gg.sbm(s, 55 + s, 3, 0.15, 0.03) for s in range(10)]
    ms = []
    with Louvain(device=0, mode=ASYNC, prune=1, max_passes=1) as lv:
        lv.load_batch(*_repeated(graphs, 10000))
        for mapping in (None, [8, 32, 128, 1024, 4095]):
            lv.set_mapping(mapping)
            best = float("inf")
            for _ in range(4):
                lv.run()
                best = min(best, lv.passes()[0].lm_ms)
            ms.append(best)
    assert ms[0] < 1.2 * ms[1], ms
