"""Which kernels a graph or a batch takes depends on it alone, not on what its context held before."""
import numpy as np
import pytest

import graphgen as gg
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
