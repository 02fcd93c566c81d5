"""Asynchronous quality of small graphs with few classes."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from engine_util import engine_run
from paper_2301_12390_gb300 import ASYNC, SYNC
from test_degree_edges_gpu import _Csr

pytestmark = pytest.mark.gpu


def _hubs(n, edges, degrees, seed):
    """Vertices of the given degrees beside short links (within 40 ids), ids permuted."""
    rng = np.random.default_rng(seed)
    k = len(degrees)
    u = [np.full(d, i) for i, d in enumerate(degrees)]
    v = [k + rng.choice(n - k, d, replace=False) for d in degrees]
    a = rng.integers(0, n, edges - sum(degrees))
    u, v = np.concatenate(u + [a]), np.concatenate(v + [(a // 40 * 40 + rng.integers(0, 40, len(a))) % n])
    name = rng.permutation(n)
    u, v = name[u[u != v]], name[v[u != v]]
    pair = np.unique(np.minimum(u, v) * n + np.maximum(u, v))
    return _Csr(n, pair // n, pair % n, np.ones(len(pair), np.int64))


FAMILIES = {
    "hubs": lambda s: _hubs(6000, 10000, [1000, 300, 200], s),
    "sbm": lambda s: gg.sbm(s, 6000, 48, 0.1, 0.001),
    "grid": lambda s: gg.grid_road(s, 80),
    "rmat": lambda s: gg.rmat(s, 12, 3, wmin=1, wmax=8),
}


def test_one_class_is_not_the_synchronous_schedule():
    # decisions of one class see moves made before them in it
    for seed in range(12):
        g = FAMILIES["hubs"](100 + seed)
        a, s = (engine_run(g, mode=m, prune=1, subrounds=1) for m in (ASYNC, SYNC))
        assert not np.array_equal(a["top"], s["top"]), seed


@pytest.mark.parametrize("classes", [4, 8])
@pytest.mark.parametrize("name", list(FAMILIES))
def test_quality_with_few_classes(name, classes):
    diff = []
    for seed in range(6):
        g = FAMILIES[name](100 + seed)
        ref = oracle.louvain(g.off, g.col, g.w, mode=oracle.ASYNC, prune=1)
        diff.append(engine_run(g, mode=ASYNC, prune=1, subrounds=classes)["q"] - ref.Q)
    assert min(diff) > -0.03 and np.mean(diff) > -0.003, diff
