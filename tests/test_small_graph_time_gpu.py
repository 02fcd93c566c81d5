"""Time of the one-block local-moving phase on graphs whose shape could make it slow."""
import numpy as np
import pytest

import graphgen as gg
from engine_util import assert_sync_parity
from paper_2301_12390_gb300 import SYNC, Louvain
from test_degree_edges_gpu import _Csr

pytestmark = pytest.mark.gpu


def _pairs(n, links, leaves):
    """`links` disjoint pairs among n vertices; with leaves, vertex 0 also joined to that many of the others."""
    u, v = 1 + 2 * np.arange(links), 2 + 2 * np.arange(links)
    if leaves:
        leaf = 1 + np.random.default_rng(1).choice(2 * links, leaves, replace=False)
        u, v = np.concatenate([u, np.zeros(leaves, np.int64)]), np.concatenate([v, leaf])
    return _Csr(n, u, v, np.ones(len(u), np.int64))


def _star(leaves):
    return _Csr(leaves + 1, np.zeros(leaves, np.int64), 1 + np.arange(leaves), np.ones(leaves, np.int64))


def _iteration_ms(g, runs=7, **opt):
    """Local-moving time of an iteration of pass 0, the shortest of several runs."""
    best = float("inf")
    with Louvain(device=0, mode=SYNC, prune=1, max_passes=1, **opt) as lv:
        lv.load_csr(g.off, g.col, g.w)
        for _ in range(runs):
            lv.run()
            p = lv.passes()[0]
            best = min(best, p.lm_ms / p.iterations)
    return best


def test_a_long_row_does_not_slow_the_other_vertices():
    # the same 3,300 pairs with and without one vertex of degree 200: searching the class for it by the
    # whole block took ten times the rest of the iteration
    plain, hub = _pairs(7000, 3300, 0), _pairs(7000, 3300, 200)
    assert_sync_parity(hub, prune=1)
    assert _iteration_ms(hub) < 3 * _iteration_ms(plain)


def test_moves_into_one_community_do_not_queue_up():
    # the leaves of a star all leave and join the same communities: four times the time of as many pairs
    # when each of their updates waits for the others'
    star, plain = _star(3400), _pairs(7000, 3300, 0)
    assert_sync_parity(star, prune=1)
    assert _iteration_ms(star) < 2 * _iteration_ms(plain)


@pytest.mark.parametrize("classes", [1, 3])
def test_totals_carry_across_32_bits(classes):
    # two communities whose totals pass 2^32 while every degree still suits 64-bit gains
    rng = np.random.default_rng(2)
    u, v = np.triu_indices(64, 1)
    keep = rng.random(len(u)) < np.where(u // 32 == v // 32, 0.7, 0.03)
    g = _Csr(64, u[keep], v[keep], rng.integers(5_000_000, 8_000_000, int(keep.sum())))
    K = np.add.reduceat(g.w.astype(np.int64), g.off[:-1])
    assert int(K.max()) <= (1 << 61) // int(K.sum())
    _, ref = assert_sync_parity(g, prune=1, subrounds=classes)
    assert np.bincount(ref.top, weights=K).min() > 1 << 32


def _blocks(n, degree):
    """Blocks of about 60 vertices, three quarters of a vertex's entries inside its block."""
    return gg.sbm(1, n, max(2, n // 60), min(1.0, 0.75 * degree / 60), 0.25 * degree / n)


@pytest.mark.parametrize("n,degree,classes", [(1000, 19, 1), (1000, 19, 4), (600, 12, 1), (1500, 12, 1), (8000, 2.5, 1)])
def test_one_block_only_where_it_pays(n, degree, classes):
    # more than 32 iterations allowed: always the launches.  The first two graphs and the last took a
    # block 2.3 to 5.8 times as long
    g = _blocks(n, degree)
    chosen = _iteration_ms(g, subrounds=classes, max_iterations=20)
    launches = _iteration_ms(g, subrounds=classes, max_iterations=33)
    assert chosen < 2 * launches


def test_wide_weights_do_not_slow_the_aggregation():
    # two blocks of 250 fully joined: their entries fall on a handful of sums, of 64 bits with large weights
    # (27 times the time of 32-bit ones while each addition waited for the others)
    ms = []
    for wmax in (1, 1_000_000):
        g = gg.sbm(1, 500, 2, 1.0, 0.002, 1, wmax)
        with Louvain(device=0, mode=SYNC, prune=1, subrounds=4) as lv:
            lv.load_csr(g.off, g.col, g.w)
            best = float("inf")
            for _ in range(7):
                lv.run()
                best = min(best, lv.passes()[0].agg_ms)
            ms.append(best)
        assert_sync_parity(g, prune=1, subrounds=4)
    assert ms[1] < 4 * ms[0]
