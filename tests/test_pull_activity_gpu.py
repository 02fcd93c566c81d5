"""Synchronous pruning by the flags of moved neighbours: which vertices are visited, and the results."""
import numpy as np
import pytest

from engine_util import assert_sync_parity, engine_run

pytestmark = pytest.mark.gpu


class _Stars:
    """Disjoint stars (centres of the given degrees, settled after a few iterations and inactive
    from then on) beside rings whose vertices go on moving; weights 1..wmax."""

    def __init__(self, degrees, ring, wmax, seed):
        rng = np.random.default_rng(seed)
        u, v, at = [], [], 0
        for d in degrees:
            u.append(np.full(d, at))
            v.append(at + 1 + np.arange(d))
            at += d + 1
        r = at + np.arange(ring)
        u += [r, r]
        v += [at + (np.arange(ring) + 1) % ring, at + rng.permutation(ring)]
        u, v = np.concatenate(u), np.concatenate(v)
        self.n = n = at + ring
        pair = np.unique((np.minimum(u, v) * n + np.maximum(u, v))[u != v])
        u, v = pair // n, pair % n
        w = rng.integers(1, wmax + 1, len(pair))
        key = np.concatenate([u * n + v, v * n + u])
        o = np.argsort(key, kind="stable")
        self.off = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int64)
        self.col = (key[o] % n).astype(np.int32)
        self.w = np.concatenate([w, w])[o].astype(np.int32)
        self.nnz = len(self.col)


DEGREES = [[1, 4, 5, 8, 9, 32, 33], [64, 128, 129, 1024, 1025], [4096, 4097, 12288, 12289, 20000]]


@pytest.mark.parametrize("classes", [{}, {"subrounds": 4}, {"colour_classes": 1}], ids=["one", "four", "colour"])
@pytest.mark.parametrize("wmax", [3, 1 << 29])
@pytest.mark.parametrize("degrees", DEGREES, ids=["-%d" % max(d) for d in DEGREES])
def test_flagged_and_stamped_iterations_visit_the_same_vertices(degrees, wmax, classes):
    g = _Stars(degrees, 30000, wmax, 5)
    assert_sync_parity(g, prune=1, max_passes=1, max_iterations=8, **classes)
    # stop rule 1 keeps the stamps, and its modularity rises in the first four iterations
    opt = dict(mode=0, prune=1, max_passes=1, max_iterations=4, tolerance=0.0, **classes)
    got, ref = engine_run(g, **opt), engine_run(g, stop_rule=1, **opt)
    assert len(ref["iters"]) == 4 and ref["iters"] == got["iters"]
    for f in ("lm_vertices", "lm_edges", "lm_bytes"):
        assert getattr(ref["stats"], f) == getattr(got["stats"], f), f
