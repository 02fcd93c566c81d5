"""Synchronous classes of which some hold no vertex with entries."""
import numpy as np
import pytest

from engine_util import assert_sync_parity
from test_degree_edges_gpu import _Csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hub", [0, 200])   # without a row above 128 entries a class is one launch, with it several
@pytest.mark.parametrize("classes,kept", [(4, [0, 2]), (5, [1, 2, 4]), (6, [5]), (64, [0, 1, 40, 63])], ids=str)
@pytest.mark.parametrize("prune", [0, 1])
def test_sync_parity(classes, kept, hub, prune):
    rng = np.random.default_rng(classes)
    n = 40000
    ids = np.flatnonzero(np.isin(np.arange(n) % classes, kept))
    a = rng.integers(0, len(ids), 3 * len(ids))
    b = np.minimum(a // 30 * 30 + rng.integers(0, 30, len(a)), len(ids) - 1)
    u, v = np.concatenate([ids[a], np.full(hub, ids[0])]), np.concatenate([ids[b], rng.choice(ids, hub)])
    pair = np.unique(np.minimum(u, v)[u != v] * n + np.maximum(u, v)[u != v])
    assert_sync_parity(_Csr(n, pair // n, pair % n, np.ones(len(pair), np.int64)), prune=prune, subrounds=classes)
