"""The order's sorts on half keys: runs of points that share a cell of 2^-32 of the box, from pairs
to runs longer than are ordered in place, with exact duplicates among them, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def crowded(run, n, seed):
    """n points of which groups of `run` share a tiny box, and two far corners."""
    g = np.random.default_rng(seed)
    c = g.random((max(1, n // run), 3))
    x = np.repeat(c, run, axis=0)[:n] + 1e-7 * g.random((min(n, len(c) * run), 3))
    x[::7] = x[::7][np.argsort(g.random(len(x[::7])))]
    x[1::11] = x[::11][:len(x[1::11])]  # exact duplicates
    return np.concatenate([np.zeros((1, 3)), x, np.ones((1, 3))])


@pytest.mark.parametrize("run", [2, 3, 63, 64, 65, 200, 1500])
def test_order_and_tetrahedra(run):
    import torch
    import paper_1805_08831_gb300 as dt
    x = crowded(run, 3000, run)
    ref, _ = oracle.delaunay(x, seed=4)
    with dt.Triangulation(seed=4) as t:
        t.insert(torch.from_numpy(x).cuda())
        assert np.array_equal(t.tets_numpy(), ref)
        k, p, r = t.order(len(x))
    assert np.array_equal(k, oracle.moore_keys(x))
    assert np.array_equal(r, oracle.brio_rounds(len(x), 4))
    assert np.array_equal(p, oracle.insertion_order(x, 4))
