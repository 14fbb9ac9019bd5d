"""A batch of small clouds, built over and over: every cloud is a mesh of its own in one store, and
no point ends up in another cloud's mesh (a wrong list, or a batch that never ends)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_batch_built_over_and_over():
    import torch
    import paper_1805_08831_gb300 as dt
    g = np.random.default_rng(7)
    clouds = [g.random((n, 3)) for n in g.integers(50, 900, 64)]
    off = np.cumsum([0] + [len(c) for c in clouds]).astype(np.uint64)
    ref = np.concatenate([oracle.delaunay(c, seed=5)[0] for c in clouds])
    x = torch.from_numpy(np.concatenate(clouds)).cuda()
    out = torch.zeros((len(ref) + 8, 4), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
    with dt.Triangulation(seed=5) as t:
        for k in range(800):
            t.batch(x, off)
            rows, _ = t.tets_batch(out=out)
            assert np.array_equal(rows, ref), k
