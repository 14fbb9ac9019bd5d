"""A small mesh built over and over: its warps walk through records that others rewrite on most
steps, so a walk whose lanes act on different versions of one record shows here (a lost point, or
slots lost to the allocator)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [63, 2047, 9001])
def test_built_over_and_over(n):
    import torch
    import paper_1805_08831_gb300 as dt
    x = np.random.default_rng(n).random((n, 3))
    ref, _ = oracle.delaunay(x, seed=1)
    ref = torch.from_numpy(ref.astype(np.int64)).cuda()
    xd = torch.from_numpy(x).cuda()
    with dt.Triangulation(seed=1) as t:
        for k in range(1500 if n < 9000 else 300):
            t.insert(xd)
            got = t.tets()
            assert got.shape == ref.shape and bool((got.long() == ref).all()), k
            t.clear()
