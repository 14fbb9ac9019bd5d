"""The canonical list's bucket sort at the sizes where it can go wrong: a vertex whose star is
just within and just beyond the largest bucket a block orders, tiles whose last bucket crosses
their end, one tetrahedron, and the same inside a batch."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def hub(n, seed):
    """A centre (input index 0) inside n points of the unit sphere: 2 n - 4 tetrahedra hold it."""
    g = np.random.default_rng(seed).normal(size=(n, 3))
    return np.concatenate([np.zeros((1, 3)), g / np.linalg.norm(g, axis=1, keepdims=True)])


def cloud(n, seed):
    return np.random.default_rng(seed).random((n, 3))


CASES = {
    "one": cloud(4, 1), "few": cloud(9, 2), "tile": cloud(163, 3), "tiles": cloud(5000, 4),
    "star_1022": hub(513, 5), "star_1024": hub(514, 6), "star_1026": hub(515, 7), "star_4996": hub(2500, 8),
}


@pytest.mark.parametrize("name", CASES)
def test_list_equals_the_oracle(name):
    import torch
    import paper_1805_08831_gb300 as dt
    x = CASES[name]
    ref, _ = oracle.delaunay(x, seed=3)
    with dt.Triangulation(seed=3) as t:
        for _ in range(2):  # the scratch of the first list must leave the engine's words zero
            t.clear()
            t.insert(torch.from_numpy(x).cuda())
            assert np.array_equal(t.tets_numpy(), ref)
            assert np.array_equal(t.tets_numpy(), ref)
            out = torch.zeros((len(ref) + 3, 4), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
            assert np.array_equal(t.tets_host(out=out), ref)
            assert t.num_tets() == len(ref)


def test_batch_lists_equal_the_oracle():
    import torch
    import paper_1805_08831_gb300 as dt
    clouds = [CASES[k] for k in ("star_1026", "one", "tile", "star_1024", "few")] + [np.zeros((5, 3)), cloud(700, 9)]
    off = np.cumsum([0] + [len(c) for c in clouds]).astype(np.uint64)
    with dt.Triangulation(seed=3) as t:
        t.batch(torch.from_numpy(np.concatenate(clouds)).cuda(), off)
        rows, coff = t.tets_batch()
        out = torch.zeros((len(rows), 4), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
        again, coff2 = t.tets_batch(out=out)
        assert np.array_equal(rows, again) and np.array_equal(coff, coff2)
        for c, x in enumerate(clouds):
            ref = np.zeros((0, 4), np.uint32) if len(x) == 5 else oracle.delaunay(x, seed=3)[0]
            assert np.array_equal(rows[int(coff[c]):int(coff[c + 1])], ref), c
