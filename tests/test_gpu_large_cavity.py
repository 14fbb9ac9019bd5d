"""Cavities at the edges of the asynchronous engine's workspaces: the centre of a sphere of n points
joins a mesh whose every tetrahedron is in conflict with it, through the borrowed workspaces (up
to 640 tetrahedra), the large-cavity kernel's (up to 6144) and the serial path, and the same with
points the FP32 stage cannot decide (a sphere of lattice points: co-spherical and coplanar)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def sphere(n, seed):
    g = np.random.default_rng(seed).normal(size=(n, 3))
    return g / np.linalg.norm(g, axis=1, keepdims=True)


def lattice_sphere(r2):
    k = int(np.sqrt(r2)) + 1
    g = np.stack(np.meshgrid(*[np.arange(-k, k + 1.0)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return g[(g * g).sum(1) == r2]


SHELLS = {"30": sphere(30, 1), "200": sphere(200, 2), "900": sphere(900, 3), "4000": sphere(4000, 4),
          "lattice_50": lattice_sphere(50), "lattice_1469": lattice_sphere(1469)}


@pytest.mark.parametrize("name", SHELLS)
def test_centre_of_a_shell(name):
    import torch
    import paper_1805_08831_gb300 as dt
    x = SHELLS[name]
    inner = np.concatenate([np.zeros((1, 3)), 0.1 * sphere(7, 9) * np.abs(x).max()])
    ref, _ = oracle.delaunay(np.concatenate([x, inner]), seed=2)
    with dt.Triangulation(seed=2) as t:
        t.insert(torch.from_numpy(x).cuda())
        t.insert(torch.from_numpy(inner).cuda())
        assert np.array_equal(t.tets_numpy(), ref)
        assert t.check()["not_delaunay"] == 0
