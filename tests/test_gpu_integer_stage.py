"""The exact stage on integers at the edges of what it accepts: coordinates of 62 significant bits
after scaling (the largest differences, minors and sums), of 63 (which go to the expansions), and
zeros, signed zeros and small lattices, against the oracle's big integers."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOP = float(2 ** 62 - 2 ** 9)  # 53 bits, the highest worth 2^61


def tuples(kind, n):
    g = np.random.default_rng(len(kind))
    if kind == "extremes":  # sums and differences that fill the words, beside a lowest bit of 1
        return g.choice([TOP, -TOP, 2.0 ** 61, -(2.0 ** 61), TOP - 2 ** 9, 1.0, 0.0], (n, 5, 3))
    if kind == "sixty_three_bits":
        return g.choice([2.0 * TOP, -2.0 * TOP, 2.0 ** 62, 1.0, 0.0], (n, 5, 3))
    if kind == "random_62":  # 53 random bits and an exponent of up to 9 more
        return g.integers(2 ** 52, 2 ** 53, (n, 5, 3)) * 2.0 ** g.integers(0, 10, (n, 5, 3)) * g.choice([-1, 1], (n, 5, 3))
    if kind == "signed_zeros":
        return g.choice([0.0, -0.0, 1.0, -1.0, 0.5], (n, 5, 3))
    p = g.integers(0, 49, (n, 5, 3)) / 48.0  # the refinement's surface lattice
    p[: n // 2, :, 2] = p[: n // 2, :1, 2]  # coplanar
    p[n // 2:, 4] = p[n // 2:, 0] + p[n // 2:, 1] - p[n // 2:, 2]  # often co-circular
    return p


@pytest.mark.parametrize("kind", ["extremes", "sixty_three_bits", "random_62", "signed_zeros", "lattice"])
def test_signs_equal_the_oracle(kind):
    import torch
    import paper_1805_08831_gb300 as dt
    p = tuples(kind, 1500)
    pt = torch.from_numpy(p).cuda()
    o, s = dt.eval_predicates(0, pt).cpu().numpy(), dt.eval_predicates(1, pt).cpu().numpy()
    assert np.array_equal(o, [oracle.orient3d(*q[:4]) for q in p])
    assert np.array_equal(s, [oracle.insphere(*q) for q in p])
