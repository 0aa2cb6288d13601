"""The FP64 pair-integral kernel at the edges of its blocks and stacks, against
the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import gpu_map

pytestmark = pytest.mark.gpu


def _shell(n):
    u = np.random.default_rng(n).normal(size=(n, 3))
    return np.concatenate([[[0.5, 0.5, 0.5]], 0.5 + 0.25 * u / np.linalg.norm(u, axis=1)[:, None]])


# one pair; a block short of and past a warp; several items per cell; a cell of
# more faces than are staged; supports from far below to far above the cells
CASES = [("uniform", 1, 0.2), ("uniform", 31, 0.3), ("uniform", 33, 0.3), ("uniform", 260, 0.4),
         ("uniform", 700, 0.004), ("shell", 60, 0.1), ("shell", 200, 0.05), ("shell", 200, 0.3)]


@pytest.mark.parametrize("kind,n,h", CASES)
def test_masses_equal_the_oracle(kind, n, h):
    """Each pair sums some 60 edges of three angles, each good to 4e-16 with a
    weight of at most 0.13: about 1e-14 per pair, the pairs' masses sum to at
    most 1 per cell; 1e-12 leaves a factor of 100.  (Not the single fractions:
    a short edge's direction is as good as its length over 1e-16.)"""
    pos = _shell(n) if kind == "shell" else np.random.default_rng(n).random((n, 3))
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(len(pos), 1.0 / len(pos)))
    g = synth.voronoi(pos)
    hh = h * np.random.default_rng(n + 1).uniform(0.6, 1.4, len(pos))
    ref = oracle.map_cells(g, p.x, p.y, p.z, p.m, hh)
    got = gpu_map(g, p, hh, 0)
    assert np.array_equal(got["idx"], ref["idx"])
    assert np.max(np.abs(got["mass"] - ref["mass"])) < 1e-12
