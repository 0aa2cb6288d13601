"""GPU pair lists at the edges of the walk, its rows and their chunks: bit for
bit the oracle's lists."""
import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import gpu_map

pytestmark = pytest.mark.gpu


def _h(n, mean_pairs):
    """h for about mean_pairs particles within 2h."""
    return 0.5 * (3.0 * mean_pairs / (4.0 * np.pi * n)) ** (1.0 / 3.0)


# (particles, pairs wanted per cell): the root as the only leaf; fewer cells
# than lanes; one warp and one cell over; rows that end at, before and after
# 256 entries; rows in several chunks; a pool that runs out
CASES = [(9, 3), (31, 8), (33, 60), (700, 150), (1500, 255), (2100, 420), (1025, 1000), (4200, 1300)]


@pytest.mark.parametrize("n,pairs", CASES)
def test_lists_equal_the_oracle(n, pairs):
    p = synth.uniform_particles(n, 100 + n)
    g = synth.voronoi(p.pos())
    h = _h(n, pairs) * np.random.default_rng(n).uniform(0.7, 1.3, n)
    got = gpu_map(g, p, h, 1)
    off, idx = oracle.pair_lists(g, p.x, p.y, p.z, h)[:2]
    assert np.array_equal(got["off"], off)
    assert np.array_equal(got["idx"], idx)


def test_cell_with_more_faces_than_are_staged():
    """A site inside a shell of 200 others: a cell of more than 64 faces, which
    the filter reads from global memory."""
    rng = np.random.default_rng(5)
    u = rng.normal(size=(200, 3))
    pos = np.concatenate([[[0.5, 0.5, 0.5]], 0.5 + 0.25 * u / np.linalg.norm(u, axis=1)[:, None]])
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(201, 1.0 / 201))
    g = synth.voronoi(pos)
    assert np.diff(g.cell_face_off).max() > 64
    h = rng.uniform(0.02, 0.15, 201)
    got = gpu_map(g, p, h, 1)
    off, idx = oracle.pair_lists(g, p.x, p.y, p.z, h)[:2]
    assert np.array_equal(got["off"], off)
    assert np.array_equal(got["idx"], idx)


def test_many_coincident_particles_in_one_leaf():
    """A leaf of more particles than a staging round (one position, deepest
    level), on a grid of 64 cells."""
    g = synth.voronoi(synth.uniform_particles(64, 8).pos())
    pos = np.concatenate([np.full((90, 3), 0.37), np.random.default_rng(9).random((110, 3))])
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(200, 1.0 / 200))
    h = np.full(200, 0.06)
    got = gpu_map(g, p, h, 1)
    off, idx = oracle.pair_lists(g, p.x, p.y, p.z, h)[:2]
    assert np.array_equal(got["off"], off) and np.array_equal(got["idx"], idx)
