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


@pytest.mark.parametrize("h", [0.03, 0.007, 1e-3])
def test_particles_on_faces_and_edges(h):
    """A particle on a face of a rectangular cell or on an edge, away from all
    else, leaves a half or a quarter in each cell around it.  An exact zero is
    moved inside by 1e-12 h per plane, which moves each fraction by at most
    2 x 0.7e-12."""
    product = lambda v: np.stack(np.meshgrid(*[v] * 3, indexing="ij"), -1).reshape(-1, 3)  # noqa: E731
    g = synth.voronoi(product(np.array([3, 13, 23]) / 32.0))
    for a in (g.vx, g.vy, g.vz, g.face_plane):  # planes at 8/32 and 18/32, each 5/32 from its sites, to the last bit
        a[...] = np.round(a * 32) / 32
    at = product(np.array([3, 8, 13, 18, 23]) / 32.0)
    on = (at == 0.25) | (at == 0.5625)
    at = at[on.sum(axis=1) < 3]
    p = synth.Particles(*(np.ascontiguousarray(at[:, k]) for k in range(3)), np.full(len(at), 1.0 / len(at)))
    got = gpu_map(g, p, np.full(len(at), h), 0)
    cell = np.repeat(np.arange(g.ncell), np.diff(got["off"]))
    r = np.abs(at[got["idx"]] - g.site[cell])
    want = np.where(np.max(r, axis=1) < 0.16, 0.5 ** np.sum(r > 0.15, axis=1), 0.0)
    assert np.allclose(np.bincount(got["idx"], want), 1.0)
    assert np.max(np.abs(got["frac"] - want)) < 1e-11


def test_small_particles_at_small_faces():
    """Particles of a 1e-9th of the cells' size just outside the corners of
    the smallest faces: the distances of such a face are hundreds of h off in
    FP32.  A particle's fractions add up to 1; each cell places its planes to
    some 1e-16 / h = 1e-6 h, so to a few 1e-6; 1e-4 leaves a factor of 30."""
    h = 1e-10
    g = synth.voronoi(np.random.default_rng(71).random((4000, 3)))
    v = np.stack([g.vx, g.vy, g.vz], axis=1)
    at = []
    for c in range(g.ncell):
        for f in range(g.cell_face_off[c], g.cell_face_off[c + 1]):
            w = v[g.face_vert[g.face_vert_off[f]:g.face_vert_off[f + 1]]]
            mid = w.mean(axis=0)
            size = np.linalg.norm(w - mid, axis=1)
            if 1e-7 < size.max() < 0.003 * np.linalg.norm(mid - g.site[c]):
                at.append(w + 0.7 * h * (w - mid) / size[:, None])
    at = np.concatenate(at)
    at = at[np.all((at > 1e-9) & (at < 1.0 - 1e-9), axis=1)]
    assert len(at) > 200
    p = synth.Particles(*(np.ascontiguousarray(at[:, k]) for k in range(3)), np.full(len(at), 1.0 / len(at)))
    got = gpu_map(g, p, np.full(len(at), h), 0)
    assert np.max(np.abs(np.bincount(got["idx"], got["frac"], len(at)) - 1.0)) < 1e-4


@pytest.mark.parametrize("h,most,tol", [(0.02, 2, 1e-11), (1e-4, 2, 1e-11), (1e-8, 3, 1e-7), (1e-10, 3, 1e-5)])
def test_particles_on_a_cubic_grid(h, most, tol):
    """The faces and edges of cells of a sixth, whose planes are no binary
    fractions, and their corners at sizes where y's rounding, 1e-16 / h of the
    cell, is more than the 1e-12 h of the displacement (it moves the fractions
    by as much: tol)."""
    product = lambda v: np.stack(np.meshgrid(*[v] * 3, indexing="ij"), -1).reshape(-1, 3)  # noqa: E731
    g = synth.voronoi(product((np.arange(6) + 0.5) / 6))
    for a in (g.vx, g.vy, g.vz, g.face_plane[:, 3]):
        a[...] = np.round(a * 6) / 6
    g.face_plane[:, :3] = np.round(g.face_plane[:, :3])
    k = product(np.arange(1, 12))
    k = k[np.sum(k % 2 == 0, axis=1) <= most]
    at = k / 12.0
    p = synth.Particles(*(np.ascontiguousarray(at[:, i]) for i in range(3)), np.full(len(at), 1.0 / len(at)))
    got = gpu_map(g, p, np.full(len(at), h), 0)
    cell = np.repeat(np.arange(g.ncell), np.diff(got["off"]))
    near = np.max(np.abs(at[got["idx"]] - g.site[cell]), axis=1) < 0.084
    want = np.where(near, 0.5 ** np.sum(k % 2 == 0, axis=1)[got["idx"]], 0.0)
    assert np.allclose(np.bincount(got["idx"], want), 1.0)
    assert np.max(np.abs(got["frac"] - want)) < tol
