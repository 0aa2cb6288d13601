"""The device octree at the edges of its maps and launches, seen through the
walk: with a source whose r_leaf covers the cube the pseudo-particles are
exactly the leaves, with a small theta they come from every level."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_pseudo import gpu_pseudo

pytestmark = pytest.mark.gpu


def _set(kind):
    rng = np.random.default_rng(23)
    if kind == "coincident":  # leaves at the deepest level, with more particles than a leaf holds
        return np.concatenate([np.full((70, 3), 0.61), rng.random((60, 3))])
    if kind == "cluster":  # a long chain of single children
        return np.concatenate([0.5 + 1e-5 * rng.random((300, 3)), rng.random((20, 3))])
    return rng.random((int(kind), 3))


def _keys(pos):
    """Morton keys: 21 bits of each coordinate interleaved, x highest (numpy)."""
    c = np.minimum(pos * 2.0 ** 21, 2.0 ** 21 - 1).astype(np.uint64)
    key = np.zeros(len(pos), np.uint64)
    for b in range(21):
        for d in range(3):
            key |= ((c[:, d] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - d)
    return key


# the places of the one-block sort (64 to 4096, one exchange per thread up to
# 2048, two above) and the sizes around its limit
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 1000, 2048, 2049, 4095, 4096, 4097, 5000])
def test_particles_come_in_stable_morton_order(n):
    """A source whose r_part covers the cube extracts every particle, listed by
    Morton position; a quarter of them share their place with another, those in
    index order."""
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    if n > 3:
        pos[rng.permutation(n)[: n // 4]] = pos[rng.permutation(n)[: n // 4]]
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(n, 1.0 / n))
    out = gpu_pseudo(p, np.full(n, 0.1), np.array([0.5, 0.5, 0.5]), r_part=2.0)
    assert np.all(out["kind"] == 1)
    assert np.array_equal(out["ident"], np.argsort(_keys(pos), kind="stable"))


# words of the maps: 31, 32, 33, 64, 65 positions; a slice of a big node and one
# particle more; a node of several slices
@pytest.mark.parametrize("kind", ["1", "16", "17", "31", "32", "33", "64", "65", "4096", "4097", "20000", "coincident",
                                  "cluster"])
@pytest.mark.parametrize("theta,r_leaf", [(1e9, 2.0), (0.3, 0.0)])
def test_walk_equals_the_oracle(kind, theta, r_leaf):
    """Labels and particles equal; masses and centres of mass to 1e-12 (sums of
    at most 20000 terms in another order); h to 1e-9, the pseudo solve's gate,
    for the nodes that have a size (the rounded centre of coincident particles
    may leave them one of 1e-17 on either side)."""
    pos = _set(kind)
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(len(pos), 2.0 ** -15))
    h = np.full(len(pos), 0.5 * len(pos) ** (-1.0 / 3.0))
    src = np.array([0.37, 0.52, 0.44])
    t = oracle.Tree(p.x, p.y, p.z, p.m)
    acc, opened = t.walk(src, theta, r_leaf=r_leaf)
    hn, _ = oracle.pseudo_h(t, acc, opened, h)
    out = gpu_pseudo(p, h, src, theta=theta, r_leaf=r_leaf)
    got = np.argsort(out["ident"][out["kind"] == 0])
    ref = np.argsort(t.label[acc])
    pick = lambda f: out[f][out["kind"] == 0][got]  # noqa: E731
    assert np.array_equal(pick("ident"), t.label[acc][ref])
    parts = np.sort(np.concatenate([t.particles_of(i) for i in opened])) if len(opened) else np.zeros(0, np.int64)
    assert np.array_equal(np.sort(out["ident"][out["kind"] == 1]), parts)
    com = t.com[acc][ref]
    assert np.max(np.abs(pick("m") / t.mass[acc][ref] - 1.0), initial=0.0) < 1e-12
    assert np.max(np.abs(np.stack([pick("x"), pick("y"), pick("z")], 1) - com), initial=0.0) < 1e-12
    sized = t.size[acc][ref] > 1e-12
    assert np.max(np.abs(pick("h") / hn[ref] - 1.0)[sized], initial=0.0) < 1e-9
