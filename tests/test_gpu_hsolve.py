"""Smoothing lengths on the GPU where a particle's candidates outgrow one of
the solver's lists, against the oracle's solve."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_helpers import lib
from gpu_helpers import dev_particles, oracle_h

pytestmark = pytest.mark.gpu


def _uniform(n):
    return np.random.default_rng(n).random((n, 3))


def _cluster(n, far, width):
    """A tight cluster and a few particles around it, whose first guess reaches
    the whole cluster: lists longer than the position buffer."""
    rng = np.random.default_rng(n + far)
    return np.concatenate([0.5 + width * rng.normal(size=(n, 3)), 0.5 + 0.3 * (rng.random((far, 3)) - 0.5)])


def _lattice(k):
    g = (np.arange(k) + 0.5) / k
    return np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)


# one particle; a root leaf; part of a window; a window and one; a list just
# past its registers; clusters whose lists need chunks, with Newton and with
# bisection; equal distances
SETS = {"one": _uniform(1), "root_leaf": _uniform(16), "two_leaves": _uniform(17), "n257": _uniform(257),
        "n4099": _uniform(4099), "cluster": _cluster(3000, 40, 0.004), "wide_cluster": _cluster(6000, 300, 0.02),
        "tight_cluster": _cluster(1500, 7, 1e-4), "lattice": _lattice(12)}


@pytest.mark.parametrize("name", SETS)
@pytest.mark.parametrize("precision,tol", [(0, 1e-11), (1, 1e-6)])
def test_h_and_route_equal_the_oracle(name, precision, tol):
    """tol: the FP64 build's last step leaves (1e-7)^3 and the rounding of the
    sums (some 1e-14); the oracle's bisection ends at 1e-12.  The mixed build
    solves on FP32 sums to 1e-6."""
    L = lib()
    pos = SETS[name]
    x, y, z = (torch.as_tensor(np.ascontiguousarray(pos[:, k]), device="cuda") for k in range(3))
    m = L.ExactMapper(precision)
    h, route = (t.cpu().numpy() for t in m.solve_h(x, y, z))
    m.close()
    p = synth.Particles(*(np.ascontiguousarray(pos[:, k]) for k in range(3)), np.full(len(pos), 1.0 / len(pos)))
    ref, want = oracle.solve_h(p.x, p.y, p.z, oracle.particle_h_guess(oracle.Tree(p.x, p.y, p.z, p.m)))
    assert np.array_equal(route, want)
    assert np.max(np.abs(h / ref - 1.0)) < tol


@pytest.mark.parametrize("kind", ["line", "plane", "pairs"])
def test_fp64_routes_are_the_oracles(kind):
    """Sets on which Newton ends near the bracket's bounds or on flat stretches:
    the FP64 build takes the oracle's route for every particle, and both stop
    within 1e-10 of the root (2e-10 apart at most)."""
    L = lib()
    ctx = L.map_init(L.map_config_default(precision=L.MAP_FP64))
    try:
        for seed in range(6):
            r = np.random.default_rng(80 + seed)
            u = r.random((3, 4000))
            if kind == "pairs":
                u[:, :2000] = np.clip(u[:, 2000:] + 1e-5 * r.normal(size=(3, 2000)), 0.0, 1.0)
            elif kind == "line":
                u[1:] = 0.5
            else:
                u[2] = 0.25
            p = synth.Particles(*u, np.full(4000, 1.0 / 4000))
            x, y, z, m, h = dev_particles(p)
            route = torch.empty(p.n, dtype=torch.int32, device="cuda")
            L.solve_h(ctx, L.make_particles(x, y, z, m, h), route)
            want, want_route = oracle_h(p)
            assert np.array_equal(route.cpu().numpy(), want_route)
            assert np.max(np.abs(h.cpu().numpy() / want - 1.0)) < 2e-10
    finally:
        L.map_destroy(ctx)
