"""Failure handling on the host side of the C ABI: bad particles, a corrupted
grid and a memory budget below one request are refused with the documented
status codes, and the context stays usable.  Every bad input here is caught
by the library's validation (host checks, or bounds-checked validation
kernels that read only inside the arrays' declared sizes) before any kernel
indexes memory with it."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_helpers import lib, dev_particles, oracle_h, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    p = synth.uniform_particles(512, synth.BASE_SEED + 11)
    g = synth.voronoi(p.pos())
    h, _ = oracle_h(p)
    return p, g, h


def _code(fn):
    L = lib()
    with pytest.raises(L.MapError) as e:
        fn()
    return e.value.code


def _map(L, ctx, g, p, h, handle=None):
    handle = L.map_grid_upload(ctx, L.grid_to_device(g)) if handle is None else handle
    x, y, z, m, hh = dev_particles(p, h)
    mass = torch.empty(g.ncell, dtype=torch.float64, device="cuda")
    L.map_particles_to_cells(ctx, L.make_particles(x, y, z, m, hh), handle, mass)
    torch.cuda.synchronize()
    return handle, mass


@pytest.mark.parametrize("bad", ["h_nan", "h_zero", "h_negative", "x_outside", "z_nan"])
def test_bad_particles_rejected(small, bad):
    L = lib()
    p, g, h = small
    ctx = L.map_init(L.map_config_default(precision=1))
    try:
        handle, ref = _map(L, ctx, g, p, h)
        x, y, z, m, hh = dev_particles(p, h)
        if bad == "h_nan":
            hh[17] = float("nan")
        elif bad == "h_zero":
            hh[3] = 0.0
        elif bad == "h_negative":
            hh[200] = -0.01
        elif bad == "x_outside":
            x[5] = 1.5
        else:
            z[9] = float("nan")
        mass = torch.empty(g.ncell, dtype=torch.float64, device="cuda")
        code = _code(lambda: L.map_particles_to_cells(ctx, L.make_particles(x, y, z, m, hh), handle, mass))
        assert code == L.MAP_EINVAL
        if bad in ("x_outside", "z_nan"):
            # solve_h reads positions only: it refuses the same positions
            hs = torch.empty_like(x)
            assert _code(lambda: L.solve_h(ctx, L.make_particles(x, y, z, None, hs))) == L.MAP_EINVAL
        # the context still maps the good particles, to the same bits
        _, again = _map(L, ctx, g, p, h, handle)
        assert torch.equal(again, ref)
    finally:
        L.map_destroy(ctx)


@pytest.mark.parametrize("bad", ["face_vert_range", "face_vert_negative", "cfo_non_monotone", "cfo_last",
                                 "fvo_short_loop"])
def test_corrupted_grid_rejected(small, bad):
    L = lib()
    p, g, h = small
    ctx = L.map_init(L.map_config_default(precision=1))
    try:
        d = L.grid_to_device(g)
        if bad == "face_vert_range":
            d["face_vert"][123] = g.vx.shape[0]  # one past the last vertex
        elif bad == "face_vert_negative":
            d["face_vert"][7] = -1
        elif bad == "cfo_non_monotone":
            d["cell_face_off"][10] = d["cell_face_off"][12] + 1
        elif bad == "cfo_last":
            d["cell_face_off"][-1] -= 1
        else:
            d["face_vert_off"][40] = d["face_vert_off"][39] + 2  # a two-vertex loop
        assert _code(lambda: L.map_grid_upload(ctx, d)) == L.MAP_EINVAL
        # the good grid still uploads and maps
        _, mass = _map(L, ctx, g, p, h)
        assert np.isfinite(mass.cpu().numpy()).all()
    finally:
        L.map_destroy(ctx)


def test_budget_below_one_request(small):
    L = lib()
    p, g, h = small
    ctx = L.map_init(L.map_config_default(precision=1, hbm_budget=64 << 10))
    try:
        assert _code(lambda: L.map_grid_upload(ctx, L.grid_to_device(g))) == L.MAP_ENOMEM
    finally:
        L.map_destroy(ctx)
    # a context with room maps the same input afterwards
    ctx = L.map_init(L.map_config_default(precision=1))
    try:
        _, mass = _map(L, ctx, g, p, h)
        ref = oracle.map_cells(g, p.x, p.y, p.z, p.m, h)
        assert rel_err(mass.cpu().numpy(), ref["mass"]).max() < 1e-5
    finally:
        L.map_destroy(ctx)


# call, particles, particles per cell, precision (0 FP64, 1 mixed) and an
# hbm_budget in MiB that holds it: half a percent above the least of the
# library's first level-by-level octree and two-pass walk
BUDGETS = [("solve_h", 2000, 1, 1, 0.489), ("map", 2000, 1, 1, 19.08), ("map", 2000, 1, 0, 24.39),
           ("inverse", 2000, 1, 1, 29.6), ("pseudo", 2000, 1, 1, 0.581), ("grid", 2000, 1, 1, 23.76),
           ("solve_h", 60013, 1, 0, 12.34), ("map", 60013, 30, 1, 38.12), ("inverse", 60013, 30, 1, 75.06),
           ("inverse", 60013, 30, 0, 80.56), ("pseudo", 60013, 1, 1, 14.16), ("grid", 60013, 1, 1, 746.4)]


@pytest.mark.parametrize("call,n,per_cell,precision,mib", BUDGETS)
def test_budgets_that_held_a_call_still_do(call, n, per_cell, precision, mib):
    """Workspaces shrink, or are given up for slower forms, before a call is
    refused; the result is the one without a budget, bit for bit."""
    L = lib()
    p = synth.lognormal_particles(n, 3 if n < 10000 else 4, ngrid=64)
    x, y, z, m, h = dev_particles(p)
    out = []
    for budget in (0, int(mib * 2 ** 20)):
        ctx = L.map_init(L.map_config_default(precision=precision, hbm_budget=budget))
        try:
            if call == "solve_h":
                L.solve_h(ctx, L.make_particles(x, y, z, None, h))
                out.append([h.clone()])
            elif call == "pseudo":
                o = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(5)]
                L.build_pseudo_particles(ctx, L.make_particles(x, y, z, m, torch.full_like(x, 0.03)), [0.5, 0.5, 0.5],
                                         L.make_particles(*o))
                out.append(o)
            elif call == "grid":
                g, _ = L.map_grid_build(ctx, x, y, z, lloyd=1, merge_tol=1e-9)
                out.append(list(L.map_grid_copy(ctx, g).values()))
            else:
                keep = np.sort(np.random.default_rng(9).choice(n, n // per_cell, replace=False))
                grid = synth.voronoi(p.pos()[keep])
                if not out:
                    hctx = L.map_init(L.map_config_default(precision=1))
                    L.solve_h(hctx, L.make_particles(x, y, z, None, h))
                    L.map_destroy(hctx)
                hd = L.map_grid_upload(ctx, L.grid_to_device(grid))
                mass = torch.empty(grid.ncell, dtype=torch.float64, device="cuda")
                L.map_particles_to_cells(ctx, L.make_particles(x, y, z, m, h), hd, mass)
                out.append([mass])
                if call == "inverse":
                    out[-1].append(L.map_cells_to_particles(ctx, torch.ones_like(mass), torch.empty_like(x)))
        finally:
            L.map_destroy(ctx)
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("precision,mib", [(1, 19.08), (0, 24.39)])
def test_a_tight_budget_walks_once_per_call(precision, mib):
    """A call whose budget did not hold the pair walk's pool leaves it out of
    the next ones, which launch as much as without a budget."""
    L = lib()
    p = synth.lognormal_particles(2000, 3, ngrid=64)
    grid = synth.voronoi(p.pos())
    x, y, z, m, h = dev_particles(p)
    hctx = L.map_init(L.map_config_default(precision=1))
    L.solve_h(hctx, L.make_particles(x, y, z, None, h))
    L.map_destroy(hctx)
    n = []
    for budget in (0, int(mib * 2 ** 20)):
        ctx = L.map_init(L.map_config_default(precision=precision, hbm_budget=budget))
        try:
            hd = L.map_grid_upload(ctx, L.grid_to_device(grid))
            mass = torch.empty(grid.ncell, dtype=torch.float64, device="cuda")
            at = []
            for _ in range(3):
                L.map_particles_to_cells(ctx, L.make_particles(x, y, z, m, h), hd, mass)
                at.append(L.map_get_work(ctx)[1])
            n.append((at[0], at[1] - at[0], at[2] - at[1]))
        finally:
            L.map_destroy(ctx)
    print(n)
    assert n[1][1:] == n[0][1:]
