"""What the framework is measured on: the calls that a radiation-hydrodynamics
program makes of it, at the sizes of this repository's configurations, tests
and benchmark.

Kinds of case
  step      one hydro step on a resident grid: solve_h, then the mapping of
            the particles to the cells, in one of the builds (mixed, fp64,
            table)
  coupling  the whole host-to-host coupling step: particles, grid and the
            cells' ionic fraction come from page-locked host memory; upload,
            solve_h, mapping, inverse mapping, results back to the host
  batch     many uneven snapshots: solve_h_batch and one map_batch
  serve     the serving loop: requests of uneven sizes submitted together,
            grids resident by id, results in host memory
  pseudo    the reduction: octree, walk, pseudo-particles and their h, then
            the mapping of the reduced set on its own grid
  grid      grid construction on the device: merging, Lloyd iterations, cells
  inverse   per-cell values carried back to the particles (Eq. 4), again and
            again with new values on one mapping's pair list

exact() gives the 64-bit values with torch alone: the smoothing length as the
root of Eq. (7) by bisection, the pair integrals from an antiderivative of the
kernel's excess over a point mass term by term, the walk level by level.
"""
import math

import numpy as np
import torch

import paper_2404_17084_gb300 as L
import synth

HFACT = 1.2
LEAF = 16
PRECISION = {"fp64": L.MAP_FP64, "mixed": L.MAP_MIXED, "table": L.MAP_TABLE}


def listed():
    return [
        # the smallest calls: a test problem or one small region, where launches and waits count
        {"name": "step_mixed_1k", "kind": "step", "precision": "mixed", "n": 1031, "field": "uniform", "sigma": 0.0},
        # the plain mapping of the uniform medium, every wedge in FP64
        {"name": "step_fp64_4k", "kind": "step", "precision": "fp64", "n": 4096, "field": "uniform", "sigma": 0.0},
        # an ordinary snapshot of the batch and serving ranges, an odd count
        {"name": "step_mixed_60k", "kind": "step", "precision": "mixed", "n": 60013, "field": "clumpy", "sigma": 1.5},
        # the clumpy cloud, the benchmark's headline size
        {"name": "step_mixed_1m", "kind": "step", "precision": "mixed", "n": 1 << 20, "field": "clumpy", "sigma": 1.5},
        # the clumpy cloud in the FP64 build: reference runs that the mixed build is checked against
        {"name": "step_fp64_50k", "kind": "step", "precision": "fp64", "n": 50021, "field": "clumpy", "sigma": 1.5},
        # one coupling step of a hydro code that lives on the host, forward and inverse
        {"name": "coupling_mixed_150k", "kind": "coupling", "precision": "mixed", "n": 150001, "field": "clumpy",
         "sigma": 1.5},
        # uneven snapshots in one batch
        {"name": "batch_mixed_24", "kind": "batch", "precision": "mixed", "nsnap": 24, "log2_lo": 10.0,
         "log2_hi": 16.0, "sizes": 3},
        # requests arriving together at the serving loop
        {"name": "serve_mixed_12", "kind": "serve", "precision": "mixed", "nreq": 12, "log2_med": 14.0,
         "log2_hi": 16.5, "sizes": 5},
        # the reduction of a large cloud around its source, and the reduced mapping
        {"name": "pseudo_4m", "kind": "pseudo", "precision": "mixed", "n": 1 << 22, "theta": 0.5, "r_part": 0.0,
         "r_leaf": 0.0},
        # the same with the walk controls on: full resolution near the source, thousands of nodes to solve for
        {"name": "pseudo_zoom_1m", "kind": "pseudo", "precision": "mixed", "n": 1000003, "theta": 0.5, "r_part": 0.02,
         "r_leaf": 0.05},
        # the grid of a clumpy snapshot with the five Lloyd iterations of Section II-A
        {"name": "grid_lloyd_130k", "kind": "grid", "n": 130003, "field": "clumpy", "sigma": 1.5, "lloyd": 5},
        # ionic fractions back to the particles after each radiative transfer iteration
        {"name": "inverse_200k", "kind": "inverse", "precision": "mixed", "n": 200003, "field": "clumpy",
         "sigma": 1.5},
    ]


def draw(rng):
    def log_size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    def field():
        return {"field": "uniform", "sigma": 0.0} if rng.random() < 0.4 else \
            {"field": "clumpy", "sigma": round(rng.uniform(1.0, 2.0), 3)}

    k = rng.choice(["step", "step", "step", "step", "coupling", "batch", "serve", "pseudo", "pseudo", "grid", "grid",
                    "inverse"])
    if k == "step":
        p = rng.choice(["mixed", "mixed", "fp64", "table"])
        hi = {"mixed": 1 << 20, "fp64": 60000, "table": 300000}[p]
        return {"kind": k, "precision": p, "n": log_size(1024, hi), **field()}
    if k == "coupling":
        return {"kind": k, "precision": "mixed", "n": log_size(4096, 150000), **field()}
    if k == "batch":
        return {"kind": k, "precision": rng.choice(["mixed", "mixed", "table"]), "nsnap": rng.randint(4, 24),
                "log2_lo": 10.0, "log2_hi": round(rng.uniform(12.0, 16.0), 2), "sizes": rng.randint(0, 1 << 20)}
    if k == "serve":
        return {"kind": k, "precision": "mixed", "nreq": rng.randint(4, 12), "log2_med": round(rng.uniform(12.5, 14.0), 2),
                "log2_hi": 16.5, "sizes": rng.randint(0, 1 << 20)}
    if k == "pseudo":
        zoom = rng.random() < 0.5
        return {"kind": k, "precision": "mixed", "n": log_size(1 << 15, (1 << 20) if zoom else (1 << 22)),
                "theta": round(rng.uniform(0.4, 0.8), 3), "r_part": round(rng.uniform(0.0, 0.02), 4) if zoom else 0.0,
                "r_leaf": round(rng.uniform(0.02, 0.05), 4) if zoom else 0.0}
    if k == "grid":
        return {"kind": k, "n": log_size(1000, 130000), **field(), "lloyd": rng.choice([0, 1, 5])}
    return {"kind": k, "precision": "mixed", "n": log_size(2000, 200000), **field()}


# ---------------------------------------------------------------- inputs

def _clumpy(n, seed, sigma):
    """synth.lognormal_particles' field and law, the voxels looked up on the GPU (a large cloud in a tenth of the time)."""
    ngrid = 128 if n > 400000 else 64
    rng = np.random.default_rng(seed)
    f = synth.gaussian_random_field(ngrid, -4.0, rng)
    cdf = np.cumsum(np.exp((f - f.mean()) / f.std() * sigma).ravel())
    vox = torch.searchsorted(_dev(cdf), _dev(rng.random(n) * cdf[-1]), right=True).clamp(max=cdf.size - 1).cpu().numpy()
    u = rng.random((3, n))
    x, y, z = ((c + u[k]) / ngrid for k, c in enumerate((vox // ngrid ** 2, vox // ngrid % ngrid, vox % ngrid)))
    return synth.Particles(x, y, z, np.full(n, 1.0 / n))


def _particles(case, seed):
    if case["field"] == "uniform":
        return synth.uniform_particles(case["n"], seed)
    return _clumpy(case["n"], seed, case["sigma"])


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _pinned(a):
    return torch.as_tensor(np.ascontiguousarray(a)).pin_memory()


_GRID = ("cell_face_off", "face_vert_off", "face_vert", "face_plane", "vx", "vy", "vz", "site")


def _several(case):
    """(particles, clumpy, sigma) of each snapshot of a batch or request of a server: the case's, whatever the seed."""
    rng = np.random.default_rng(case["sizes"])
    if case["kind"] == "batch":
        spec = synth.batch_specs(case["nsnap"], case["sizes"], case["log2_lo"], case["log2_hi"])
        return [(n, kind == "clumpy", sigma) for n, kind, sigma, _ in spec]
    return [(int(2 ** np.clip(rng.normal(case["log2_med"], 1.5), 12.0, case["log2_hi"])), j % 2 == 0,
             float(rng.uniform(1.0, 2.0))) for j in range(case["nreq"])]


def _several_inputs(case, seed):
    seeds = np.random.default_rng(seed).integers(1, 2 ** 31, 64)
    parts = [_clumpy(n, int(s), sigma) if clumpy else synth.uniform_particles(n, int(s))
             for (n, clumpy, sigma), s in zip(_several(case), seeds)]
    return parts, [synth.voronoi(p.pos()) for p in parts]


def _cell_values(n, seed):
    return np.random.default_rng(seed + 77).random(n)


def _pseudo_inputs(case, seed):
    p = _clumpy(case["n"], seed, 1.5)
    x, y, z, m = (_dev(a) for a in (p.x, p.y, p.z, p.m))
    h = _leaf_guess(torch.stack([x, y, z], 1))  # the smoothing lengths a program carries along
    i = int(torch.argmin(h))  # the source sits at the densest particle
    src = [float(x[i]), float(y[i]), float(z[i])]
    return x, y, z, m, h, src


def _room(case):
    """Places for pseudo-particles: a program's own estimate, ample."""
    return 65536 if case["r_leaf"] == 0.0 else 65536 + case["n"] // 2


class _Server:
    """A serving loop that ends with its state."""

    def __init__(self, precision):
        self.srv = L.map_server_create(L.map_server_config_default(precision=precision))

    def __del__(self):
        L.map_server_destroy(self.srv)


def prepare(case, seed):
    k = case["kind"]
    S = {"case": case}
    if k == "grid":
        p = _particles(case, seed)
        S.update(x=_dev(p.x), y=_dev(p.y), z=_dev(p.z), mapper=L.ExactMapper(L.MAP_MIXED), tol=1e-6 * p.n ** (-1.0 / 3.0))
        # the program's own grid arrays, with room for what a seed may give: a site has about 15.5 faces, 82 loop
        # entries and 27 vertices, fewer in a small cube
        nf, nl, nv = 18 * p.n + 64, 96 * p.n + 256, 32 * p.n + 128
        z = lambda n, t=torch.float64: torch.zeros(n, dtype=t, device="cuda")  # noqa: E731
        S["out"] = {"cell_face_off": z(p.n + 1, torch.int64), "face_vert_off": z(nf, torch.int64),
                    "face_vert": z(nl, torch.int32), "face_plane": z((nf, 4)), "vx": z(nv), "vy": z(nv), "vz": z(nv),
                    "site": z((p.n, 3)), "volume": z(p.n), "kept": z(p.n, torch.int64)}
        return S
    precision = PRECISION[case["precision"]]
    if k == "serve":
        parts, grids = _several_inputs(case, seed)
        S.update(server=_Server(precision), parts=parts, grids=grids)
        return S
    S["mapper"] = M = L.ExactMapper(precision, theta=case.get("theta", 0.5))
    if k == "batch":
        parts, grids = _several_inputs(case, seed)
        S["handles"] = [M.upload(g) for g in grids]
        S["parts"] = [tuple(_dev(a) for a in (p.x, p.y, p.z, p.m)) for p in parts]
        S["n"] = sum(p.n for p in parts)
        S["out"] = {f: torch.empty(S["n"], dtype=torch.float64, device="cuda") for f in ("h", "mass", "rho")}
        S["route"] = torch.empty(S["n"], dtype=torch.int32, device="cuda")
        return S
    if k == "pseudo":
        x, y, z, m, h, src = _pseudo_inputs(case, seed)
        w = _walk(case, x, y, z, m, h, src)
        pos = torch.stack([w["x"], w["y"], w["z"]], 1).cpu().numpy()
        g = synth.voronoi(pos[synth.dedupe_sites(pos)])
        S.update(x=x, y=y, z=z, m=m, h=h, src=src, grid=M.upload(g), ncell=g.ncell)
        z = lambda t=torch.float64: torch.zeros(_room(case), dtype=t, device="cuda")  # noqa: E731
        S["out"] = {**{f: z() for f in ("x", "y", "z", "m", "h", "mass", "rho")}, "kind": z(torch.int32),
                    "ident": z(torch.int64)}
        return S
    p = _particles(case, seed)
    g = synth.voronoi(p.pos())
    S["ncell"] = g.ncell
    if k == "coupling":
        S["host"] = [_pinned(a) for a in (p.x, p.y, p.z, p.m)]
        S["grid"] = {f: _pinned(getattr(g, f)) for f in _GRID}
        S["ion"] = _pinned(_cell_values(g.ncell, seed))
        S["back"] = [torch.empty(c, dtype=torch.float64).pin_memory() for c in (p.n, g.ncell, g.ncell, p.n)]
        return S
    S["x"], S["y"], S["z"], S["m"] = (_dev(a) for a in (p.x, p.y, p.z, p.m))
    S["handle"] = M.upload(g)
    if k == "inverse":
        h, _ = M.solve_h(S["x"], S["y"], S["z"])
        M.map(S["handle"], g.ncell, S["x"], S["y"], S["z"], S["m"], h)
        S["ion"] = _dev(_cell_values(g.ncell, seed))
        S["h"] = h
    return S


# ---------------------------------------------------------------- one pass

def run(S):
    return _RUN[S["case"]["kind"]](S)


def _run_step(S):
    M = S["mapper"]
    h, route = M.solve_h(S["x"], S["y"], S["z"])
    mass, rho = M.map(S["handle"], S["ncell"], S["x"], S["y"], S["z"], S["m"], h)
    return {"h": h, "route": route, "mass": mass, "rho": rho}


def _run_coupling(S):
    M = S["mapper"]
    x, y, z, m = (a.to("cuda", non_blocking=True) for a in S["host"])
    grid = L.map_grid_upload(M.ctx, S["grid"])
    h, _ = M.solve_h(x, y, z)
    mass, rho = M.map(grid, S["ncell"], x, y, z, m, h)
    ion = L.map_cells_to_particles(M.ctx, S["ion"].to("cuda", non_blocking=True), torch.empty_like(x))
    for to, a in zip(S["back"], (h, mass, rho, ion)):
        to.copy_(a, non_blocking=True)
    L.map_grid_release(M.ctx, grid)
    torch.cuda.current_stream().synchronize()
    return dict(zip(("h", "mass", "rho", "ion"), S["back"]))


def _run_batch(S):
    ctx, out = S["mapper"].ctx, S["out"]
    cut = np.cumsum([0] + [p[0].numel() for p in S["parts"]])
    of = lambda t: [t[a:b] for a, b in zip(cut[:-1], cut[1:])]  # noqa: E731
    h, mass, rho, route = of(out["h"]), of(out["mass"]), of(out["rho"]), of(S["route"])
    sets = [L.make_particles(x, y, z, m, hh) for (x, y, z, m), hh in zip(S["parts"], h)]
    L.solve_h_batch(ctx, sets, route)
    L.map_batch(ctx, sets, S["handles"], mass, rho)
    return {**out, "route": S["route"]}


def _run_serve(S):
    srv, tickets, out = S["server"].srv, [], {"h": [], "mass": [], "rho": []}
    for j, (p, g) in enumerate(zip(S["parts"], S["grids"])):
        mass, rho, h = np.empty(g.ncell), np.empty(g.ncell), np.empty(p.n)
        tickets.append(L.map_server_submit(srv, p.x, p.y, p.z, p.m, g, mass, rho, h, grid_id=j))
        for f, a in (("h", h), ("mass", mass), ("rho", rho)):
            out[f].append(a)
    for t in tickets:
        L.map_server_wait(srv, t)
    return out


def _run_pseudo(S):
    ctx, case, out = S["mapper"].ctx, S["case"], S["out"]
    full = L.make_particles(S["x"], S["y"], S["z"], S["m"], S["h"])
    of = [out[f] for f in ("x", "y", "z", "m", "h")]
    n = L.build_pseudo_particles(ctx, full, S["src"], L.make_particles(*of), out["kind"], out["ident"],
                                 r_part=case["r_part"], r_leaf=case["r_leaf"])
    L.map_particles_to_cells(ctx, L.make_particles(*(a[:n] for a in of)), S["grid"], out["mass"][:S["ncell"]],
                             out["rho"][:S["ncell"]])
    return {**out, "n": n}


def _run_grid(S):
    ctx = S["mapper"].ctx
    grid, n = L.map_grid_build(ctx, S["x"], S["y"], S["z"], lloyd=S["case"]["lloyd"], merge_tol=S["tol"],
                               kept=S["out"]["kept"])
    L.map_grid_volumes(ctx, grid, S["out"]["volume"][:n])
    for f, a in L.map_grid_copy(ctx, grid).items():
        S["out"][f][:a.shape[0]].copy_(a)
    L.map_grid_release(ctx, grid)
    return S["out"]


def _run_inverse(S):
    return L.map_cells_to_particles(S["mapper"].ctx, S["ion"], torch.empty_like(S["x"]))


_RUN = {"step": _run_step, "coupling": _run_coupling, "batch": _run_batch, "serve": _run_serve, "pseudo": _run_pseudo,
        "grid": _run_grid, "inverse": _run_inverse}


# ---------------------------------------------------------------- what a pass cannot do without

PAIRS = 125.0  # pairs per cell
PAIR_OPS = 10400.0  # arithmetic of one pair integral: faces, edges within the support, pieces
GRID_BYTES = 1560.0  # a cell's CSR arrays: 15.4 faces, 81 loop entries, 27 vertices


def work(case):
    k = case["kind"]
    if k == "batch":
        lo, hi = 2.0 ** case["log2_lo"], 2.0 ** case["log2_hi"]
        n = case["nsnap"] * (hi - lo) / math.log(hi / lo)
    elif k == "serve":
        n = case["nreq"] * 1.5 * 2.0 ** case["log2_med"]
    else:
        n = case["n"]
    if k == "inverse":
        return {"bytes": n * (PAIRS * 12.0 + 32.0), "flops": n * PAIRS * 2.0}
    if k == "pseudo":
        out = 900.0 if case["r_leaf"] == 0.0 else n * 0.016
        return {"bytes": n * 40.0 + out * (60.0 + GRID_BYTES), "flops": n * 40.0 + out * PAIRS * PAIR_OPS}
    if k == "grid":
        return {"bytes": n * (48.0 * (1 + case["lloyd"]) + GRID_BYTES), "flops": n * (1 + case["lloyd"]) * 9000.0}
    more = PAIRS * 2.0 if k == "coupling" else 0.0
    return {"bytes": n * (56.0 + GRID_BYTES + (24.0 if k == "coupling" else 0.0)),
            "flops": n * (PAIRS * PAIR_OPS + more)}


# ---------------------------------------------------------------- 64-bit values

def _sorted_keys(pos):
    c = torch.clamp(torch.floor(pos * 2097152.0), 0.0, 2097151.0).to(torch.int64)
    key = torch.zeros(pos.shape[0], dtype=torch.int64, device=pos.device)
    for b in range(21):
        for ax in range(3):
            key |= ((c[:, ax] >> b) & 1) << (3 * b + 2 - ax)
    return torch.sort(key, stable=True)


def _leaf_guess(pos):
    """hfact * side / count^(1/3) of each particle's octree leaf."""
    key, order = _sorted_keys(pos)
    level = torch.full_like(key, -1)
    count = torch.ones_like(key)
    for lev in range(22):
        _, inv, c = torch.unique_consecutive(key >> (3 * (21 - lev)), return_inverse=True, return_counts=True)
        c = c[inv]
        new = (level < 0) & ((c <= LEAF) | (lev == 21))
        level[new], count[new] = lev, c[new]
        if bool((level >= 0).all()):
            break
    h0 = torch.empty(pos.shape[0], dtype=torch.float64, device=pos.device)
    h0[order] = HFACT * torch.pow(2.0, -level.double()) / count.double() ** (1.0 / 3.0)
    return h0


def _root(dist, h0):
    """h = hfact n(h)^(-1/3) on [h0/16, 16 h0], n from each row's distances; h0 where there is none."""
    def g(h):
        q = dist / h[:, None]
        w = torch.where(q < 1.0, 1.0 - 1.5 * q * q + 0.75 * q ** 3, 0.25 * torch.clamp(2.0 - q, min=0.0) ** 3).sum(1)
        return h - HFACT * (w / (math.pi * h ** 3)) ** (-1.0 / 3.0)

    a, b = h0 / 16.0, h0 * 16.0
    none = (g(a) >= 0.0) | (g(b) <= 0.0)
    for _ in range(62):
        mid = 0.5 * (a + b)
        low = g(mid) < 0.0
        a, b = torch.where(low, mid, a), torch.where(low, b, mid)
    return torch.where(none, h0, 0.5 * (a + b))


def _exact_h(pos, h0):
    n = pos.shape[0]
    k = min(n, 192)
    p32 = (pos - 0.5).float()
    h = torch.empty_like(h0)
    rows = max(1, int(4e8 // n))
    for r in range(0, n, rows):
        d2 = sum((p32[r:r + rows, None, ax] - p32[None, :, ax]) ** 2 for ax in range(3))
        nb = torch.topk(d2, k, dim=1, largest=False).indices
        del d2
        d = (pos[nb] - pos[r:r + rows, None, :]).square().sum(2).sqrt()
        h[r:r + rows] = _root(d, h0[r:r + rows])
        far = (2.0 * h[r:r + rows] > 0.9999 * d.max(1).values) & (k < n)
        for i in torch.nonzero(far).flatten().tolist():
            h[r + i] = _root((pos - pos[r + i]).square().sum(1).sqrt()[None], h0[r + i:r + i + 1])[0]
    return h


class _Cells:
    """A grid's faces and edges on the GPU, in 64 bits."""

    def __init__(self, g):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
        self.cfo, self.fvo = t(g.cell_face_off), t(g.face_vert_off)
        self.site, plane = t(g.site), t(g.face_plane)
        self.n, self.d = plane[:, :3].contiguous(), plane[:, 3].contiguous()
        v = torch.stack([t(g.vx), t(g.vy), t(g.vz)], 1)
        nf, nl = len(self.d), len(g.face_vert)
        face_of = torch.repeat_interleave(torch.arange(nf, device="cuda"), self.fvo[1:] - self.fvo[:-1])
        self.cell_of = torch.repeat_interleave(torch.arange(len(self.site), device="cuda"), self.cfo[1:] - self.cfo[:-1])
        nxt = torch.arange(1, nl + 1, device="cuda")
        last = self.fvo[1:] - 1
        nxt[last] = self.fvo[:-1]
        fv = t(g.face_vert).long()
        self.va, vb = v[fv], v[fv[nxt]]
        e = vb - self.va
        self.len = e.norm(dim=1)
        self.e = e / self.len.clamp(min=1e-300)[:, None]
        self.m = torch.linalg.cross(self.n[face_of], self.e)
        s = self.site[self.cell_of[face_of]]
        far2 = torch.zeros(len(self.site), dtype=torch.float64, device="cuda")
        far2.scatter_reduce_(0, self.cell_of[face_of], (self.va - s).square().sum(1), "amax")
        self.R = far2.sqrt()
        cnt = (self.fvo[1:] - self.fvo[:-1]).double()
        self.mid = torch.zeros_like(self.n).index_add_(0, face_of, self.va) / cnt[:, None]
        rad2 = torch.zeros_like(self.d).scatter_reduce_(0, face_of, (self.va - self.mid[face_of]).square().sum(1), "amax")
        self.rad = rad2.sqrt()
        cr = torch.linalg.cross(self.va - self.mid[face_of], vb - self.mid[face_of])
        area = 0.5 * (torch.zeros_like(self.n).index_add_(0, face_of, cr) * self.n).sum(1)
        hgt = self.d - (self.n * self.site[self.cell_of]).sum(1)
        self.vol = torch.zeros_like(self.R).index_add_(0, self.cell_of, area * hgt / 3.0)


def _spread(lo, cnt):
    """(row, position) of every entry of the ranges [lo, lo + cnt)."""
    row = torch.repeat_interleave(torch.arange(len(cnt), device=cnt.device), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    return row, lo[row] + torch.arange(len(row), device=cnt.device) - first[row]


def _excess(u):
    """4 pi E(u): what the kernel's H differs by from a point mass."""
    i = 1.0 / u - 1.4 + u ** 2 * (2.0 / 3.0) - 0.3 * u ** 4 + 0.1 * u ** 5
    o = torch.clamp(2.0 - u, min=0.0) ** 5 * (1.0 + u) / u / 30.0
    return torch.where(u < 1.0, i, o)


def _edge_integral(r0, R0, a, b):
    """4 pi int_a^b r0 [E(U) - E(r0)] R0 / (R0^2 + s^2) ds, U^2 = r0^2 + R0^2 + s^2."""
    c2 = r0 * r0 + R0 * R0
    s1, s2 = torch.clamp(1.0 - c2, min=0.0).sqrt(), torch.clamp(4.0 - c2, min=0.0).sqrt()

    def terms(s):
        U = (c2 + s * s).sqrt()
        Lg = torch.asinh(s / c2.sqrt())
        om = torch.atan2(s, R0) - torch.atan2(r0 * s, R0 * U)
        k = r0 * R0
        i1 = 0.5 * (s * U + c2 * Lg)
        g1 = k * Lg - r0 ** 2 * om
        g2 = k * s
        g3 = k * i1 + r0 ** 2 * g1
        g4 = k * (c2 * s + s ** 3 / 3.0) + r0 ** 2 * g2
        g5 = k * 0.25 * (s * U ** 3 + 3.0 * c2 * i1) + r0 ** 2 * g3
        return om, g2, g3, g4, g5

    def inner(t):
        om, g2, g3, g4, g5 = t
        return -om + g2 * (2.0 / 3.0) - 0.3 * g4 + 0.1 * g5

    def middle(t):
        om, g2, g3, g4, g5 = t
        return (-32.0 * om + 40.0 * g2 - 30.0 * g3 + 9.0 * g4 - g5) / 30.0

    x0, x1 = torch.minimum(torch.maximum(a, -s2), b), torch.maximum(torch.minimum(b, s2), a)
    x1 = torch.maximum(x0, x1)
    y0, y1 = torch.minimum(torch.maximum(x0, -s1), x1), torch.maximum(torch.minimum(x1, s1), x0)
    y1 = torch.maximum(y0, y1)
    t0, t1 = terms(y0), terms(y1)
    out = inner(t1) - inner(t0) - middle(t1) + middle(t0) + middle(terms(x1)) - middle(terms(x0))
    phi = lambda lo, hi: torch.atan2((hi - lo) * R0, R0 * R0 + lo * hi)  # noqa: E731
    e0 = r0 * _excess(r0)
    em = (2.0 - r0) ** 5 * (1.0 + r0) / 30.0
    dm = phi(x0, y0) + phi(y1, x1)
    return out + (em - e0) * dm - e0 * (phi(a, x0) + phi(x1, b))


def _exact_pairs(C, pos, h, each):
    """each(cell, particle, fraction) over all pairs that can be nonzero, in chunks."""
    n, nc = pos.shape[0], len(C.R)
    p32, s32 = (pos - 0.5).float(), (C.site - 0.5).float()
    reach = (2.0 * h).float()
    rows = max(1, int(4e8 // n))
    for r in range(0, nc, rows):
        d2 = sum((s32[r:r + rows, None, ax] - p32[None, :, ax]) ** 2 for ax in range(3))
        hit = torch.nonzero(d2 < (reach[None, :] + C.R[r:r + rows, None].float()) ** 2 * 1.00001 + 1e-12)
        del d2
        for k in range(0, len(hit), 500000):
            c, p = hit[k:k + 500000, 0] + r, hit[k:k + 500000, 1]
            pair, f = _spread(C.cfo[c], C.cfo[c + 1] - C.cfo[c])
            y, hi = pos[p], 1.0 / h[p]
            r0 = (C.d[f] - (C.n[f] * y[pair]).sum(1)) * hi[pair]
            out = torch.zeros(len(c), dtype=torch.float64, device="cuda").index_add_(0, pair, (r0 < 0.0).double())
            near = (r0.abs() < 2.0) & (((C.mid[f] - y[pair]).norm(dim=1) - C.rad[f]) * hi[pair] < 2.0)
            pair, f, r0 = pair[near], f[near], r0[near]
            frac = (out == 0.0).double()
            rec, e = _spread(C.fvo[f], C.fvo[f + 1] - C.fvo[f])
            pair, r0 = pair[rec], r0[rec]
            d, hi = y[pair] - C.va[e], hi[pair]
            R0 = (C.m[e] * d).sum(1) * hi
            a = -(C.e[e] * d).sum(1) * hi
            one = torch.ones_like(R0)
            sign = torch.where((r0 >= 0.0) == (R0 >= 0.0), one, -one)
            v = _edge_integral(r0.abs().clamp(min=1e-12), R0.abs().clamp(min=1e-12), a, a + C.len[e] * hi)
            frac.index_add_(0, pair, sign * v / (4.0 * math.pi))
            each(c, p, frac)


def _exact_map(p, g, ion=None):
    x = [_dev(a) for a in (p.x, p.y, p.z)]
    pos, m = torch.stack(x, 1), _dev(p.m)
    h = _exact_h(pos, _leaf_guess(pos))
    C = _Cells(g)
    mass, back = torch.zeros_like(C.R), torch.zeros_like(h)

    def each(c, a, f):
        mass.index_add_(0, c, m[a] * f)
        if ion is not None:
            back.index_add_(0, a, ion[c] * f)

    _exact_pairs(C, pos, h, each)
    return h, mass, mass / C.vol, back


def _walk(case, x, y, z, m, h, src):
    """The walk's pseudo-particles in depth-first order; h of the accepted nodes where every member is a candidate."""
    pos = torch.stack([x, y, z], 1)
    key, order = _sorted_keys(pos)
    pos, m, h = pos[order], m[order], h[order]
    s = torch.tensor(src, dtype=torch.float64, device="cuda")
    lo = torch.zeros(1, dtype=torch.int64, device="cuda")
    cnt = torch.full_like(lo, len(m))
    rows, members, extracted = [], [], []
    for lev in range(22):
        node, at = _spread(lo, cnt)
        z1 = torch.zeros(len(lo), dtype=torch.float64, device="cuda")
        mass = z1.index_add(0, node, m[at])
        com = torch.zeros(len(lo), 3, dtype=torch.float64, device="cuda").index_add_(0, node, pos[at] * m[at, None]) / mass[:, None]
        size = z1.scatter_reduce(0, node, (pos[at] - com[node]).square().sum(1), "amax").sqrt()
        r = (com - s).norm(dim=1)
        leaf = (cnt <= LEAF) | (lev == 21)
        opened = (r == 0.0) | (size ** 2 > case["theta"] ** 2 * r ** 2)
        if case["r_part"] > 0.0:
            opened |= r < case["r_part"] + size
        if case["r_leaf"] > 0.0:
            opened |= ~leaf & (r < case["r_leaf"] + size)
        keep, ext = ~opened, opened & leaf
        guess = torch.where(size > 0.0, HFACT * 2.0 * size, h[lo])
        rows.append(torch.cat([lo[keep, None].double(), com[keep], mass[keep, None], guess[keep, None]], 1))
        members += [com[keep], com[ext]]
        extracted.append(_spread(lo[ext], cnt[ext])[1])
        down = opened & ~leaf
        if not bool(down.any()):
            break
        node, at = _spread(lo[down], cnt[down])
        new = torch.ones(len(at), dtype=torch.bool, device="cuda")
        pre = key[at] >> (3 * (20 - lev))
        new[1:] = (pre[1:] != pre[:-1]) | (node[1:] != node[:-1])
        first = torch.nonzero(new).flatten()
        lo = at[first]
        cnt = torch.diff(first, append=torch.tensor([len(at)], device="cuda"))
    rows, members, at = torch.cat(rows), torch.cat(members), torch.cat(extracted)
    hn = None
    if len(members) <= 10000:
        hn = torch.cat([_root((members[None] - q[:, None, 1:4]).square().sum(2).sqrt(), q[:, 5])
                        for q in rows.split(1024)]) if len(rows) else rows[:, 5]
    first = torch.cat([rows[:, 0], at.double()])
    by = torch.argsort(first)
    cat = lambda i, v: torch.cat([rows[:, i], v[at]])[by]  # noqa: E731
    return {"x": cat(1, pos[:, 0]), "y": cat(2, pos[:, 1]), "z": cat(3, pos[:, 2]), "m": cat(4, m),
            "h": None if hn is None else torch.cat([hn, h[at]])[by]}


def exact(case, seed):
    k = case["kind"]
    if k == "grid" or case["precision"] == "table":
        return None  # cells: no form of them in plain tensor operations; the table is not exact by its nature
    if k == "pseudo":
        # the mapping's values depend on the walk's own h: left to the other kinds
        w = _walk(case, *_pseudo_inputs(case, seed))
        return {f: None if v is None else torch.nn.functional.pad(v, (0, _room(case) - len(v))) for f, v in w.items()}
    if k in ("batch", "serve"):
        got = [_exact_map(p, g) for p, g in zip(*_several_inputs(case, seed))]
        if k == "serve":
            return {"h": [v[0] for v in got], "mass": [v[1] for v in got], "rho": [v[2] for v in got]}
        return {"h": torch.cat([v[0] for v in got]), "mass": torch.cat([v[1] for v in got]),
                "rho": torch.cat([v[2] for v in got])}
    if case["n"] > 260000:
        return None  # over 20 seconds
    p = _particles(case, seed)
    g = synth.voronoi(p.pos())
    h, mass, rho, back = _exact_map(p, g, _dev(_cell_values(g.ncell, seed)) if k in ("coupling", "inverse") else None)
    if k == "inverse":
        return back
    return {"h": h, "mass": mass, "rho": rho, **({"ion": back} if k == "coupling" else {})}
