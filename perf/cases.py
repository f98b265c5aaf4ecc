"""The work this framework is used for, as cases that can be timed: single
Poisson solves in both precisions, under every kind of boundary rule, from
device and host memory, with and without the acceleration, a batch of uneven
grids and a burst of requests to the serving loop.

``listed()`` names the cases, ``draw(rng)`` makes another one of the same
ranges, ``prepare`` / ``run`` are one call as a user's program makes it,
``work`` is what the call cannot do without and ``exact`` is the solution of
the discrete problem by separable eigenvectors in 64 bits.

Grid sides are powers of two (the solver takes no others); what is uneven here
is the shape of the boxes and the mix of sizes in batches and bursts.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2302_13903_gb300 as mg

KINDS = {"P": mg.PERIODIC, "F": mg.FIXED, "Z": mg.ZEROGRAD, "O": mg.OPEN}
# A rule is one letter for all faces, or three pairs (x- x+, y- y+, z- z+).
SLAB = "PPPPFF"  # periodic in x and y, phi = 0 on both z faces

BATCH_SIZES = (16, 32, 64, 128)
SERVE_SIZES = (32, 64, 128, 256)


def listed():
    def solve(name, nx, ny, nz, rule, prec, tol, **kw):
        c = dict(name=name, kind="solve", nx=nx, ny=ny, nz=nz, rule=rule, prec=prec, tol=tol,
                 fixed_value=0.0, blobs=64, start="fmg", gravity=False, memory="device")
        c.update(kw)
        return c

    return [
        # The plain FP64 solver (the default precision).  Smallest: a code that
        # solves one small block at a time, where launches are all there is.
        solve("fp64_32_fixed", 32, 32, 32, "F", "fp64", 1e-8, fixed_value=0.25, blobs=4),
        # The paper's accuracy test at its size (Sec. 4.1.1).
        solve("fp64_64_periodic", 64, 64, 64, "P", "fp64", 1e-10),
        # An isolated object with multipole boundary values (Sec. 4.2.1).
        solve("fp64_256_open", 256, 256, 256, "O", "fp64", 1e-10, blobs=8),
        # The largest FP64 solve: the one the mixed path is compared with.
        solve("fp64_512_periodic", 512, 512, 512, "P", "fp64", 1e-10),
        # The mixed path.  Smallest request of the serving mix, loose tolerance.
        solve("mixed_32_zerograd", 32, 32, 32, "Z", "mixed", 1e-6, blobs=4),
        # A small accurate solve: latency of the coarse levels.
        solve("mixed_64_periodic", 64, 64, 64, "P", "mixed", 1e-10),
        # A CPU code that hands over page-locked host arrays.
        solve("mixed_128_fixed_host", 128, 128, 128, "F", "mixed", 1e-8, fixed_value=0.25, blobs=8,
              memory="host"),
        # A stratified box in a time-stepping code: flat box, a rule per face,
        # started from the last step's potential.
        solve("mixed_slab_restart", 256, 256, 128, SLAB, "mixed", 1e-9, start="guess"),
        # Self-gravity of an isolated object: potential and acceleration.
        solve("mixed_256_open_gravity", 256, 256, 256, "O", "mixed", 1e-10, blobs=8, gravity=True),
        # The headline: a cosmological box.
        solve("mixed_512_periodic", 512, 512, 512, "P", "mixed", 1e-10),
        # Many independent grids at once (mesh blocks, ensembles).
        dict(name="batch_512", kind="batch", grids=512, mix=1, tol=1e-10),
        # A burst of requests of mixed sizes, rules and tolerances to a server
        # whose hierarchies are resident.
        dict(name="serve_burst", kind="serve", requests=24, mix=1, slots=8),
    ]


def draw(rng: random.Random):
    kind = rng.choice(["solve"] * 6 + ["batch", "serve"])
    if kind == "batch":
        return dict(kind="batch", grids=int(2 ** rng.uniform(3, 8.5)) | 1, mix=rng.randrange(1 << 20),
                    tol=10.0 ** rng.uniform(-10, -8))
    if kind == "serve":
        return dict(kind="serve", requests=rng.randrange(4, 24), mix=rng.randrange(1 << 20),
                    slots=rng.choice([2, 4, 8]))
    prec = rng.choice(["fp64", "mixed"])
    # cells over the logarithm of the range; boxes halve y, z or both
    k = rng.choice([5, 6, 7, 8, 9] if prec == "mixed" else [5, 6, 7, 8])
    nx = 1 << k
    ny = nz = nx
    if rng.random() < 0.4:
        ny = nx >> rng.choice([0, 1])
        nz = nx >> rng.choice([0, 1, 2] if nx > 64 else [0, 1])
    rules = ["P", "P", "F", "Z", SLAB, "PPFZPP", "FZZZPP"]
    if ny == nx and nz == nx and nx <= 256:
        rules += ["O", "O"]
    rule = rng.choice(rules)
    return dict(kind="solve", nx=nx, ny=ny, nz=nz, rule=rule, prec=prec,
                tol=10.0 ** rng.uniform(-10, -6),
                fixed_value=rng.choice([0.0, 0.25]) if rule == "F" else 0.0,
                blobs=rng.randrange(1, 9) if rule == "O" else rng.randrange(4, 65),
                start=rng.choice(["fmg", "fmg", "fmg", "guess"]),
                gravity=rng.random() < 0.25,
                memory="device")


# --- inputs ---------------------------------------------------------------

def _faces(rule):
    return rule * 6 if len(rule) == 1 else rule


def _mean_free(rule):
    return not set(_faces(rule)) & {"F", "O"}


def _source(n, h, rule, blobs, seed, shift=0.0):
    """Gaussian blobs (z, y, x) on the GPU, sigma 0.02-0.08 of the longest side
    and lognormal amplitudes; along periodic axes by the nearest image; around
    the centre for an open rule; ``shift`` moves every blob.  The mean is
    removed where no face fixes the potential's zero point."""
    rng = np.random.default_rng([seed, blobs])
    ext = np.array([m * h for m in n])
    if rule == "O":
        centres = ext * (0.5 + 0.15 * (rng.random((blobs, 3)) - 0.5))
        sigma = rng.uniform(0.02, 0.05, blobs)
    else:
        centres = ext * rng.random((blobs, 3))
        sigma = rng.uniform(0.02, 0.08, blobs)
    centres = centres + shift * rng.standard_normal((blobs, 3))
    amp = np.exp(rng.normal(0.0, 1.0, blobs))
    fac = []
    for a in range(3):
        d = (np.arange(n[a]) + 0.5) * h - centres[:, a:a + 1]
        if _faces(rule)[2 * a] == "P":
            d -= ext[a] * np.round(d / ext[a])
        fac.append(torch.from_numpy(np.exp(-0.5 * (d / sigma[:, None]) ** 2)).cuda())
    zy = (fac[2] * torch.from_numpy(amp).cuda()[:, None])[:, :, None] * fac[1][:, None, :]
    rho = (zy.reshape(blobs, -1).t() @ fac[0]).reshape(n[2], n[1], n[0]).contiguous()
    if _mean_free(rule):
        rho -= rho.mean()
    return rho


def _batch_grids(case):
    """[(n, rule, blobs)]: sizes with Zipf weights, rules evenly."""
    rng = np.random.default_rng([case["mix"], 7])
    w = 1.0 / np.arange(1, len(BATCH_SIZES) + 1)
    k = case["grids"]
    return list(zip(rng.choice(BATCH_SIZES, k, p=w / w.sum()).tolist(),
                    rng.choice(["P", "F", "Z"], k).tolist(), rng.integers(1, 9, k).tolist()))


def _requests(case):
    """[(n, rule, lmax, tol, blobs)]: sizes and rules evenly, tolerances over
    their logarithm."""
    rng = np.random.default_rng([case["mix"], 11])
    k = case["requests"]
    return list(zip(rng.choice(SERVE_SIZES, k).tolist(), rng.choice(["P", "F", "Z", "O"], k).tolist(),
                    rng.integers(0, 5, k).tolist(), (10.0 ** rng.uniform(-10, -6, k)).tolist(),
                    rng.integers(1, 9, k).tolist()))


def _box(case):
    return (case["nx"], case["ny"], case["nz"]), 1.0 / case["nx"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        grids = _batch_grids(case)
        rhos = [_source((n, n, n), 1.0 / n, rule, b, seed * 1009 + g)
                for g, (n, rule, b) in enumerate(grids)]
        flat = torch.zeros(sum(r.numel() for r in rhos), dtype=torch.float64, device="cuda")
        phis = [p.view(r.shape) for p, r in zip(flat.split([r.numel() for r in rhos]), rhos)]
        batch = mg.Batch([n for n, _, _ in grids], [1.0 / n for n, _, _ in grids],
                         [KINDS[r] for _, r, _ in grids])
        return dict(case=case, batch=batch, rhos=rhos, phis=phis, flat=flat)
    if kind == "serve":
        reqs = _requests(case)
        rhos = [_source((n, n, n), 1.0 / n, rule, b, seed * 1013 + q)
                for q, (n, rule, _, _, b) in enumerate(reqs)]
        server = mg.Server(64 << 30, slots=case["slots"])
        state = dict(case=case, reqs=reqs, rhos=rhos, phis=[torch.zeros_like(r) for r in rhos],
                     server=server)
        torch.cuda.synchronize()
        run(state)  # the server's hierarchies are resident before the burst
        return state
    n, h = _box(case)
    rule = case["rule"]
    rho = _source(n, h, rule, case["blobs"], seed)
    opts = dict(prec=case["prec"], mode_fmg=int(case["start"] == "fmg"),
                fixed_value=case["fixed_value"])
    bc = KINDS[rule] if len(rule) == 1 else [KINDS[r] for r in rule]
    solver = mg.Solver(n, h, bc, **opts)
    if case["prec"] == "mixed":
        solver.autotune()
    state = dict(case=case, solver=solver, rho=rho, phi=torch.zeros_like(rho))
    if case["gravity"]:
        state["g"] = torch.empty((3,) + tuple(rho.shape), dtype=torch.float64, device="cuda")
    if case["start"] == "guess":  # the last step's potential: every blob a little elsewhere
        before = _source(n, h, rule, case["blobs"], seed, shift=0.25 * h)
        state["guess"] = _solution(before, h, rule, case["fixed_value"])[0]
    if case["memory"] == "host":
        state["rho"] = rho.cpu().pin_memory()
        state["phi"] = torch.zeros_like(state["rho"]).pin_memory()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        _, _, statuses = state["batch"].solve(state["rhos"], state["phis"], 1.0, case["tol"])
        return {"phi": state["flat"], "status": statuses}
    if case["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(rho, phi, bc=KINDS[rule], tol=tol, lmax=lmax)
                   for (n, rule, lmax, tol, _), rho, phi in zip(state["reqs"], state["rhos"],
                                                                state["phis"])]
        statuses = [int(server.wait(t)[0].status) for t in tickets]
        return {"phi": state["phis"], "status": np.array(statuses)}
    solver, rho, phi = state["solver"], state["rho"], state["phi"]
    if "guess" in state:
        phi.copy_(state["guess"])
    if case["gravity"]:
        _, g, _, status = solver.solve_gravity(rho, 1.0, case["tol"], phi=phi, g=state["g"])
        return {"phi": phi, "g": g, "status": status}
    if case["memory"] == "host":
        _, _, status = solver.solve_host(rho, 1.0, case["tol"], phi=phi)
    else:
        _, _, status = solver.solve(rho, 1.0, case["tol"], phi=phi)
    return {"phi": phi, "status": status}


def _solve_work(cells, tol, gravity=False, guess=False):
    # rho in, phi out (the acceleration out, the guess in); a factor of ten per
    # V-cycle, each cycle's two SMOOTHs, defect, restriction and prolongation
    # on all levels
    cycles = max(1.0, -math.log10(tol))
    return np.array([cells * (16 + 24 * gravity + 8 * guess), cells * 8 / 7 * 33 * cycles])


def work(case):
    if case["kind"] == "batch":
        w = sum(_solve_work(n ** 3, case["tol"]) for n, _, _ in _batch_grids(case))
    elif case["kind"] == "serve":
        w = sum(_solve_work(n ** 3, tol) for n, _, _, tol, _ in _requests(case))
    else:
        w = _solve_work(case["nx"] * case["ny"] * case["nz"], case["tol"], case["gravity"],
                        case["start"] == "guess")
    return {"bytes": float(w[0]), "flops": float(w[1])}


# --- the discrete problem's own solution ----------------------------------

def _axis(n, h, lo, hi):
    """Eigenvalues and orthonormal eigenvectors (columns) of the second
    difference along one axis with the ghost rules lo and hi (homogeneous)."""
    i = np.arange(n)[:, None] + 0.5
    k = np.arange(n)[None, :]
    if lo == "P":
        m = (k + 1) // 2
        q = np.where(k % 2 == 0, np.cos(2 * np.pi * m * i / n), np.sin(2 * np.pi * m * i / n))
        t = 2 * np.pi * m / n
    else:
        lo, hi = (x.replace("O", "F") for x in (lo, hi))
        m = k + (1.0 if lo + hi == "FF" else 0.0 if lo + hi == "ZZ" else 0.5)
        t = np.pi * m / n
        q = np.sin(t * i) if lo == "F" else np.cos(t * i)
    q = q / np.sqrt((q * q).sum(0, keepdims=True))
    lam = -4.0 / (h * h) * np.sin(0.5 * t[0]) ** 2
    return torch.from_numpy(lam).cuda(), torch.from_numpy(np.ascontiguousarray(q)).cuda()


def _open_values(rho, h, lmax):
    """Potential of the expansion to order lmax about the centre of mass on the
    six faces (x-, x+, y-, y+, z-, z+), 4 pi G = 1, by Cartesian moments."""
    nz, ny, nx = rho.shape
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * m) * h
          for m in (nx, ny, nz)]
    mass = rho.sum()
    com = [(rho.sum(tuple(d for d in range(3) if d != 2 - a)) * ax[a]).sum() / mass
           for a in range(3)]
    powers = [torch.stack([(ax[a] - com[a]) ** p for p in range(5)]) for a in range(3)]
    raw = torch.einsum("zyx,ax->zya", rho, powers[0])
    raw = torch.einsum("zya,by->zab", raw, powers[1])
    raw = (torch.einsum("zab,cz->abc", raw, powers[2]) * h ** 3).cpu()

    def moment(idx):
        return float(raw[idx.count(0), idx.count(1), idx.count(2)])

    m1 = [moment([i]) for i in range(3)]
    m2 = torch.tensor([[moment([i, j]) for j in range(3)] for i in range(3)], dtype=torch.float64)
    m3 = torch.tensor([[[moment([i, j, k]) for k in range(3)] for j in range(3)]
                       for i in range(3)], dtype=torch.float64)
    m4 = torch.tensor([[[[moment([i, j, k, l]) for l in range(3)] for k in range(3)]
                        for j in range(3)] for i in range(3)], dtype=torch.float64)
    m1, m2, m3, m4 = (torch.as_tensor(m, dtype=torch.float64).cuda() for m in (m1, m2, m3, m4))
    out = []
    for q in range(6):
        a = q // 2
        pts = list(ax)
        pts[a] = torch.tensor([(1 if q % 2 else -1) * 0.5 * rho.shape[2 - a] * h],
                              dtype=torch.float64, device="cuda")
        z, y, x = torch.meshgrid(pts[2] - com[2], pts[1] - com[1], pts[0] - com[0], indexing="ij")
        v = torch.stack([x, y, z], -1)
        r2 = (v * v).sum(-1)
        e = lambda s, *t: torch.einsum(s, *t)  # noqa: E731
        terms = [
            mass * h ** 3 * torch.ones_like(r2),
            v @ m1,
            1.5 * e("...i,...j,ij->...", v, v, m2) - 0.5 * r2 * m2.trace(),
            2.5 * e("...i,...j,...k,ijk->...", v, v, v, m3) - 1.5 * r2 * (v @ e("ijj->i", m3)),
            (35 * e("...i,...j,...k,...l,ijkl->...", v, v, v, v, m4)
             - 30 * r2 * e("...i,...j,ijkk->...", v, v, m4) + 3 * r2 * r2 * e("iijj->", m4)) / 8,
        ]
        phi = sum(t / r2 ** (l + 0.5) for l, t in enumerate(terms[:lmax + 1]))
        out.append(-phi / (4 * math.pi))
    return out


def _solution(rho, h, rule, fixed_value=0.0, lmax=4, gravity=False):
    """(phi, g or None) of the discrete equations with 4 pi G = 1."""
    faces = _faces(rule)
    f = rho.clone()
    values = [fixed_value if r == "F" else 0.0 for r in faces]
    if rule == "O":
        values = _open_values(rho, h, lmax)
    if _mean_free(rule):
        f -= f.mean()

    def edge(t, q):  # the cells next to face q
        d = 2 - q // 2
        return t.narrow(d, t.shape[d] - 1 if q % 2 else 0, 1)

    for q in range(6):
        if faces[q] in "FO":
            edge(f, q).sub_(2.0 * values[q] / (h * h))
    (lx, qx), (ly, qy), (lz, qz) = (
        _axis(rho.shape[2 - a], h, faces[2 * a], faces[2 * a + 1]) for a in range(3))
    t = torch.einsum("zyx,xa->zya", f, qx)
    t = torch.einsum("zya,yb->zba", t, qy)
    t = torch.einsum("zba,zc->cba", t, qz)
    lam = lz[:, None, None] + ly[None, :, None] + lx[None, None, :]
    if _mean_free(rule):
        lam[0, 0, 0] = 1.0
        t[0, 0, 0] = 0.0
    t /= lam
    t = torch.einsum("cba,zc->zba", t, qz)
    t = torch.einsum("zba,yb->zya", t, qy)
    phi = torch.einsum("zya,xa->zyx", t, qx).contiguous()
    if not gravity:
        return phi, None
    g = []
    for a in range(3):
        d = 2 - a
        ghost = []
        for q in (2 * a, 2 * a + 1):
            if faces[q] == "P":
                ghost.append(edge(phi, q ^ 1))
            else:
                ghost.append(edge(phi, q) if faces[q] == "Z" else 2.0 * values[q] - edge(phi, q))
        p = torch.cat([ghost[0], phi, ghost[1]], d)
        m = phi.shape[d]
        g.append((p.narrow(d, 0, m) - p.narrow(d, 2, m)) / (2 * h))
    return phi, torch.stack(g)


def exact(case, seed):
    if case["kind"] == "batch":
        grids = _batch_grids(case)
        phi = [_solution(_source((n, n, n), 1.0 / n, rule, b, seed * 1009 + k), 1.0 / n, rule)[0]
               for k, (n, rule, b) in enumerate(grids)]
        return {"phi": torch.cat([p.reshape(-1) for p in phi]), "status": None}
    if case["kind"] == "serve":
        phi = [_solution(_source((n, n, n), 1.0 / n, rule, b, seed * 1013 + k), 1.0 / n, rule,
                         lmax=lmax)[0]
               for k, (n, rule, lmax, _, b) in enumerate(_requests(case))]
        return {"phi": phi, "status": None}
    n, h = _box(case)
    rho = _source(n, h, case["rule"], case["blobs"], seed)
    phi, g = _solution(rho, h, case["rule"], case["fixed_value"], gravity=case["gravity"])
    out = {"phi": phi, "status": None}
    if g is not None:
        out["g"] = g
    return out
