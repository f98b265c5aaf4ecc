"""The FP64 path's finest level in 64-bit fixed point (mg_fx64.cu) and the FP64
level kernels, against the oracle.

Whole solves with the same schedule differ from the oracle's in rounding order
only: e_max <= 1e-11 as in the other same-schedule tests.  The shapes cover one
tile and several, a z-chunk shorter than its halo's reach, ragged last chunks
and tiles whose window wraps twice.  A source scaled by a power of two gives
the same integers, so the same bits scaled.
"""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_2302_13903_gb300 as mg

pytestmark = pytest.mark.gpu

NO_STALL = 1e300
P, F, Z = mg.PERIODIC, mg.FIXED, mg.ZEROGRAD
RULES = {
    "periodic": ((P,) * 6, (0,) * 6),
    "fixed": ((F,) * 6, (0.4,) * 6),
    "zerograd": ((Z,) * 6, (0,) * 6),
    "x_walls": ((Z, F, P, P, P, P), (0, 0.3, 0, 0, 0, 0)),
    "yz_walls": ((P, P, F, Z, Z, F), (0, 0, -0.5, 0, 0, 0.2)),
}


def source(dims, seed):
    nx, ny, nz = dims
    rho = np.random.default_rng(seed).standard_normal((nz, ny, nx))
    return rho - rho.mean()


def oracle_args(rule):
    kinds, values = RULES[rule]
    bc = kinds[0] if len(set(kinds)) == 1 else orc.PER_FACE
    return bc, dict(bc_value=values[0],
                    faces=orc.mixed_rule(kinds, values) if bc == orc.PER_FACE else None)


def gpu(rho, rule, tol=0.0, phi=None, **kw):
    kinds, values = RULES[rule]
    nz, ny, nx = rho.shape
    with mg.Solver((nx, ny, nz), 1.0 / nx, list(kinds), face_values=list(values), prec=mg.FP64,
                   **kw) as s:
        p, hist, st = s.solve(torch.from_numpy(rho).cuda(), 1.0, tol, phi=phi, raise_on_error=False)
    return p.cpu().numpy(), hist, st


@pytest.mark.parametrize("rule", sorted(RULES))
@pytest.mark.parametrize("dims", [(64, 16, 16), (64, 64, 64), (128, 32, 16), (128, 128, 64),
                                  (256, 64, 64)])
def test_same_schedule(dims, rule):
    rho = source(dims, sum(dims))
    bc, kw = oracle_args(rule)
    for k in (0, 2):
        ref = orc.solve(rho, 1.0 / dims[0], bc, tol=0.0, max_cycles=k, stall_ratio=NO_STALL, **kw)
        phi, hist, st = gpu(rho, rule, max_cycles=k, stall_ratio=NO_STALL)
        assert st == ref.status and len(hist) == len(ref.hist)
        assert np.abs(phi - ref.phi).max() <= 1e-11 * np.abs(ref.phi).max()
        assert np.allclose(hist, ref.hist, rtol=1e-6, atol=1e-14)


def test_power_of_two_scaling_is_exact_and_misaligned_phi_agrees():
    rho = source((64, 32, 32), 3)
    base, h0, _ = gpu(rho, "periodic", max_cycles=2, stall_ratio=NO_STALL)
    for e in (-300, 300):
        p, h, _ = gpu(rho * 2.0 ** e, "periodic", max_cycles=2, stall_ratio=NO_STALL)
        assert np.array_equal(p, base * 2.0 ** e) and np.array_equal(h, h0)
    # 8-byte aligned phi: the general FP64 kernels
    odd = torch.zeros(rho.size + 1, dtype=torch.float64, device="cuda")[1:].view(rho.shape)
    p, _, _ = gpu(rho, "periodic", phi=odd, max_cycles=2, stall_ratio=NO_STALL)
    assert np.abs(p - base).max() <= 1e-12 * np.abs(base).max()


def test_sources_outside_the_fixed_point_range():
    rho = source((64, 64, 64), 5)
    zero, hist, st = gpu(np.zeros_like(rho), "fixed", tol=1e-10)
    ref = orc.solve(np.zeros_like(rho), 1.0 / 64, F, bc_value=0.4, tol=1e-10)
    assert st == ref.status and np.abs(zero - ref.phi).max() <= 1e-11 * 0.4
    phi, hist, st = gpu(np.zeros_like(rho), "periodic", tol=1e-10)
    assert st == 0 and not phi.any()
    bad = rho.copy()
    bad[3, 4, 5] = np.nan
    assert gpu(bad, "periodic", tol=1e-10)[2] == 5  # MG_ERR_DIVERGED
    # relaxation far past the stable range: the oracle's status
    ref = orc.solve(rho, 1.0 / 64, F, bc_value=0.4, tol=1e-10, omega=1.99)
    assert gpu(rho, "fixed", tol=1e-10, omega=1.99)[2] == ref.status


def test_in_place_is_the_general_path():
    """rho and phi the same array: the general FP64 kernels, as for a misaligned phi."""
    rho = source((64, 32, 32), 4)
    odd = torch.zeros(rho.size + 1, dtype=torch.float64, device="cuda")[1:].view(rho.shape)
    ref, h0, _ = gpu(rho, "fixed", phi=odd, max_cycles=2, stall_ratio=NO_STALL)
    both = torch.from_numpy(rho).cuda()
    with mg.Solver((64, 32, 32), 1.0 / 64, [F] * 6, face_values=[0.4] * 6, prec=mg.FP64,
                   max_cycles=2, stall_ratio=NO_STALL) as s:
        p, h, _ = s.solve(both, 1.0, 0.0, phi=both, raise_on_error=False)
    assert np.array_equal(p.cpu().numpy(), ref) and np.array_equal(h, h0)


@pytest.mark.parametrize("rule", sorted(RULES))
@pytest.mark.parametrize("dims", [(2, 2, 2), (6, 4, 2), (10, 6, 4), (64, 6, 10), (34, 2, 64)])
@pytest.mark.parametrize("prec", [mg.FP64, mg.MIXED])
def test_level_kernels_on_even_sizes(dims, rule, prec):
    """SMOOTH, defect + restriction and prolongation on sizes that are even but
    no powers of two; FP64 to 1e-13 of the largest output, FP32 to 2e-6, as the
    operator tests on cubes."""
    if len(set(RULES[rule][0])) > 1:
        pytest.skip("the operators take one rule for all faces")
    bc, kw = oracle_args(rule)
    nx, ny, nz = dims
    rng = np.random.default_rng(nx + ny + nz)
    dt, tol = (np.float64, 1e-13) if prec == mg.FP64 else (np.float32, 2e-6)
    u, f = (rng.standard_normal((nz, ny, nx)).astype(dt) for _ in range(2))
    h = 0.125
    gu, gf = (torch.from_numpy(a).cuda() for a in (u, f))
    value = dict(bc_value=kw["bc_value"])

    def close(got, ref):
        assert np.abs(got.cpu().numpy() - ref).max() <= tol * max(1.0, np.abs(ref).max())

    ud, fd = u.astype(np.float64), f.astype(np.float64)
    close(mg.op_smooth(gu.clone(), gf, h, bc, **value),
          orc.smooth(ud.copy(), fd, h, bc, **value))
    d = orc.defect(ud, fd, h, bc, **value)
    close(mg.op_defect_restrict(gu, gf, h, bc, **value), orc.restrict(d))
    c = rng.standard_normal((nz, ny, nx)).astype(dt)
    gc = torch.from_numpy(c).cuda()
    fine = rng.standard_normal((2 * nz, 2 * ny, 2 * nx)).astype(dt)
    got = mg.op_prolong(gc, bc, bc_value=0.0, add=True, uf=torch.from_numpy(fine).cuda())
    ref = orc.prolong(c.astype(np.float64), bc, bc_value=0.0, add=True, uf=fine.astype(np.float64))
    close(got, ref)


def test_autotune_after_a_solve():
    """mg_ctx_autotune has nothing to time on an FP64 context, before a solve or
    after one."""
    rho = torch.from_numpy(source((128, 32, 16), 6)).cuda()  # a shape no other test tunes
    with mg.Solver((128, 32, 16), 1.0 / 128, mg.PERIODIC, prec=mg.FP64) as s:
        first = s.solve(rho, 1.0, 1e-9)
        s.autotune()
        again = s.solve(rho, 1.0, 1e-9)
    assert torch.equal(first[0], again[0]) and np.array_equal(first[1], again[1])


@pytest.mark.parametrize("rule", ["periodic", "fixed"])
def test_a_solve_that_diverges_is_the_general_path(rule):
    """Where the relaxation diverges the integers' ranges end first: status,
    history and phi are those of the FP64 kernels (as for a misaligned phi)."""
    rho = source((64, 64, 64), 7)
    odd = torch.zeros(rho.size + 1, dtype=torch.float64, device="cuda")[1:].view(rho.shape)
    ref, h0, st0 = gpu(rho, rule, tol=1e-10, phi=odd, omega=1.999, stall_ratio=NO_STALL)
    phi, hist, st = gpu(rho, rule, tol=1e-10, omega=1.999, stall_ratio=NO_STALL)
    assert st == st0
    if st == 5:  # MG_ERR_DIVERGED
        assert np.array_equal(hist, h0) and np.array_equal(phi, ref)


def test_solve_buffers_are_counted_and_can_be_declined():
    """The first solve adds mg_solve_bytes to the context, or with the buffers
    declined nothing, and runs on the FP64 kernels (as for a misaligned phi)."""
    rho = source((64, 64, 64), 8)
    odd = torch.zeros(rho.size + 1, dtype=torch.float64, device="cuda")[1:].view(rho.shape)
    plain = gpu(rho, "periodic", tol=1e-9, phi=odd)[0]
    dev = torch.from_numpy(rho).cuda()
    with mg.Solver(64, 1.0 / 64, P, prec=mg.FP64) as s:
        need, extra = mg.required_bytes(64, P, prec=mg.FP64), mg.solve_bytes(64, prec=mg.FP64)
        assert s.device_bytes == need
        first = s.solve(dev, 1.0, 1e-9)[0]
        assert s.device_bytes == need + extra and s.fixed_point
        s.set_solve_buffers(False)
        assert s.device_bytes == need
        for _ in range(3):  # launch by launch, captured, replayed
            assert np.array_equal(s.solve(dev, 1.0, 1e-9)[0].cpu().numpy(), plain)
            assert s.device_bytes == need and not s.fixed_point
        s.set_solve_buffers(True)
        for _ in range(3):
            assert torch.equal(s.solve(dev, 1.0, 1e-9)[0], first)
            assert s.device_bytes == need + extra and s.fixed_point


def test_server_counts_the_solve_buffers_or_does_without():
    """A budget that holds them: a solve's own bits; one that holds the hierarchy
    alone: accepted, with the FP64 kernels' bits."""
    rho = source((64, 64, 64), 9)
    odd = torch.zeros(rho.size + 1, dtype=torch.float64, device="cuda")[1:].view(rho.shape)
    plain, fixed = gpu(rho, "periodic", tol=1e-9, phi=odd)[0], gpu(rho, "periodic", tol=1e-9)[0]
    need = mg.required_bytes(64, P, prec=mg.FP64)
    for budget, want in ((need + mg.solve_bytes(64, prec=mg.FP64), fixed), (need, plain)):
        with mg.Server(budget, slots=1, prec=mg.FP64) as s:
            phi = torch.zeros(rho.shape, dtype=torch.float64, device="cuda")
            for _ in range(2):
                t = s.submit(torch.from_numpy(rho).cuda(), phi, bc=P, tol=1e-9)
                assert s.wait(t, 60)[0].status == 0
                assert np.array_equal(phi.cpu().numpy(), want)
            assert s.stats()["peak_bytes"] == budget


# --- the rounding floor: errors against the discrete solution in double-double ---

def two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def dd(*parts):
    """Sum of (high, low) pairs."""
    hi, lo = parts[0]
    for h, l in parts[1:]:
        hi, e = two_sum(hi, h)
        hi, lo = two_sum(hi, lo + e + l)
    return hi, lo


def neighbours(t, kind):
    """The six neighbours of every cell under one homogeneous rule."""
    for d in range(3):
        for end in (0, t.shape[d] - 1):
            r = torch.roll(t, 1 if end == 0 else -1, d)
            if kind != P:
                own = t.narrow(d, end, 1)
                r.narrow(d, end, 1).copy_(own if kind == Z else -own)
            yield r


def modes(m, kind, h):
    """Eigenvalues and orthonormal eigenvectors of the second difference."""
    a = -2.0 * np.eye(m) + np.eye(m, k=1) + np.eye(m, k=-1)
    if kind == P:
        a[0, -1] += 1
        a[-1, 0] += 1
    else:
        a[0, 0] += 1 if kind == Z else -1
        a[-1, -1] += 1 if kind == Z else -1
    w, v = np.linalg.eigh(a)
    return torch.from_numpy(w / h ** 2).cuda(), torch.from_numpy(v).cuda()


def discrete_solution(rho, kind, h):
    """(high, low) of phi with L phi = rho, by refinement on exact residuals."""
    free = kind != F
    axes = [modes(m, kind, h) for m in rho.shape]
    lam = axes[0][0][:, None, None] + axes[1][0][:, None] + axes[2][0]
    null = lam.abs() < 1e-6 * lam.abs().max() if free else torch.zeros_like(lam, dtype=torch.bool)
    lam = torch.where(null, 1.0, lam)

    def minus_mean(x):
        if not free:
            return x
        m = sum(np.sum(v.cpu().numpy().astype(np.longdouble)) for v in x) / x[0].numel()
        hi = float(m)
        return dd(x, (torch.full_like(x[0], -hi), torch.full_like(x[0], -float(m - hi))))

    zero = torch.zeros_like(rho)
    f, phi = minus_mean((rho, zero)), (zero, zero)
    for _ in range(4):
        lap = dd((-4 * phi[0], -4 * phi[1]), (-2 * phi[0], -2 * phi[1]),
                 *zip(neighbours(phi[0], kind), neighbours(phi[1], kind)))
        r = sum(dd(f, (-lap[0] / h ** 2, -lap[1] / h ** 2)))  # h is a power of two
        t = torch.einsum("zyx,za,yb,xc->abc", r, *(v for _, v in axes))
        t = torch.where(null, 0.0, t / lam)
        phi = dd(phi, (torch.einsum("abc,za,yb,xc->zyx", t, *(v for _, v in axes)), zero))
    return minus_mean(phi)


def blobs(n, count, kind):
    """Gaussian blobs of width 0.02 to 0.08 of the side (tails wrapped if periodic)."""
    rng = np.random.default_rng(count)
    x = (np.arange(n) + 0.5) / n
    rho = np.zeros((n, n, n))
    for _ in range(count):
        s, amp, c = rng.uniform(0.02, 0.08), rng.lognormal(), rng.random(3)
        d = [x - v for v in c]
        if kind == P:
            d = [v - np.round(v) for v in d]
        g = [np.exp(-0.5 * (v / s) ** 2) for v in d]
        rho += amp * g[2][:, None, None] * g[1][:, None] * g[0]
    return torch.from_numpy(rho - (rho.mean() if kind != F else 0.0)).cuda()


FLOOR_SIZES = [64, 128]


@pytest.mark.parametrize("count", [4, 64])
@pytest.mark.parametrize("kind", [P, F, Z])
@pytest.mark.parametrize("n", FLOOR_SIZES)
def test_rounding_floor_is_that_of_doubles(n, kind, count):
    """Iterated until it stalls, the solve on the integer grid is as near the
    discrete solution as the FP64 kernels (an 8-byte aligned phi takes those),
    to one bit, by the largest and by the mean error of phi and of g."""
    rho = blobs(n, count, kind)
    hi, lo = discrete_solution(rho, kind, 1.0 / n)
    err = []
    for off in (0, 1):
        phi = torch.zeros(n ** 3 + 1, dtype=torch.float64, device="cuda")
        phi = phi[off:off + n ** 3].view(rho.shape)
        with mg.Solver(n, 1.0 / n, kind, prec=mg.FP64) as s:
            phi, g, _, st = s.solve_gravity(rho, 1.0, 0.0, phi=phi)
        assert st == 0
        e = (phi - hi) - lo
        nb = list(zip(neighbours(hi, kind), neighbours(lo, kind)))
        eg = []
        for a in range(3):
            low, high = nb[4 - 2 * a], nb[5 - 2 * a]
            eg.append(g[a] - sum(dd(low, (-high[0], -high[1]))) * (0.5 * n))
        eg = torch.stack(eg)
        err.append([e.abs().max(), e.norm(), eg.abs().max(), eg.norm()])
    for a, b in zip(*err):
        assert float(a) <= 2.0 * float(b), [[float(x) for x in row] for row in err]
