"""The coarse levels in one launch (mg_coarse.cu) against the oracle: levels cut
into slabs over a cluster (along z, or along y where z is short), levels whole
in one CTA, the level whose cycle is a matrix, coarsest levels of one and of
several cells, each kind of face, and every count of smoothing steps.

FP64: the same schedule as the oracle's differs in rounding order only, e_max
<= 1e-11 as in the other same-schedule tests.  Mixed: the residual of the
returned phi, by the oracle's own defect operator, is below the tolerance the
solve was given (1e-10, plus 1e-3 of it for the two sides' rounding).
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
    "faces": ((Z, F, P, P, F, Z), (0, 0.3, 0, 0, -0.2, 0)),
}


def source(dims, seed):
    nx, ny, nz = dims
    rho = np.random.default_rng(seed).standard_normal((nz, ny, nx))
    return rho - rho.mean()


def solve_both(dims, rule, tol, *, max_cycles, stall, prec, **kw):
    kinds, values = RULES[rule]
    rho = source(dims, sum(dims) + len(rule))
    h = 1.0 / dims[0]
    bc = kinds[0] if len(set(kinds)) == 1 else orc.PER_FACE
    faces = orc.mixed_rule(kinds, values) if bc == orc.PER_FACE else None
    okw = {k: kw[k] for k in ("pre", "post", "coarse_literal") if k in kw}
    ref = orc.solve(rho, h, bc, bc_value=values[0], faces=faces,
                    tol=tol, stall_ratio=stall, max_cycles=max_cycles, **okw)
    with mg.Solver(dims, h, list(kinds), face_values=list(values), prec=prec, stall_ratio=stall,
                   max_cycles=max_cycles, **kw) as s:
        phi, hist, st = s.solve(torch.from_numpy(rho).cuda(), 1.0, tol)
    err = float(np.abs(phi.cpu().numpy() - ref.phi).max() / np.abs(ref.phi).max())
    return err, hist, ref.hist, st


@pytest.mark.parametrize("rule", sorted(RULES))
@pytest.mark.parametrize("dims", [(2, 2, 2), (4, 4, 4), (16, 16, 16), (16, 4, 2), (32, 16, 16),
                                  (32, 32, 8), (32, 8, 32), (64, 16, 8), (128, 8, 8),
                                  (64, 64, 32)])
def test_fp64_same_schedule(dims, rule):
    err, hist, ref, _ = solve_both(dims, rule, 0.0, max_cycles=2, stall=NO_STALL, prec=mg.FP64)
    assert err <= 1e-11, err
    assert np.allclose(hist, ref, rtol=1e-6, atol=1e-14)


@pytest.mark.parametrize("steps", [(0, 1), (1, 0), (2, 2), (0, 2)])
@pytest.mark.parametrize("dims", [(16, 16, 16), (32, 32, 8)])
def test_fp64_smoothing_counts(dims, steps):
    for rule in ("fixed", "faces"):
        err, _, _, _ = solve_both(dims, rule, 0.0, max_cycles=2, stall=NO_STALL, prec=mg.FP64,
                                  pre=steps[0], post=steps[1])
        assert err <= 1e-11, (rule, err)


def test_fp64_literal_coarse_rule():
    """The level a cycle starts on and the levels below have different rules."""
    for dims in ((16, 16, 16), (32, 32, 32)):
        err, _, _, _ = solve_both(dims, "zerograd", 0.0, max_cycles=3, stall=NO_STALL,
                                  prec=mg.FP64, coarse_literal=1)
        assert err <= 1e-11, (dims, err)


@pytest.mark.parametrize("rule", sorted(RULES))
@pytest.mark.parametrize("dims", [(4, 4, 4), (16, 16, 16), (64, 64, 16), (64, 16, 64), (128, 32, 32)])
def test_mixed_residual(dims, rule):
    kinds, values = RULES[rule]
    rho, h = source(dims, sum(dims)), 1.0 / dims[0]
    with mg.Solver(dims, h, list(kinds), face_values=list(values), prec=mg.MIXED) as s:
        phi, hist, st = s.solve(torch.from_numpy(rho).cuda(), 1.0, 1e-10)
    assert st == 0 and hist[-1] < 1e-10, (st, hist)
    bc = kinds[0] if len(set(kinds)) == 1 else orc.PER_FACE
    f = rho if F in kinds else rho - rho.mean()
    d = orc.defect(phi.cpu().numpy(), f, h, bc, bc_value=values[0],
                   faces=orc.mixed_rule(kinds, values) if bc == orc.PER_FACE else None)
    r = float(np.sqrt((d * d).mean() / (f * f).mean()))
    assert r < 1.001e-10, r
