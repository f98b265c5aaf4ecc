"""The staged batched solve (a launch per phase and class of like grids) against
the persistent kernel, which runs the same programs: the same bits, histories
and statuses."""
import numpy as np
import pytest
import torch

import paper_2302_13903_gb300 as mg
from paper_2302_13903_gb300 import inputs

pytestmark = pytest.mark.gpu

RULES = (mg.PERIODIC, mg.FIXED, mg.ZEROGRAD)


def solve(b, rhos, tol):
    phis = [None if r is None else torch.full_like(r, 7.0) for r in rhos]
    st, hists, sts = b.solve(rhos, phis, 1.0, tol)
    return phis, st, hists, list(sts)


@pytest.mark.parametrize("sizes,spread", [
    ((2, 4, 8, 16), 1), ((16, 32), 1), ((32, 64, 128), 1), ((128,), 1), ((256, 2), 1),
    ((8, 16, 32), 9),  # more classes than streams: the persistent kernel by itself
])
@pytest.mark.parametrize("tol", [1e-10, 1e-3])
def test_staged_solve_gives_the_persistent_kernels_bits(sizes, spread, tol):
    """Every rule at every size, two grids of the first class, one slot empty, a
    grid with rho = 0; `spread` spacings."""
    specs = [(n, bc, (1.0 + q) / n) for n in sizes for bc in RULES for q in range(spread)]
    specs.append(specs[0])
    rhos, fixed = [], []
    for k, (n, bc, _) in enumerate(specs):
        rho = inputs.batch_source(dict(n=n, bc=bc, seed=40 + k, n_blobs=3))
        rhos.append(torch.from_numpy(rho).cuda())
        fixed.append(0.3 if bc == mg.FIXED and k % 2 else 0.0)
    rhos[1] = None
    rhos[2] = torch.zeros_like(rhos[2])
    with mg.Batch([n for n, _, _ in specs], [h for _, _, h in specs], [bc for _, bc, _ in specs],
                  fixed) as b:
        first = solve(b, rhos, tol)
        again = solve(b, rhos, tol)  # its graphs replayed
        b.set_blocks(7)
        ref = solve(b, rhos, tol)
    for got in (first, again):
        assert got[1] == ref[1] and got[3] == ref[3]
        for p, q, h, k in zip(got[0], ref[0], got[2], ref[2]):
            assert (p is None and q is None) or torch.equal(p, q)
            assert np.array_equal(h, k)


def test_max_cycles_ends_every_class():
    specs = [(16, mg.PERIODIC), (64, mg.FIXED), (32, mg.ZEROGRAD)]
    rhos = [torch.from_numpy(inputs.batch_source(dict(n=n, bc=bc, seed=n, n_blobs=3))).cuda()
            for n, bc in specs]
    for m in (1, 2):
        with mg.Batch([n for n, _ in specs], [1.0 / n for n, _ in specs], [bc for _, bc in specs],
                      max_cycles=m) as b:
            got = solve(b, rhos, 1e-13)
            b.set_blocks(7)
            ref = solve(b, rhos, 1e-13)
        assert got[3] == ref[3] and all(len(h) == m for h in got[2])
        for p, q in zip(got[0], ref[0]):
            assert torch.equal(p, q)


def test_phi_in_another_grids_source():
    """Every rho is read before any phi is written, also where they share memory
    across sizes: the results are those of separate arrays."""
    specs = [(64, mg.PERIODIC), (16, mg.FIXED), (32, mg.ZEROGRAD)]
    rhos = [torch.from_numpy(inputs.batch_source(dict(n=n, bc=bc, seed=n, n_blobs=3))).cuda()
            for n, bc in specs]
    with mg.Batch([n for n, _ in specs], [1.0 / n for n, _ in specs],
                  [bc for _, bc in specs]) as b:
        ref, st, hists, sts = solve(b, rhos, 1e-10)
        # the small grids' phi in the large grid's rho, the large one's over both
        # small sources
        big = rhos[0].clone().view(-1)
        both = torch.zeros(64 ** 3, dtype=torch.float64, device="cuda")
        both[:16 ** 3] = rhos[1].view(-1)
        both[16 ** 3:16 ** 3 + 32 ** 3] = rhos[2].view(-1)
        src = [big.view(64, 64, 64), both[:16 ** 3].view(16, 16, 16),
               both[16 ** 3:16 ** 3 + 32 ** 3].view(32, 32, 32)]
        out = [both.view(64, 64, 64), big[:16 ** 3].view(16, 16, 16),
               big[16 ** 3:16 ** 3 + 32 ** 3].view(32, 32, 32)]
        # (the large grid's phi is written over the small ones' sources, theirs
        # over its source)
        got = b.solve(src, out, 1.0, 1e-10)
        assert got[0] == st and list(got[2]) == sts
        for p, q, h, k in zip(out, ref, got[1], hists):
            assert torch.equal(p, q) and np.array_equal(h, k)


BLOCKING = r"""
import ctypes, sys, time
sys.path.insert(0, sys.argv[1])
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0  # CU_CTX_SCHED_BLOCKING_SYNC, of this process
import torch
import paper_2302_13903_gb300 as mg
from paper_2302_13903_gb300 import inputs
specs = [(256, mg.PERIODIC), (256, mg.FIXED), (128, mg.FIXED)][:int(sys.argv[2])]
rhos = [torch.from_numpy(inputs.batch_source(dict(n=n, bc=bc, seed=n, n_blobs=3))).cuda()
        for n, bc in specs]
phis = [torch.zeros_like(r) for r in rhos]
with mg.Batch([n for n, _ in specs], [1.0 / n for n, _ in specs], [bc for _, bc in specs]) as b:
    for _ in range(3):
        b.solve(rhos, phis, 1.0, 1e-10)
    torch.cuda.synchronize()
    wall, cpu = time.perf_counter(), time.thread_time()
    for _ in range(10):
        b.solve(rhos, phis, 1.0, 1e-10)
    wall, cpu = time.perf_counter() - wall, time.thread_time() - cpu
print(cpu / wall)
"""


@pytest.mark.parametrize("classes", [1, 3])
def test_a_blocking_process_blocks(classes):
    """Where the process asked for waits that block, the calling thread is idle for
    most of a solve of large grids (its launches take some tenths of it)."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", BLOCKING, root, str(classes)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert float(r.stdout) < 0.6, r.stdout


def test_phase_times_after_set_blocks_and_back():
    """The shares of a staged solve, the barrier times of a persistent one, and the
    former again: no negative time, and no more in all than the call took."""
    import time
    rhos = [torch.from_numpy(inputs.batch_source(dict(n=n, bc=bc, seed=n, n_blobs=3))).cuda()
            for n, bc in ((64, mg.PERIODIC), (32, mg.FIXED))]
    with mg.Batch([64, 32], [1 / 64, 1 / 32], [mg.PERIODIC, mg.FIXED]) as b:
        for blocks in (0, 7, 0):
            b.set_blocks(blocks)
            for _ in range(2):
                t = time.perf_counter()
                solve(b, rhos, 1e-10)
                wall = 1e3 * (time.perf_counter() - t)
                ms = b.phase_ms()
                ms = list(ms.values()) if isinstance(ms, dict) else list(ms)
                assert min(ms) >= 0.0 and 0.0 < sum(ms) <= wall
