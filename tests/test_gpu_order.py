"""Solves come after the work that is pending on the stream they are given: the
legacy default stream (with the blocking streams that it waits for), a context's
set-up, another stream."""
import ctypes
import glob
import os

import pytest
import torch

import paper_2302_13903_gb300 as mg
from paper_2302_13903_gb300 import inputs

pytestmark = pytest.mark.gpu

PAUSE = 100_000_000  # GPU clocks, some 50 ms: far longer than a solve of 32^3 takes to start


def source(n=32, seed=3):
    return torch.from_numpy(inputs.batch_source(dict(n=n, bc=mg.FIXED, seed=seed, n_blobs=3))).cuda()


def blocking_stream():
    """A stream that the legacy default stream waits for (torch's own are not)."""
    names = glob.glob(os.path.join(os.path.dirname(torch.__file__), "..", "nvidia", "**",
                                   "libcudart.so*"), recursive=True)
    for name in names + ["libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"]:
        try:
            rt = ctypes.CDLL(name)
            break
        except OSError:
            continue
    else:
        pytest.skip("no libcudart to load")
    p = ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(p)) == 0
    return torch.cuda.ExternalStream(p.value)


@pytest.mark.parametrize("prec", [mg.FP64, mg.MIXED])
@pytest.mark.parametrize("pending", ["default", "blocking"])
def test_default_stream_solve_follows_pending_work(pending, prec):
    rho, rho2 = source(seed=3), source(seed=4)
    stream = torch.cuda.default_stream() if pending == "default" else blocking_stream()
    with mg.Solver(32, 1.0 / 32, mg.FIXED, prec=prec) as s:
        want = s.solve(rho2, 1.0, 1e-9)[0]
        for _ in range(3):  # launch by launch, captured, replayed
            buf, phi = rho.clone(), torch.zeros_like(rho)
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                torch.cuda._sleep(PAUSE)
                buf.copy_(rho2)
            s.solve(buf, 1.0, 1e-9, phi=phi, stream=torch.cuda.default_stream())
            assert torch.equal(phi, want)


@pytest.mark.parametrize("prec", [mg.FP64, mg.MIXED])
def test_a_solve_on_another_stream_follows_the_contexts_set_up(prec):
    """mg_create forms the coarse matrix on the default stream and does not wait."""
    rho = source()
    with mg.Solver(32, 1.0 / 32, mg.FIXED, prec=prec) as s:
        want = s.solve(rho, 1.0, 1e-9)[0]
    side = torch.cuda.Stream()
    phi = torch.zeros_like(rho)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.default_stream()):
        torch.cuda._sleep(PAUSE)  # the set-up waits behind it
    with mg.Solver(32, 1.0 / 32, mg.FIXED, prec=prec) as s:
        s.solve(rho, 1.0, 1e-9, phi=phi, stream=side)
    assert torch.equal(phi, want)


@pytest.mark.parametrize("stream", ["default", "own"])
def test_batched_solve_follows_pending_work(stream):
    rhos, rhos2 = [source(16), source(32)], [source(16, 5), source(32, 5)]
    st = torch.cuda.default_stream() if stream == "default" else torch.cuda.Stream()
    with mg.Batch([16, 32], [1 / 16, 1 / 32], [mg.FIXED, mg.FIXED]) as b:
        want = [torch.zeros_like(r) for r in rhos]
        b.solve(rhos2, want, 1.0, 1e-9)
        bufs, phis = [r.clone() for r in rhos], [torch.zeros_like(r) for r in rhos]
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            torch.cuda._sleep(PAUSE)
            for p, q in zip(bufs, rhos2):
                p.copy_(q)
        b.solve(bufs, phis, 1.0, 1e-9, stream=st)
        for p, q in zip(phis, want):
            assert torch.equal(p, q)
