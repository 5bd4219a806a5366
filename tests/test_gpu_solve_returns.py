"""What a host-polled pressure solve leaves behind when it returns."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2206_07732_gb300 import build as B  # noqa: E402
from paper_2206_07732_gb300 import synth  # noqa: E402
from paper_2206_07732_gb300 import wec  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    wec.load()


@pytest.mark.parametrize("zero", [False, True])
def test_stream_has_drained(zero):
    # the caller may free or reuse b and x, or read x on any stream, once the call is back
    nx, ny = 32, 16
    s = torch.cuda.Stream()
    bu, bv = synth.random_coefficients(nx, ny, seed=1, contrast=10.0)
    P = wec.Poisson(nx, ny, stream=s.cuda_stream)
    P.set_coefficients(torch.from_numpy(bu).cuda(), torch.from_numpy(bv).cuda())
    b = np.zeros((ny, nx)) if zero else np.random.default_rng(2).standard_normal((ny, nx))
    b, x = torch.from_numpy(b).cuda(), torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    solve, args = wec.load().wec_poisson_solve, (P.h, wec._dev(b), wec._dev(x), 1e-8, 100, C.byref(C.c_int()),
                                                 C.byref(C.c_double()))
    early = 0
    for _ in range(500):
        assert solve(*args) == wec.WEC_OK
        early += not s.query()
    assert early == 0
    P.close()


def test_stream_has_drained_after_a_tank_solve():
    s = torch.cuda.Stream()
    cfg = synth.tank_small(seed=0, nx=64, ny=32)
    t = wec.Tank(cfg, stream=s.cuda_stream)
    t.step(cfg["dt"])
    b = torch.from_numpy(np.random.default_rng(3).standard_normal((32, 64))).cuda()
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    early = 0
    for _ in range(200):
        t.pressure_solve(b, x, 1e-8)
        early += not s.query()
    assert early == 0
    t.close()


SLEEPS = """
import ctypes as C, time
cu, d = C.CDLL("libcuda.so.1"), C.c_int()
assert cu.cuInit(0) == 0 and cu.cuDeviceGet(C.byref(d), 0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(d, 4) == 0  # CU_CTX_SCHED_BLOCKING_SYNC, this process's context
import torch
from paper_2206_07732_gb300 import synth, wec
n = (256, 128, 128)
b = torch.randn(n[::-1], dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(0))
P, x = wec.Poisson3(*n), torch.zeros_like(b)
P.set_coefficients(*[torch.from_numpy(a).cuda() for a in synth.random_coefficients3(*n, seed=1, contrast=10.0)])
P.solve(b, x, rtol=1e-8)
w, c = time.perf_counter(), time.thread_time()
for _ in range(10):
    x.zero_()
    P.solve(b, x, rtol=1e-10)
print((time.thread_time() - c) / (time.perf_counter() - w))
"""


def test_a_process_that_asked_to_sleep_sleeps():
    # an Arnoldi step of this grid is some 0.8 ms of GPU time and a few dozen launches of
    # a few us each: a host that sleeps meanwhile uses well under half of its core, one
    # that spins all of it
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SLEEPS], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert float(r.stdout) < 0.5
