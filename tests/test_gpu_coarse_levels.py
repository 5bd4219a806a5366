"""The coarse part of a V-cycle -- one thread-block cluster down to a level
applied as a matrix, the coarsest level's explicit inverse -- at the sizes where
its cut into slabs, its cell pairs per thread and its banded factor change form,
against the FP64 oracle's V-cycle and against the per-level kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import poisson3d as O3  # noqa: E402
from oracle import tank as O  # noqa: E402
from paper_2206_07732_gb300 import build as B  # noqa: E402
from paper_2206_07732_gb300 import synth  # noqa: E402
from paper_2206_07732_gb300 import wec  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    wec.load()


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


# FP64 V-cycles agree with the oracle's to 1e-11 (some 10^2 roundings of size
# 1.1e-16 per cell, amplified by the coarse inverse's norm); FP32 ones to 1e-4.
TOL = {wec.PREC_FP64: 1e-11, wec.PREC_MIXED: 1e-4}

# 2D: coarsest levels of 484 (22 x 22: widest band), 511, 18 and 2 cells; grids of
# one, two and all cluster levels; slabs that leave CTAs of the cluster without rows
GRIDS2 = [(22, 22), (14, 146), (36, 18), (4, 4), (88, 88), (352, 176), (24, 416), (704, 96), (512, 256)]


@pytest.mark.parametrize("prec", [wec.PREC_FP64, wec.PREC_MIXED])
@pytest.mark.parametrize("nx,ny", GRIDS2)
def test_vcycle_2d_matches_oracle(nx, ny, prec):
    bu, bv = synth.random_coefficients(nx, ny, seed=nx + 3 * ny, contrast=10.0)
    b = np.random.default_rng(4).standard_normal((ny, nx))
    P = wec.Poisson(nx, ny, precision=prec)
    P.set_coefficients(cuda(bu), cuda(bv))
    z = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    P.vcycle(cuda(b), z)
    assert rel(z.cpu().numpy(), O.vcycle(bu, bv, b)[0]) < TOL[prec]
    P.close()


# 3D: coarsest levels of 504 (7 x 8 x 9: a band larger than shared memory in
# FP64), 490, 45 and 8 cells, each side the longest once; uneven slabs
GRIDS3 = [(14, 16, 18), (18, 16, 14), (16, 18, 14), (14, 10, 28), (36, 40, 8), (4, 4, 8), (56, 20, 28), (40, 72, 24),
          (64, 32, 32)]


@pytest.mark.parametrize("prec", [wec.PREC_FP64, wec.PREC_MIXED])
@pytest.mark.parametrize("shape", GRIDS3)
def test_vcycle_3d_matches_oracle_and_level_kernels(shape, prec):
    nx, ny, nz = shape
    coef = synth.random_coefficients3(nx, ny, nz, seed=sum(shape), contrast=10.0)
    b = np.random.default_rng(5).standard_normal((nz, ny, nx))
    z = {}
    for on in (0, 1):
        wec.set_option("mg3_bottom", on)
        P = wec.Poisson3(nx, ny, nz, precision=prec)
        P.set_coefficients(*(cuda(a) for a in coef))
        t = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
        P.vcycle(cuda(b), t)
        z[on] = t.cpu().numpy()
        P.close()
    wec.set_option("mg3_bottom", 1)
    assert rel(z[1], O3.vcycle(*coef, b)[0]) < TOL[prec]
    assert np.array_equal(z[0], z[1])


@pytest.mark.parametrize("prec", [wec.PREC_FP64, wec.PREC_MIXED])
@pytest.mark.parametrize("pre,post", [(1, 0), (1, 1), (3, 0), (2, 4)])
def test_sweep_counts(pre, post, prec):
    # 3D: the per-level kernels' bits; 2D: the one-pass kernels' values to rounding
    # (an FP32 V-cycle: a few hundred roundings of 6e-8)
    shape = (64, 24, 40)
    nx, ny, nz = shape
    coef = synth.random_coefficients3(nx, ny, nz, seed=2, contrast=10.0)
    b3 = cuda(np.random.default_rng(6).standard_normal((nz, ny, nx)))
    z = []
    for on in (0, 1):
        wec.set_option("mg3_bottom", on)
        P = wec.Poisson3(nx, ny, nz, precision=prec, mg_pre=pre, mg_post=post)
        P.set_coefficients(*(cuda(a) for a in coef))
        t = torch.zeros_like(b3)
        P.vcycle(b3, t)
        z.append(t.cpu().numpy())
        P.close()
    wec.set_option("mg3_bottom", 1)
    assert np.array_equal(z[0], z[1])
    bu, bv = synth.random_coefficients(256, 96, seed=8, contrast=10.0)
    b2 = cuda(np.random.default_rng(7).standard_normal((96, 256)))
    z = []
    for fused in (0, 1):
        wec.set_option("mg_fused", fused)
        P = wec.Poisson(256, 96, precision=prec, mg_pre=pre, mg_post=post)
        P.set_coefficients(cuda(bu), cuda(bv))
        t = torch.zeros_like(b2)
        P.vcycle(b2, t)
        z.append(t.cpu().numpy())
        P.close()
    wec.set_option("mg_fused", 1)
    assert rel(z[1], z[0]) < (1e-12 if prec == wec.PREC_FP64 else 1e-4)
