"""Strongly cancelling Arnoldi columns.  On a grid that is its own coarsest level the
preconditioner is the operator's inverse to its working precision, so the new vector w
of an Arnoldi step lies in the span of the basis to 1e-7 (FP32 cycle) or 1e-15 (FP64):
the orthogonalised rest u is small beside w, and its rounding is amplified by |w| / |u|.
The Givens estimate then still has to end the cycle where the true residual does."""
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


def solve(P, coef, b, rtol):
    P.set_coefficients(*(cuda(a) for a in coef))
    x = torch.zeros_like(cuda(b))
    r = P.solve(cuda(b), x, rtol=rtol, max_iters=100)
    P.close()
    return r, x.cpu().numpy()


# The conditions are 4e2 to 7e3, so a step leaves at most 1.1e-16 times that of the
# residual with an FP64 inverse and 6e-8 times it, 4e-4, with an FP32 one: 1e-12 takes
# two steps, or four, at most.  An estimate that the lost orthogonality spoiled would
# end the cycle late (further steps) or early (a further cycle, one step at least).
# The residual as the oracle forms it differs by its own rounding, a few 1e-16 times
# the condition.
@pytest.mark.parametrize("contrast", [1.0, 1e2])
@pytest.mark.parametrize("shape", [(15, 15), (21, 22), (7, 8, 9), (9, 5, 11)])
@pytest.mark.parametrize("prec", [wec.PREC_FP64, wec.PREC_MIXED, wec.PREC_MIXED_DF])
def test_direct_preconditioner(shape, prec, contrast):
    d3 = len(shape) == 3
    if prec == wec.PREC_MIXED_DF and not d3:
        pytest.skip("float-pair Arnoldi steps are the 3D operator's")
    coef = (synth.random_coefficients3 if d3 else synth.random_coefficients)(*shape, seed=5, contrast=contrast)
    b = np.random.default_rng(1).standard_normal(shape[::-1])
    r, x = solve((wec.Poisson3 if d3 else wec.Poisson)(*shape, precision=prec, restart=32), coef, b, 1e-12)
    assert r["status"] == wec.WEC_OK and r["relres"] <= 1e-12
    assert r["iters"] <= (2 if prec == wec.PREC_FP64 else 4)
    ax = O3.apply(*coef, x) if d3 else O.poisson_apply(*coef, x)
    assert np.linalg.norm(b - ax) <= 4e-12 * np.linalg.norm(b)


# Long cycles on a high contrast, against the oracle's two measured passes: the same
# Krylov space, so the same number of steps (one more or less where the estimate
# passes the tolerance by less than its rounding).
@pytest.mark.parametrize("shape", [(64, 32), (16, 16, 16)])
def test_long_cycles_take_the_oracles_steps(shape):
    d3 = len(shape) == 3
    coef = (synth.random_coefficients3 if d3 else synth.random_coefficients)(*shape, seed=1, contrast=1e3)
    b = np.random.default_rng(2).standard_normal(shape[::-1])
    r, _ = solve((wec.Poisson3 if d3 else wec.Poisson)(*shape, restart=32), coef, b, 1e-12)
    o = (O3.solve if d3 else O.poisson_solve)(*coef, b, rtol=1e-12, restart=32)
    assert r["status"] == wec.WEC_OK
    assert abs(r["iters"] - o[1]["iters"]) <= 1
