"""The network's weight and bias gradients where their GEMMs' cut changes form:
rows of one and several 64-pixel segments with and without a remainder, fewer
units than CTAs and more, a batch below the allocated one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import unet as U  # noqa: E402
from paper_2206_07732_gb300 import build as B  # noqa: E402
from paper_2206_07732_gb300 import synth  # noqa: E402
from paper_2206_07732_gb300 import wec  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    wec.load()


def _gradients(n, h, w, max_batch):
    flat, x, t = synth.unet_dyadic_case(U.param_shapes(32), 11, n, h, w)
    net = wec.Net(h, w, max_batch=max_batch)
    net.set_params(flat)
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    g = net.grads().astype(np.float64)
    net.close()
    _, ref = U.loss_and_grads(flat.astype(np.float64), x.astype(np.float64), t.astype(np.float64), 32, emulate_bf16=True)
    return g, ref


@pytest.mark.parametrize("n,h,w,mb", [(1, 8, 8, 1), (1, 8, 128, 1), (2, 16, 64, 3), (1, 32, 256, 2)])
def test_exact_case(n, h, w, mb):
    # power-of-two pixel counts: every product and sum is exact on both sides
    g, ref = _gradients(n, h, w, mb)
    assert np.array_equal(g, ref)


@pytest.mark.parametrize("n,h,w,mb", [(1, 24, 136, 2), (1, 8, 312, 1), (3, 40, 72, 3)])
def test_ragged_rows(n, h, w, mb):
    # 1 / M is inexact: sums differ in FP32's last bits, and a BF16 rounding falls the
    # other way about once in 10^4 values (2^-8 of one value): 1e-4 of a tensor's norm,
    # bounded at 2e-3
    g, ref = _gradients(n, h, w, mb)
    k = 0
    for s in U.param_shapes(32):
        m = int(np.prod(s))
        assert np.linalg.norm(g[k:k + m] - ref[k:k + m]) <= 2e-3 * np.linalg.norm(ref[k:k + m]) + 1e-12, s
        k += m
