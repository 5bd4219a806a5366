"""The network's row-block convolutions where a CTA walks several tiles with its full
number of rows, the last row block of an image is shorter and the last column tile
partial; the pooled input gradient of an upsampling layer on the same shapes."""
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


@pytest.mark.parametrize("n,h,w", [(3, 312, 520), (1, 8, 1040), (4, 256, 512)])
def test_rows_of_several_tiles(n, h, w):
    # weights, biases and inputs are short dyadic numbers: the activations are exact on
    # both sides; in the gradients 1 / M is not, and a BF16 rounding falls the other
    # way about once in 10^4 values (2^-8 of one value): bounded at 2e-3 of the norm
    flat, x, t = synth.unet_dyadic_case(U.param_shapes(32), 5, n, h, w)
    net = wec.Net(h, w, max_batch=n)
    net.set_params(flat)
    out = torch.zeros((n, h, w), dtype=torch.float32, device="cuda")
    net.forward(torch.from_numpy(x).cuda(), out)
    ref, A = U.forward(flat.astype(np.float64), x.astype(np.float64), 32, emulate_bf16=True)
    for li, (name, _, _, _) in enumerate(U.layers(32)[:-1]):
        assert np.array_equal(net.activation(li, n, A[name].shape).astype(np.float64), A[name]), name
    assert np.array_equal(out.cpu().numpy().astype(np.float64), ref)
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    g = net.grads().astype(np.float64)
    net.close()
    _, gref = U.loss_and_grads(flat.astype(np.float64), x.astype(np.float64), t.astype(np.float64), 32, emulate_bf16=True)
    k = 0
    for s in U.param_shapes(32):
        m = int(np.prod(s))
        assert np.linalg.norm(g[k:k + m] - gref[k:k + m]) <= 2e-3 * np.linalg.norm(gref[k:k + m]) + 1e-12, s
        k += m
