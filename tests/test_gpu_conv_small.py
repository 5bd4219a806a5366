"""The rule between one-row tiles and row blocks: a network made for one image runs its
convolutions in one-row tiles where these are at most one per SM, one made for a large
batch in row blocks.  Both add an output's products in the same order, so the same
image gives the same bits in all activations, the output and the gradients."""
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


LEVELS = [0, 0, 1, 1, 1, 2, 2, 2, 3, 3, 3, 2, 2, 2, 1, 1, 1, 0, 0, 0]  # of the layers' outputs


# the smallest image; partial column tiles; at level 0 exactly as many tiles as a GB300
# has SMs, and one row block more
@pytest.mark.parametrize("h,w", [(8, 8), (24, 136), (64, 128), (96, 200), (152, 128), (160, 128), (8, 1040)])
def test_one_row_tiles_and_row_blocks_agree(h, w):
    x = np.random.default_rng(h + w).standard_normal((1, h, w, 2)).astype(np.float32)
    t = np.random.default_rng(h * w).standard_normal((1, h, w)).astype(np.float32)
    x, t = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    flat = synth.unet_weights(wec.net_param_shapes(), 3)
    got = []
    for max_batch in (1, 4096 // h + 1):  # (at level 2 more than 4 tiles per SM)
        net = wec.Net(h, w, max_batch=max_batch)
        net.set_params(flat)
        out = torch.zeros((1, h, w), dtype=torch.float32, device="cuda")
        net.forward(x, out)
        r = [out.cpu().numpy()]
        for li, ((_, _, _, c), lev) in enumerate(zip(U.layers(32)[:-1], LEVELS)):
            r.append(net.activation(li, 1, (1, h >> lev, w >> lev, c)))
        net.loss_grad(x, t)
        got.append(r + [net.grads()])
        net.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
