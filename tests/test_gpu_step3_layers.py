"""The 3D transport kernel on grids large enough that a thread walks several layers
(two; eight), against the one-kernel form of the momentum
system, which forms every face for itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2206_07732_gb300 import build as B  # noqa: E402
from paper_2206_07732_gb300 import synth  # noqa: E402
from paper_2206_07732_gb300 import wec  # noqa: E402

FIELDS = (wec.F3_SIGMA, wec.F3_U, wec.F3_V, wec.F3_W, wec.F3_P)


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    wec.load()


@pytest.mark.parametrize("prec", [wec.PREC_FP64, wec.PREC_MIXED_DF])
@pytest.mark.parametrize("shape", [(128, 32, 80), (128, 128, 80)])
def test_walked_layers_agree_with_single_faces(shape, prec):
    # the same arithmetic per face: the same bits in float pairs (explicit products and
    # sums); in FP64 a product may be contracted into a sum in one kernel and not in the
    # other, an ulp per face value: 1e-12 after a step that solves to 1e-12
    c = synth.tank3d(seed=3, nx=shape[0], ny=shape[1], nz=shape[2], rtol=1e-12)
    rng = np.random.default_rng(3)
    out = []
    try:
        for split in (1, 0):
            wec.set_option("tank3_split_momentum", split)
            t = wec.Tank3(c, precision=prec)
            if not out:  # both flow directions in every limiter
                start = {f: t.get(f) + 0.05 * rng.standard_normal(t.shapes[f]) for f in (wec.F3_U, wec.F3_V, wec.F3_W)}
            for f, a in start.items():
                t.set(f, a)
            assert t.step(c["dt"])["status"] == 0
            out.append([t.get(f) for f in FIELDS])
            t.close()
    finally:
        wec.set_option("tank3_split_momentum", 1)
    for f, a, b in zip(FIELDS, *out):
        assert np.max(np.abs(a - b)) <= (1e-12 if prec == wec.PREC_FP64 else 0.0) * max(np.max(np.abs(b)), 1e-12), f
