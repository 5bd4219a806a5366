"""The 2D step's stencil kernels at the sizes where their cut changes form --
grids without a cell whose stencil is inside, rows of 31 control volumes per
warp and one more, rows of one and two tiles -- one step against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import tank as O  # noqa: E402
from paper_2206_07732_gb300 import build as B  # noqa: E402
from paper_2206_07732_gb300 import synth  # noqa: E402
from paper_2206_07732_gb300 import wec  # noqa: E402

FIELDS = [("sigma", O.F_SIGMA, 1e-9), ("u", O.F_U, 1e-6), ("v", O.F_V, 1e-6), ("p", O.F_P, 1e-6),
          ("ustar", O.F_USTAR, 1e-6), ("vstar", O.F_VSTAR, 1e-6), ("beta_u", O.F_BETA_U, 1e-300),
          ("beta_v", O.F_BETA_V, 1e-300), ("sigma_adv", O.F_SIGMA_ADV, 1e-9)]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    wec.load()


@pytest.mark.parametrize("nx,ny", [(8, 8), (16, 8), (32, 16), (62, 14), (124, 32), (128, 16), (248, 32), (256, 24)])
def test_one_step_matches_oracle(nx, ny):
    # the plain path's bar: 1e-10 of the field's largest value, from a state with
    # random velocities (both flow directions in every limiter)
    cfg = synth.tank_small(seed=nx + ny, rtol=1e-13)
    h = 1.0 / 32.0
    cfg.update(nx=nx, ny=ny, lx=nx * h, ly=ny * h, depth=0.5 * ny * h, damp_x0=0.75 * nx * h, damp_len=0.25 * nx * h,
               probe_x=0.25 * nx * h)
    cfg["wave"]["H"] = 0.02 * ny * h
    cfg["body"] = None if ny < 16 else synth.box_body(0.5 * nx * h, 0.2 * nx * h, 0.3 * ny * h, 0.15 * ny * h,
                                                      cfg["depth"], cfg["rho_w"])
    g, o = wec.Tank(cfg), O.OracleTank(cfg)
    r = synth.random_fields(nx, ny, seed=nx, scale=0.05)
    u, v = o.get(O.F_U) + r["u"], o.get(O.F_V) + r["v"]
    u[:, -1] = 0.0
    v[0, :] = 0.0
    g.set("u", u)
    o.set(O.F_U, u)
    g.set("v", v)
    o.set(O.F_V, v)
    g.step(cfg["dt"], 2.0)
    o.step(cfg["dt"], 2.0)
    for name, fo, floor in FIELDS:
        a, b = g.get(name), o.get(fo)
        assert np.max(np.abs(a - b)) < 1e-10 * max(np.max(np.abs(b)), floor), name
