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


# FP32 stencils where the viscous terms carry the step (mu dt / (rho h^2) from 1e-1 to
# 1e3; the tanks' is 1e-6): u* = R / D' + Q S is then a weighted mean of neighbouring
# velocities in some ten FP32 roundings (the mirror of u, four products and their sums,
# the reciprocal and the two factors, the last sum), 2^-24 of the value each -- the
# explicit half among them, as long as its rounding scales with the velocity's
# differences or is no larger than these.
@pytest.mark.parametrize("n_jacobi", [1, 3])
@pytest.mark.parametrize("mu", [1e2, 1e4, 1e6])
def test_fp32_stencils_at_large_viscosity(mu, n_jacobi):
    nx, ny = 128, 64
    cfg = synth.tank_small(seed=0)
    cfg["body"] = None
    cfg["solver"]["n_jacobi"] = n_jacobi
    cfg["mu_w"] = cfg["mu_a"] = mu
    g, o = wec.Tank(cfg, precision=wec.PREC_MIXED), O.OracleTank(cfg)
    x, y = np.linspace(0.0, 6.0, nx + 1), np.linspace(0.0, 5.0, ny + 1)[:, None]
    u, v = 0.37 + 0.01 * np.sin(x + y[:-1]), 0.21 + 0.01 * np.cos(y - x[:-1])
    u[:, -1] = 0.0
    v[0, :] = 0.0
    g.set("u", u)
    o.set(O.F_U, u)
    g.set("v", v)
    o.set(O.F_V, v)
    g.step(cfg["dt"], 0.0)
    o.step(cfg["dt"], 0.0)
    a, b = g.get("ustar")[8:-8, 8:-8], o.get(O.F_USTAR)[8:-8, 8:-8]
    assert np.max(np.abs(a - b)) < 10 * 2.0 ** -24 * np.max(np.abs(b))
