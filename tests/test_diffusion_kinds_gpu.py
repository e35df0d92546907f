"""Every diffusion kind that the tile kernels (FP64 periodic, rectangles with ends) and the
1D kernels compile in, and the 32 x 12 tiles of FP32 rectangles at the tile's edges, against
the oracle."""
import numpy as np
import pytest

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_11527_gb300 import build
    build.build()


DIFF = {"none": ("none", ()), "const": ("const", (0.01,)), "pwl": ("pwl", (0.05, 0.25, 0.08, 0.75)),
        "pwl_lo": ("pwl", (0.05, 0.6, 0.0, 0.75)), "pwl_hi": ("pwl", (0.0, 0.25, 0.08, 0.4)), "pme2": ("pme", (2,)),
        "pme3": ("pme", (3,)), "cubic": ("cubic", (0.0, 0.02, -0.04 / 3)), "cubic01": ("cubic01", (0.0, 0.02, -0.04 / 3)),
        "ramp": ("ramp", (0.05, 0.4, 0.2))}


def run(spec, prec, st, tau):
    from paper_2510_11527_gb300 import Solver
    with Solver(spec, precision=prec) as s:
        s.set_state(st)
        s.forward_euler(tau)
        assert s.stats()["errors"] == 0
        return [np.asarray(a, dtype=np.float64) for a in s.get_state()]


@pytest.mark.parametrize("diff", list(DIFF))
@pytest.mark.parametrize("dim,bc,prec", [(1, "periodic", "fp64"), (1, "outflow", "fp32_mixed"), (2, "periodic", "fp64"),
                                         (2, "outflow", "fp64"), (2, "outflow", "fp32_mixed")])
def test_every_diffusion_kind(diff, dim, bc, prec):
    k = dict(flux=("burgers", (0.5,)), diff=DIFF[diff], umin=0.0, umax=1.0, limiter=True, bc=bc, x0=-0.4, x1=0.8)
    if dim == 1:
        spec = ai.Spec(dim=1, nx=61, **k)
        st = [a.numpy() for a in ai.random_state_1d(spec, seed=11)]
    else:
        spec = ai.Spec(dim=2, nx=41, ny=19, y0=0.0, y1=0.5, **k)
        st = [a.numpy() for a in ai.random_state_2d(spec, seed=11)]
    tau = oracle.dt_cfl(spec, st[0])
    want, got = oracle.fe(spec, st, tau), run(spec, prec, st, tau)
    # the bounds of the other parity tests: rounding (FP64), FP32 stencils on values in [0, 1]
    tol = 1e-12 if prec == "fp64" else 1e-5
    assert max(float(np.max(np.abs(g - w))) for g, w in zip(got, want)) <= tol


# padded columns and rows around whole tiles; (639, 143) is 20 x 12 tiles
@pytest.mark.parametrize("nx,ny", [(607, 143), (607, 144), (608, 145), (639, 143), (640, 144), (641, 145)])
@pytest.mark.parametrize("limiter", [True, False])
def test_taller_tiles_of_fp32_rectangles(nx, ny, limiter):
    spec = ai.Spec(dim=2, nx=nx, ny=ny, x0=-1.0, x1=2.0, y0=0.0, y1=0.7, flux=("burgers", (0.5,)), diff=DIFF["pwl"],
                   umin=0.0, umax=1.0, limiter=limiter, bc="outflow")
    st = [a.numpy() for a in ai.random_state_2d(spec, seed=nx)]
    tau = oracle.dt_cfl(spec, st[0])
    want, got = oracle.fe(spec, st, tau), run(spec, "fp32_mixed", st, tau)
    assert max(float(np.max(np.abs(g - w))) for g, w in zip(got, want)) <= 1e-5
