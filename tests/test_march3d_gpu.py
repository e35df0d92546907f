"""The z-marching 3D stage at the sizes where its tiles (28 columns; 4, 8 or 12 rows) and
strips of layers begin and end, every flux and compiled diffusion kind, against the FP64
oracle; conservation of the FP32-mixed update."""
import math

import numpy as np
import pytest

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_11527_gb300 import build
    build.build()


def solver(spec, rk=3, prec="fp64"):
    from paper_2510_11527_gb300 import Solver
    return Solver(spec, precision=prec, rk=rk)


FLUX = {"zero": ("zero", ()), "linear": ("linear", (1.0, -0.6, 0.3)), "burgers": ("burgers", (0.5,))}
DIFF = {"none": ("none", ()), "const": ("const", (0.01,)), "pme2": ("pme", (2,)), "pme3": ("pme", (3,)),
        "pwl": ("pwl", (0.05, 0.25, 0.05, 0.75))}


def box(n, flux, diff, limiter=True):
    return ai.Spec(dim=3, nx=n[0], ny=n[1], nz=n[2], x0=0.0, x1=1.3, y0=0.0, y1=0.9, z0=0.0, z1=0.7, umin=0.0,
                   umax=1.0, limiter=limiter, flux=FLUX[flux], diff=DIFF[diff])


def far(a, b):
    return max(float(np.max(np.abs(np.asarray(x, dtype=np.float64) - y))) for x, y in zip(a, b))


SIZES = [(1, 1, 1), (2, 9, 1), (28, 12, 3), (29, 13, 4), (27, 25, 9), (57, 5, 2), (3, 4, 40)]
MODELS = [("zero", "pme2"), ("zero", "const"), ("zero", "pwl"), ("linear", "const"), ("linear", "none"),
          ("burgers", "pme3"), ("burgers", "none"), ("burgers", "pme2")]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("flux,diff", MODELS)
@pytest.mark.parametrize("limiter", [True, False])
def test_forward_euler_at_tile_edges(n, flux, diff, limiter):
    spec = box(n, flux, diff, limiter)
    st = [a.numpy() for a in ai.random_state_3d(spec, seed=sum(n))]
    tau = oracle.dt_cfl(spec, st[0])
    want = oracle.fe(spec, st, tau)
    with solver(spec) as s:
        s.set_state(st)
        s.forward_euler(tau)
        assert far(s.get_state(), want) <= 1e-12
    # FP32-mixed: inputs rounded to FP32 (2^-24), stencils in FP32 (the bound of the
    # other 3D tests)
    with solver(spec, prec="fp32_mixed") as s:
        s.set_state(st)
        s.forward_euler(tau)
        got = s.get_state()
    assert far(got, want) <= 1e-5
    if spec.cells > 1000:   # a mean over a few values is no mean
        assert max(float(np.mean(np.abs(g - w))) for g, w in zip(got, want)) <= 1e-6


@pytest.mark.parametrize("rk", [3, 54])
@pytest.mark.parametrize("n", [(30, 14, 5), (5, 30, 33)])
@pytest.mark.parametrize("flux,diff", [("zero", "pme2"), ("burgers", "const")])
def test_steps_at_tile_edges(rk, n, flux, diff):
    spec = box(n, flux, diff)
    spec.rk = rk
    st = [a.numpy() for a in ai.random_state_3d(spec, seed=3)]
    ref = [a.copy() for a in st]
    with solver(spec, rk=rk) as s:
        s.set_state(st)
        for _ in range(2):
            dt = oracle.dt_cfl(spec, ref[0])
            ref, stats = oracle.step(spec, rk, ref, dt)
            s.step(dt)
        assert s.stats()["errors"] == 0
        assert far(s.get_state(), ref) <= 1e-12


@pytest.mark.parametrize("flux,diff", [("zero", "pme2"), ("burgers", "pwl"), ("linear", "none")])
def test_fp32_mixed_conserves_mass(flux, diff):
    """A face's terms enter its two cells from the same FP32 values with opposite signs,
    each cell's sum of them good to ~46 bits and then rounded to FP64."""
    spec = box((40, 27, 30), flux, diff)
    st = [a.numpy() for a in ai.random_state_3d(spec, seed=8)]
    tau = oracle.dt_cfl(spec, st[0])
    with solver(spec, prec="fp32_mixed") as s:
        s.set_state(st)
        s.forward_euler(tau)
        got = s.get_state()[0]
    # increments are below 1 per cell: 2^-44 each at worst, added up
    assert abs(math.fsum(got.ravel()) - math.fsum(st[0].ravel())) <= got.size * 2.0 ** -44
    assert float(np.max(np.abs(got - st[0]))) > 1e-3


@pytest.mark.parametrize("flux", ["zero", "linear"])
def test_fp32_mixed_averages_are_updated_in_fp64(flux):
    """A linear problem scaled by 2^-100 has the same roundings: the values (0.5 .. 1 before),
    potentials and fluxes (coefficients 2^-1 and 2^-2) keep FP32's normal range, with their
    last places at 2^-126 or above, and FP64 is far from its own. So the result is the
    unscaled one times 2^-100 bit for bit, if the averages' increment holds FP64: FP32 parts
    of it would lose their last bits below 2^-149."""
    spec = box((40, 27, 30), "zero", "const", limiter=False)
    spec.diff = ("const", (0.5,))
    if flux == "linear":
        spec.flux = ("linear", (1.0, -0.5, 0.25))
    spec.umin, spec.umax = 0.5, 1.0
    st = [a.numpy() for a in ai.random_state_3d(spec, seed=5, lo=0.5, hi=1.0)]
    st = [st[0]] + [a.astype(np.float32).astype(np.float64) for a in st[1:]]
    tau = oracle.dt_cfl(spec, st[0])
    out = []
    for scale in (1.0, 2.0 ** -100):
        spec.umin, spec.umax = 0.5 * scale, scale
        with solver(spec, prec="fp32_mixed") as s:
            s.set_state([a * scale for a in st])
            s.forward_euler(tau)
            out.append(s.get_state())
    assert far([out[0][0]], [st[0]]) > 1e-3
    for a, b in zip(*out):
        assert np.array_equal(a * 2.0 ** -100, b)
