"""Short meshes: whole steps of a 1D mesh in one cluster launch against the launched
stages, and the tile shapes of short meshes against the oracle, at the sizes where the
choice or the last tile changes."""
import numpy as np
import pytest

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_11527_gb300 import build
    build.build()


def solver(spec, prec="fp64", rk=3):
    from paper_2510_11527_gb300 import Solver
    return Solver(spec, precision=prec, rk=rk)


def spec1d(n, bc, flux, blend="off", limiter=True):
    f = {"burgers": ("burgers", (0.5,)), "bl": ("bl", (5.0,)), "linear": ("linear", (1.0, 0.0)), "zero": ("zero", ())}[flux]
    return ai.Spec(dim=1, nx=n, x0=-0.3, x1=0.9, flux=f, diff=("ramp", (0.05, 0.4, 0.2)), umin=0.0, umax=1.0,
                   limiter=limiter, blend=blend, bc=bc, bc_values=(1.0, 0.0))


def far(a, b):
    return max(float(np.max(np.abs(x - y))) for x, y in zip(a, b))


# tiles of 26 cells, 8 CTAs of up to 4 of them: 208 cells is one tile each, 832 the longest
@pytest.mark.parametrize("n", [4, 26, 27, 208, 209, 832])
@pytest.mark.parametrize("bc,flux,prec,rk,blend", [
    ("dirichlet", "burgers", "fp64", 3, "off"), ("outflow", "burgers", "fp32_mixed", 54, "plain"),
    ("periodic", "bl", "fp64", 54, "plain"), ("dirichlet", "bl", "fp32_mixed", 3, "off"),
    ("outflow", "bl", "fp64", 3, "off"), ("periodic", "linear", "fp64", 3, "off"), ("periodic", "zero", "fp64", 54, "off")])
def test_whole_steps_equal_launched_stages(n, bc, flux, prec, rk, blend):
    spec = spec1d(n, bc, flux, blend)
    st = [a.numpy() for a in ai.random_state_1d(spec, seed=n)]
    # the two forms round alike up to the compiler's contraction: a few ulps (of the FP32
    # stencils in the mixed form) per evaluation, grown at most fourfold per stage
    tol = 6 * 4 ** 3 * (2.0 ** -52 if prec == "fp64" else 2.0 ** -23)
    with solver(spec, prec, rk) as a, solver(spec, prec, rk) as b:
        a.set_state(st)
        b.set_state(st)
        dt = a.step(want_dt=True)
        b.dt_device()
        for k in range(b.num_stages):
            b.stage(k, 0.0)
        assert abs(a.time() - b.time()) <= 1e-14 * b.time() and abs(a.time() - dt) <= 1e-15
        assert far(a.get_state(), b.get_state()) <= tol
        # a step of given size
        a.set_state(st)
        b.set_state(st)
        a.step(0.5 * dt)
        b.stage(0, 0.5 * dt)
        for k in range(1, b.num_stages):
            b.stage(k, 0.0)
        assert far(a.get_state(), b.get_state()) <= tol


def test_run_of_a_short_mesh_counts_and_lands():
    """More steps than one launch takes, the last one clipped; a second call adds none."""
    spec = spec1d(60, "dirichlet", "burgers")
    st = [a.numpy() for a in ai.random_state_1d(spec, seed=2)]
    dt = oracle.dt_cfl(spec, st[0])
    T = 150.5 * dt
    ref, n, _ = oracle.run(spec, 3, st, T)
    with solver(spec) as s:
        s.set_state(st)
        assert s.run(T) == n
        assert abs(s.time() - T) <= 1e-14 * T
        assert far(s.get_state(), ref) <= 1e-12
        assert s.run(T) == 0


# one-warp tiles up to 152 * 256 cells, 256-cell tiles beyond
@pytest.mark.parametrize("n", [833, 152 * 256, 152 * 256 + 1])
@pytest.mark.parametrize("bc,flux,blend", [("dirichlet", "burgers", "off"), ("outflow", "bl", "plain"), ("periodic", "linear", "off")])
def test_tile_shapes_match_oracle(n, bc, flux, blend):
    spec = spec1d(n, bc, flux, blend)
    st = [a.numpy() for a in ai.random_state_1d(spec, seed=5)]
    dt = oracle.dt_cfl(spec, st[0])
    ref, _ = oracle.step(spec, 3, st, dt)
    with solver(spec) as s:
        s.set_state(st)
        assert abs(s.dt_cfl() - dt) <= 1e-14 * dt
        s.step(dt)
        assert far(s.get_state(), ref) <= 1e-12
