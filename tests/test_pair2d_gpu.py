"""The column-marching FP32-mixed stage with two columns per lane against the FP64 oracle on
meshes large enough to take it, at the edges of its bands of 60 columns (even and odd
widths: paired and single memory accesses), every compiled diffusion kind; and the strip
heights of the column-marching kernels, which change no value, with every flux."""
import numpy as np
import pytest

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_11527_gb300 import build
    build.build()


FLUX = {"zero": ("zero", ()), "linear": ("linear", (1.0, -0.6)), "burgers": ("burgers", (0.5,))}
DIFF = {"none": ("none", ()), "const": ("const", (0.01,)), "pme2": ("pme", (2,)), "pme3": ("pme", (3,)),
        "pwl": ("pwl", (0.05, 0.25, 0.05, 0.75)), "cubic": ("cubic", (0.0, 0.02, -0.04 / 3)), "ramp": ("ramp", (0.05, 0.4, 0.2))}


def solver(spec, rk=3):
    from paper_2510_11527_gb300 import Solver
    return Solver(spec, precision="fp32_mixed", rk=rk)


def mesh(nx, ny, flux, diff, limiter=True):
    return ai.Spec(dim=2, nx=nx, ny=ny, x0=-1.5, x1=1.5, y0=-1.5, y1=1.2, flux=FLUX[flux], diff=DIFF[diff], umin=0.0,
                   umax=1.0, limiter=limiter)


# 60 x 21 and 61 x 20 columns: one wave of its warps, where the choice takes two columns
@pytest.mark.parametrize("nx", [1259, 1260, 1261])
@pytest.mark.parametrize("flux,diff,rk,limiter", [
    ("zero", "pme2", 3, True), ("zero", "pme3", 54, True), ("zero", "cubic", 3, True), ("zero", "pwl", 54, True),
    ("zero", "const", 3, False), ("zero", "ramp", 3, True), ("burgers", "pwl", 54, True),
    ("burgers", "none", 3, True), ("burgers", "ramp", 3, False), ("linear", "const", 3, True), ("linear", "pme2", 54, True)])
def test_column_marching_on_larger_meshes(nx, flux, diff, rk, limiter):
    """A band of the mesh's rows is repeated, so the oracle steps one period (40 rows) of
    the 1200: the mesh is periodic in y with that period."""
    period, reps = 40, 30
    small = mesh(nx, period, flux, diff, limiter)
    small.y1 = small.y0 + 0.09
    spec = mesh(nx, period * reps, flux, diff, limiter)
    spec.y1 = spec.y0 + 0.09 * reps
    st = [a.numpy() for a in ai.random_state_2d(small, seed=nx)]
    st = [st[0]] + [a.astype(np.float32).astype(np.float64) for a in st[1:]]
    dt = oracle.dt_cfl(small, st[0])
    ref, _ = oracle.step(small, rk, st, dt)
    with solver(spec, rk) as s:
        s.set_state([np.tile(a, (reps, 1)) for a in st])
        s.step(dt)
        got = s.get_state()
        assert s.stats()["errors"] == 0
        if limiter:
            lo, hi = s.bounds()
            assert lo >= 0.0 and hi <= 1.0
    for g, r in zip(got, ref):
        d = np.abs(g - np.tile(r, (reps, 1)))
        assert float(d.max()) <= 1e-5 and float(d.mean()) <= 1e-6   # FP32 stencils, as the other FP32 tests
        # every period rounds alike whatever strip and band it falls into
        assert all(np.array_equal(g[:period], g[k * period:(k + 1) * period]) for k in range(reps))


@pytest.mark.parametrize("ny,flux,diff", [(1000, "zero", "pme2"), (1400, "zero", "const"), (1000, "burgers", "pwl")])
def test_mass_is_conserved_exactly(ny, flux, diff):
    """Face terms cancel across bands and strips: the mass moves by FP64 rounding only."""
    import math
    spec = mesh(1330, ny, flux, diff)
    st = [a.numpy() for a in ai.random_state_2d(spec, seed=1, lo=0.2, hi=0.8)]
    with solver(spec) as s:
        s.set_state(st)
        s.forward_euler(0.5 * s.dt_cfl())
        got = s.get_state()[0]
    assert abs(math.fsum(got.ravel()) - math.fsum(st[0].ravel())) <= got.size * 2.0 ** -52


def _device_arrays(b, spec):
    """The device arrays (FP64 averages, FP32 points) of a batch's first mesh."""
    import torch
    from paper_2510_11527_gb300 import capi

    def view(ptr, kind):
        class _View:
            __cuda_array_interface__ = {"shape": (spec.ny, spec.nx), "typestr": kind, "data": (ptr, False), "version": 3}
        return torch.as_tensor(_View(), device="cuda")

    ptrs, _ = capi.af_batch_device_ptrs(b, 0)
    return [view(p, "<f8" if k == 0 else "<f4") for k, p in enumerate(ptrs)]


@pytest.mark.parametrize("nx", [1259, 1260, 1261])
@pytest.mark.parametrize("diff", ["const", "pme2", "pme3", "pwl", "cubic", "ramp"])
@pytest.mark.parametrize("rk,limiter", [(3, True), (54, True), (3, False)])
def test_two_columns_equal_one_column(nx, diff, rk, limiter):
    """The mesh's size decides between one and two columns per lane, so both have to give the
    same bits (a zero's sign aside). A batch marches with one column per lane at every size:
    two steps of a batch of one mesh against the single mesh."""
    from paper_2510_11527_gb300 import capi
    spec = mesh(nx, 1200, "zero", diff, limiter)
    st = [a.numpy() for a in ai.random_state_2d(spec, seed=nx + rk)]
    f, d = capi.af_flux(), capi.af_diff()
    f.kind, d.kind = capi.FLUX["zero"], capi.DIFF[spec.diff[0]]
    for k, v in enumerate(spec.diff[1]):
        d.p[k] = v
    b = capi.af_batch_create([capi.af_grid(2, spec.nx, spec.ny, spec.x0, spec.x1, spec.y0, spec.y1)], [f], [d],
                             [capi.af_bounds_t(spec.umin, spec.umax, 0)],
                             capi.af_opts(capi.PREC["fp32_mixed"], rk, 0.0, 0.0, int(limiter), 0, 1.0))
    try:
        capi.af_batch_set_state(b, 0, spec.cells, *st)
        capi.af_batch_step(b, 2)
        capi.af_batch_sync(b)
        want, t = [a.cpu().numpy() for a in _device_arrays(b, spec)], capi.af_batch_time(b, 0)
    finally:
        capi.af_batch_destroy(b)
    with solver(spec, rk) as s:
        s.set_state(st)
        for _ in range(2):
            s.step(0.0)
        assert s.time() == t > 0.0
        got = [a.cpu().numpy() for a in s.device_tensors()]
    assert float(np.max(np.abs(got[0] - st[0]))) > 1e-3
    # the arrays as they are on the device. An unlimited run of the cubic potential, which is
    # unstable outside [0, 1], overflows FP32; there one column forms the convection terms,
    # zero times an infinity, and holds a NaN where two columns hold the infinity
    for g, w in zip(got, want):
        finite = np.isfinite(w)
        assert np.array_equal(finite, np.isfinite(g)) and np.array_equal(g[finite], w[finite])
