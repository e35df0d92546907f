"""The CFL rate of a state that holds a NaN or an average too large for FP32: neither hides
behind the other cells' rates. A NaN average makes the step 0, so that a run ends at once; a
large finite one decides the rate as any other does."""
import numpy as np
import pytest
import torch

import af_inputs as ai
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2510_11527_gb300 import build
    build.build()


FLUX = {"bl": ("bl", (5.0,)), "burgers": ("burgers", (0.5,))}
# a short 1D mesh (whole steps in one launch), a longer one, 2D meshes with several segments
# per row and rows per block, a 3D mesh
MESH = {"1d-200": dict(dim=1, nx=200), "1d-3000": dict(dim=1, nx=3000), "2d-70x40": dict(dim=2, nx=70, ny=40),
        "2d-1030x700": dict(dim=2, nx=1030, ny=700), "3d": dict(dim=3, nx=20, ny=11, nz=9, z0=0.0, z1=1.0)}


def _spec(mesh, flux, limiter):
    # (no diffusion, whose cap on the step would stand in for a rate that is NaN)
    return ai.Spec(x0=0.0, x1=1.0, y0=0.0, y1=1.0, flux=FLUX[flux], umin=0.0, umax=1.0, limiter=limiter, **MESH[mesh])


def _state(spec, value):
    kinds = 2 ** spec.dim
    shape = {1: (spec.nx,), 2: (spec.ny, spec.nx), 3: (spec.nz, spec.ny, spec.nx)}[spec.dim]
    st = [np.full(shape, value) for _ in range(kinds)]
    st[0].ravel()[0] = 0.4   # the largest rate is this cell's
    return st


CASES = [("1d-200", "bl"), ("1d-3000", "bl"), ("2d-70x40", "bl"), ("2d-1030x700", "bl"), ("1d-200", "burgers"),
         ("1d-3000", "burgers"), ("2d-70x40", "burgers"), ("3d", "burgers")]


@pytest.mark.parametrize("mesh,flux", CASES)
@pytest.mark.parametrize("limiter", [True, False])
@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
@pytest.mark.parametrize("bits", [0x7FF8000000000000, 0xFFF8000000000000, 0xFFFFFFFFFFFFFFFF])
def test_a_nan_average_stops_the_run(mesh, flux, limiter, prec, bits):
    from paper_2510_11527_gb300 import Solver, capi
    spec = _spec(mesh, flux, limiter)
    for cell in (0, 1, spec.cells // 2 + 3, spec.cells - 1):
        with Solver(spec, precision=prec) as s:
            s.set_state(_state(spec, 0.02))
            T = 2.5 * s.dt_cfl()
            ub = s.device_tensors()[0].view(-1)
            ub.view(torch.int64)[cell] = int(np.array(bits, dtype=np.uint64).view(np.int64))
            assert bool(torch.isnan(ub[cell]))
            with pytest.raises(capi.AfError) as ei:
                s.run(T)
            assert ei.value.status == capi.AF_E_STATE
            assert s.time() == 0.0


@pytest.mark.parametrize("mesh", ["1d-3000", "2d-70x40", "2d-1030x700"])
def test_an_average_beyond_fp32_decides_the_rate(mesh):
    """f_2' of the gravity flux grows with u: 1e25 is a finite rate in FP64, while its square
    overflows in FP32."""
    from paper_2510_11527_gb300 import Solver
    spec = _spec(mesh, "bl", False)
    for cell in (1, spec.cells // 2 + 3, spec.cells - 1):
        st = _state(spec, 0.02)
        st[0].ravel()[cell] = 1e25
        want = oracle.dt_cfl(spec, st[0])
        with Solver(spec) as s:
            s.set_state(st)
            got = s.dt_cfl()
            assert abs(got - want) <= 1e-12 * want
