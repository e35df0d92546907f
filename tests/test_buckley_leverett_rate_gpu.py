"""Buckley-Leverett wave speeds: the CFL rate over rows in segments (1024 columns, one per
block at a time) with its largest value or the interior extremum that decides it at a
segment's, row's or mesh's edge; and the speeds of the LLF flux over intervals that hold
extrema on either side of zero, with and without the limiter, against the oracle."""
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


@pytest.mark.parametrize("nx,ny", [(5, 4), (1023, 5), (1024, 4), (1025, 5), (2049, 4)])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
@pytest.mark.parametrize("prec", ["fp64", "fp32_mixed"])
def test_rate_at_segment_edges(nx, ny, bc, prec):
    from paper_2510_11527_gb300 import Solver
    spec = ai.Spec(dim=2, nx=nx, ny=ny, x0=0, x1=0.02 * nx, y0=0, y1=0.015 * ny, flux=("bl", (5.0,)),
                   diff=("const", (0.001,)), umin=0.0, umax=1.0, bc=bc)
    flat = [np.full_like(a.numpy(), 0.02) for a in ai.random_state_2d(spec, seed=1)]
    with Solver(spec, precision=prec) as s:
        for i in sorted({0, nx // 2, min(1023, nx - 1), min(1024, nx - 1), nx - 1}):
            # 0.4: the largest rate is a cell's; 0.95: an extremum between the cell and its
            # neighbours
            for j, u in ((0, 0.4), (ny - 1, 0.95), (ny // 2, 0.95)):
                st = [a.copy() for a in flat]
                st[0][j, i] = u
                s.set_state(st)
                want = oracle.dt_cfl(spec, st[0])
                assert abs(s.dt_cfl() - want) <= 1e-14 * want, (i, j, u)


@pytest.mark.parametrize("gravity", [0.0, 1.0, 5.0, -5.0])   # extrema per direction: 2, 1 or 2
@pytest.mark.parametrize("limiter", [True, False])
@pytest.mark.parametrize("blend", ["off", "plain"])
def test_speeds_over_intervals_with_extrema(gravity, limiter, blend):
    from paper_2510_11527_gb300 import Solver
    spec = ai.Spec(dim=2, nx=61, ny=47, x0=0, x1=1.5, y0=0, y1=1.0, flux=("bl", (gravity,)), diff=("const", (0.01,)),
                   umin=-0.8, umax=0.95, limiter=limiter, blend=blend)
    st = [a.numpy() for a in ai.random_state_2d(spec, seed=7)]
    tau = oracle.dt_cfl(spec, st[0])
    want = oracle.fe(spec, st, tau)
    with Solver(spec, precision="fp32_mixed") as s:
        s.set_state(st)
        s.forward_euler(tau)
        got = s.get_state()
        assert s.stats()["errors"] == 0
    # FP32 stencils: the bounds of the other FP32-mixed comparisons (values of order 1)
    assert max(float(np.max(np.abs(np.asarray(g, np.float64) - w))) for g, w in zip(got, want)) <= 1e-5
    assert max(float(np.mean(np.abs(np.asarray(g, np.float64) - w))) for g, w in zip(got, want)) <= 1e-6


@pytest.mark.parametrize("gravity", [0.0, 5.0])
@pytest.mark.parametrize("blend", ["off", "plain"])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_speeds_of_a_state_written_beyond_the_bounds(gravity, blend, bc):
    """A state written in place can reach beyond the bounds, over extrema of f' that no
    limited state meets (f_1': 1.366 and -0.366): its speeds are still those of the interval,
    FP32-mixed as FP64."""
    from paper_2510_11527_gb300 import Solver
    spec = ai.Spec(dim=2, nx=61, ny=47, x0=0, x1=1.5, y0=0, y1=1.0, flux=("bl", (gravity,)), diff=("const", (0.01,)),
                   umin=0.0, umax=1.0, blend=blend, bc=bc)
    inside = [a.numpy() for a in ai.random_state_2d(spec, seed=7)]
    got = {}
    for prec in ("fp64", "fp32_mixed"):
        rng = np.random.default_rng(3)
        with Solver(spec, precision=prec) as s:
            s.set_state(inside)
            for t in s.device_tensors():
                t.copy_(torch.from_numpy(rng.uniform(-0.8, 1.8, tuple(t.shape)).astype(np.float32)))
            torch.cuda.synchronize()
            s.forward_euler(0.25 * oracle.dt_cfl(spec, inside[0]))
            got[prec] = s.get_state()
    # FP32 stencils: the bounds of the other FP32-mixed comparisons (values of order 1)
    d = [np.abs(a - b) for a, b in zip(got["fp64"], got["fp32_mixed"])]
    assert max(float(x.max()) for x in d) <= 1e-5
    assert max(float(x.mean()) for x in d) <= 1e-6
