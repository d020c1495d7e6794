"""The CFL rate of a written state (bracketed in FP32, evaluated in FP64) and the conversion between
the canonical FP64 layout and the FP32 form's storage."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19169_gb300 import _native as N
from paper_2407_19169_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _state(shape, dim, kind, seed):
    ranges = I.EULER1D_AVG if dim == 1 else I.EULER2D_AVG
    u = I.random_modal_state(shape, seed, ranges, high_scale=0.1)
    if kind == "constant":                       # every cell a candidate, none with higher modes
        u[:] = 0.0
        u[0, 0], u[1, 0], u[-1, 0] = 1.0, 0.3, 2.5
    elif kind == "peak":                         # one cell far above the others
        u[1, 1] *= 0.01
        u[1, 1, shape[2] // 2] = 0.5
    return u


# 1, 255, 257: around a block of the rate kernel; 70001: threads that take several cells
@pytest.mark.parametrize("kind", ["rough", "constant", "peak"])
@pytest.mark.parametrize("dim,nx,ny,k,basis", [(1, 3, 1, 1, "Q"), (1, 257, 1, 3, "Q"), (1, 700001, 1, 2, "Q"),
                                               (2, 5, 51, 1, "Q"), (2, 16, 16, 2, "P"), (2, 33, 29, 2, "Q"),
                                               (2, 31, 9, 3, "Q"), (2, 257, 3, 3, "P")])
@pytest.mark.parametrize("limiter", [0, 1])
def test_first_dt_is_the_fp64_rate(kind, dim, nx, ny, k, basis, limiter):
    p = O.Problem(dim=dim, nx=nx, ny=ny, k=k, eq=O.EQ_EULER, basis=O.BASIS_Q if basis == "Q" else O.BASIS_P,
                  bc=(O.BC_PERIODIC,) * 4, positivity=limiter)
    u = _state(p.shape, dim, kind, 90 + k).astype(np.float32).astype(np.float64)   # exact in both forms
    for precision in (N.PREC_FP64, N.PREC_FP32_MIXED):
        s = N.Solver(dim=dim, nx=nx, ny=ny, k=k, eq=N.EQ_EULER, basis=N.BASIS_Q if basis == "Q" else N.BASIS_P,
                     bc=(N.BC_PERIODIC,) * 4, positivity=limiter, precision=precision)
        s.write_state(u)
        dt = s.step()
        # the same FP64 formulas on the same point values: a few operations' rounding
        assert abs(dt - O.dt(p, u)) <= 1e-13 * dt


@pytest.mark.parametrize("dim,nx,ny,k,eq,basis", [(1, 1, 1, 1, "euler", "Q"), (1, 257, 1, 2, "euler", "Q"),
                                                  (1, 300, 1, 3, "burgers", "Q"), (2, 1, 1, 1, "euler", "P"),
                                                  (2, 17, 15, 1, "euler", "Q"), (2, 19, 27, 2, "euler", "Q"),
                                                  (2, 16, 16, 3, "euler", "Q"), (2, 257, 2, 2, "euler", "P"),
                                                  (2, 13, 11, 3, "advection", "P")])
def test_storage_round_trip(dim, nx, ny, k, eq, basis):
    s = N.Solver(dim=dim, nx=nx, ny=ny, k=k, eq={"euler": N.EQ_EULER, "burgers": N.EQ_BURGERS,
                                                 "advection": N.EQ_ADVECTION}[eq],
                 basis=N.BASIS_Q if basis == "Q" else N.BASIS_P, precision=N.PREC_FP32_MIXED)
    u = np.random.default_rng(7).uniform(0.5, 1.5, s.shape)
    s.write_state(u, 0.25)
    r, t = s.read_state()
    assert t == 0.25
    hi = u[:, 0].astype(np.float32)
    lo = (u[:, 0] - hi).astype(np.float32)
    assert np.array_equal(r[:, 0], hi.astype(np.float64) + lo)
    assert np.array_equal(r[:, 1:], u[:, 1:].astype(np.float32).astype(np.float64))
