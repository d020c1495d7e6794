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


# Densities of 1e-30 (intergalactic gas in CGS units), and of 1e-20 and 1e25 with velocities of 1e-12 and
# 1e10 (FP64; their energies leave FP32's range): squared momenta leave that range long before the rate does.
@pytest.mark.parametrize("rho,speed,precision", [(1e-30, 1e6, N.PREC_FP64), (1e-30, 1e6, N.PREC_FP32_MIXED),
                                                 (1e-30, 1.0, N.PREC_FP64), (1e-30, 1.0, N.PREC_FP32_MIXED),
                                                 (1e-20, 1e-12, N.PREC_FP64), (1e25, 1e10, N.PREC_FP64)])
@pytest.mark.parametrize("dim,nx,ny", [(1, 300, 1), (2, 20, 15)])
@pytest.mark.parametrize("limiter", [0, 1])
def test_first_dt_of_states_far_from_one(rho, speed, precision, dim, nx, ny, limiter):
    # a fast cold stream (rate 1.5 speed / h) hides the one hot cell at rest (1.6 speed / h) only where its
    # kinetic energy is lost from its pressure (1.73 in 1D, 1.9 in 2D)
    p = O.Problem(dim=dim, nx=nx, ny=ny, k=2, eq=O.EQ_EULER, bc=(O.BC_PERIODIC,) * 4, positivity=limiter)
    u = np.zeros(p.shape)
    c, v = np.full(nx * ny, 0.5 * speed), np.full(nx * ny, speed)
    hot = nx * ny // 3
    c[hot], v[hot] = 1.6 * speed, 0.0
    u[0, 0] = rho
    for d in range(dim):
        u[1 + d, 0] = rho * v
    u[-1, 0] = rho * (c * c / (1.4 * 0.4) + 0.5 * dim * v * v)
    if precision == N.PREC_FP32_MIXED:               # averages as the form holds them
        hi = u.astype(np.float32)
        u = hi.astype(np.float64) + (u - hi).astype(np.float32)
    s = N.Solver(dim=dim, nx=nx, ny=ny, k=2, eq=N.EQ_EULER, bc=(N.BC_PERIODIC,) * 4, positivity=limiter,
                 precision=precision)
    s.write_state(u)
    dt = s.step()
    assert abs(dt - O.dt(p, u)) <= 1e-13 * dt


@pytest.mark.parametrize("rho,speed", [(1.0, 1.0), (1e-30, 1e6)])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_later_dt_of_states_far_from_one(rho, speed, k):
    # the rate over the limiter's points that a step leaves for the next (2D, FP32 form): a narrow mesh, where
    # a warp's lanes see, in one column, rows that vary smoothly from the stream to the hot gas at rest
    p = O.Problem(dim=2, nx=3, ny=40, k=k, eq=O.EQ_EULER, bc=(O.BC_PERIODIC,) * 4, positivity=1)
    u = np.zeros(p.shape)
    part = np.repeat(0.5 + 0.5 * np.cos(2 * np.pi * np.arange(40) / 40), 3)
    c, v = speed * (1.6 - 1.1 * part), speed * part
    u[0, 0], u[1, 0], u[2, 0] = rho, rho * v, rho * v
    u[3, 0] = rho * (c * c / (1.4 * 0.4) + v * v)
    s = N.Solver(dim=2, nx=3, ny=40, k=k, eq=N.EQ_EULER, bc=(N.BC_PERIODIC,) * 4, positivity=1,
                 precision=N.PREC_FP32_MIXED, tile_rows=40)
    s.write_state(u)
    s.step()
    after, _ = s.read_state()
    # FP32 rates of the state as stored
    assert s.step() == pytest.approx(O.dt(p, after), rel=1e-5)
