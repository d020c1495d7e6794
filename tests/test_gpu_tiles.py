"""The 2D tile shape (rows per warp item, warps per block) changes only the schedule: every shape
the autotuner may pick, 1-warp blocks and the library's default schedule (0, 0) give bitwise the
same state."""
import time

import numpy as np
import pytest

from paper_2407_19169_gb300 import _native as N
from paper_2407_19169_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TILES = [(8, 2), (16, 4), (32, 8), (64, 2), (128, 4), (8, 1), (0, 0)]


def run(tile, precision, k):
    s = N.Solver(dim=2, nx=90, ny=70, k=k, eq=N.EQ_EULER, bc=(N.BC_OUTFLOW,) * 4, precision=precision,
                 tile_rows=tile[0], tile_warps=tile[1])
    s.set_initial(N.IC_QUADRANT2D, I.quadrant_params(1))
    s.advance_steps(12)
    st, t, n = s.sync()
    assert st == 0 and n == 12
    u, t = s.read_state()
    s.close()
    return u, t


@pytest.mark.parametrize("precision", [N.PREC_FP32_MIXED, N.PREC_FP64])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_tile_shape_does_not_change_the_result(precision, k):
    ref, t_ref = run(TILES[0], precision, k)
    for tile in TILES[1:]:
        u, t = run(tile, precision, k)
        assert t == t_ref, tile
        np.testing.assert_array_equal(u, ref, err_msg=str(tile))


@pytest.mark.parametrize("k,limiter", [(2, 1), (3, 1), (2, 0)])
def test_solvers_with_different_default_tiles_side_by_side(k, limiter):
    # the default block of a small and of a large mesh differ; each solver's first launches come after
    # the other was created
    def make(n):
        s = N.Solver(dim=2, nx=n, ny=n, k=k, eq=N.EQ_EULER, bc=(N.BC_OUTFLOW,) * 4, precision=N.PREC_FP32_MIXED,
                     positivity=limiter)
        s.set_initial(N.IC_QUADRANT2D, I.quadrant_params(1))
        return s
    sizes = [40, 90, 214, 300, 64]
    solvers = [make(n) for n in sizes]
    for s in solvers + solvers[::-1]:
        s.advance_steps(3)
        assert s.sync()[0] == 0
    for s in solvers:
        s.set_target(1.0)
    assert N.batch_run(solvers, 2) == 0
    assert N.batch_run(solvers, 2, persistent=True) == 0
    for s in solvers:
        assert s.sync()[2] == 10


def _limited(tile, k, kind, precision=N.PREC_FP32_MIXED):
    s = N.Solver(dim=2, nx=90, ny=70, k=k, eq=N.EQ_EULER, bc=(N.BC_OUTFLOW,) * 4, precision=precision,
                 tile_rows=tile[0], tile_warps=tile[1], positivity=1)
    if kind == "quadrants":
        s.set_initial(N.IC_QUADRANT2D, I.quadrant_params(1))
    else:
        # a stream whose waves run across the strips: the largest rate is met in every row, to rounding
        x = (np.arange(90) + 0.5) / 90
        rho = np.broadcast_to(1.0 + 0.2 * np.sin(6 * np.pi * x), (70, 90)).ravel()
        u = np.zeros(s.shape)
        u[0, 0], u[1, 0], u[2, 0], u[3, 0] = rho, 0.7 * rho, 0.3 * rho, 2.5 + 0.29 * rho
        u[:, 1] = 0.01 * u[:, 0]
        s.write_state(u)
    return s


# with the limiter in the FP32 form the rate that sets dt is summed again for the cells with the largest rates:
# which they are must not follow the cut into tiles, nor how far a clipped step was
@pytest.mark.parametrize("kind", ["quadrants", "stream"])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_tile_shape_does_not_change_the_limited_result(k, kind):
    def steps(tile):
        s = _limited(tile, k, kind)
        s.advance_steps(40)
        s.advance_to(s.sync()[1] * 1.0101)              # ends on a clipped step
        s.advance_steps(40)
        assert s.sync()[0] == 0
        out = s.read_state()
        s.close()
        return out
    ref, t_ref = steps(TILES[0])
    for tile in TILES[1:]:
        u, t = steps(tile)
        assert t == t_ref, tile
        np.testing.assert_array_equal(u, ref, err_msg=str(tile))


# the batched runs cut a class's meshes into chunks of their own
@pytest.mark.parametrize("kind", ["quadrants", "stream"])
@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("persistent", [False, True])
def test_batched_limited_results_equal_solo(k, kind, persistent):
    solo, batched = (_limited((0, 0), k, kind) for _ in range(2))
    others = [_limited((0, 0), k, "quadrants") for _ in range(3)]
    solo.advance_steps(30)
    T = solo.sync()[1] * 1.0101
    solo.advance_to(T)
    clipped = solo.sync()[2]
    solo.advance_steps(30)
    for s in others:
        s.set_target(T, 1 << 40)
    batched.set_target(T, 1 << 40)
    assert N.batch_run([batched] + others, clipped, persistent=persistent) == 0
    assert batched.sync() == (0, T, clipped)
    batched.set_target(float("inf"), 1 << 40)
    assert N.batch_run([batched] + others, 30, persistent=persistent) == 0
    u, t = solo.read_state()
    ub, tb = batched.read_state()
    assert tb == t
    np.testing.assert_array_equal(ub, u)


@pytest.mark.parametrize("limiter", [0, 1])
def test_eight_warps_cost_no_more_than_two_blocks_of_four(limiter):
    # 2048^2 in 128 rows: 1184 items, a round of 1216 resident warps with either block; seven-warp blocks take two
    def step_time(warps):
        s = N.Solver(dim=2, nx=2048, ny=2048, k=2, eq=N.EQ_EULER, bc=(N.BC_OUTFLOW,) * 4, positivity=limiter,
                     precision=N.PREC_FP32_MIXED, tile_rows=128, tile_warps=warps)
        s.set_initial(N.IC_QUADRANT2D, I.quadrant_params(1))
        best = np.inf
        for _ in range(4):                                    # the first pass warms up
            t0 = time.perf_counter()
            s.advance_steps(8)
            assert s.sync()[0] == 0
            best = min(best, time.perf_counter() - t0)
        s.close()
        print("%d warps: %.1f us per step" % (warps, best / 8 * 1e6))
        return best

    assert step_time(8) <= 1.3 * step_time(4)
