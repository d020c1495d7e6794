"""The whole-step 1D kernel at the edges of its tiles (20 output cells for 32 threads, 116 for 128), alone
and batched, and the 2D limiter on total-degree spaces, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2407_19169_gb300 import _native as N
from paper_2407_19169_gb300 import inputs as I

from _helpers import pair, rel_l1

pytestmark = pytest.mark.gpu
INF = float("inf")


# meshes smaller than a tile's halo, one cell short of, at and past one and two tiles of 20
@pytest.mark.parametrize("nx", [1, 2, 5, 13, 19, 20, 21, 40, 41])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
@pytest.mark.parametrize("eq,k", [("burgers", 2), ("euler", 1), ("euler", 3), ("advection", 2)])
def test_tile_edges_match_oracle(nx, bc, eq, k):
    p, s = pair(dim=1, nx=nx, k=k, eq=eq, bc=bc)
    ranges = I.EULER1D_AVG if eq == "euler" else [(0.5, 1.5)]
    u0 = I.random_modal_state(p.shape, 300 + nx, ranges, high_scale=0.02)
    s.write_state(u0)
    s.advance_steps(5)
    st, t, n = s.sync()
    assert st == 0 and n == 5
    ug, tg = s.read_state()
    uo, to, _ = O.advance(p, u0, 0.0, INF, 5)
    assert abs(tg - to) <= 1e-11 * to
    assert rel_l1(p, ug, uo) <= 1e-11


@pytest.mark.parametrize("nx", [21, 115, 116, 117, 232, 233])
@pytest.mark.parametrize("bc", [N.BC_PERIODIC, N.BC_OUTFLOW])
def test_batched_tiles_equal_solo(nx, bc):
    # 32-thread tiles alone, 128-thread tiles in the batch: the same cells, the same digits
    def make():
        s = N.Solver(dim=1, nx=nx, k=2, eq=N.EQ_EULER, bc=(bc,) * 4, precision=N.PREC_FP32_MIXED, positivity=1)
        s.write_state(I.random_modal_state(s.shape, 7, I.EULER1D_AVG, high_scale=0.05))
        return s
    a, b, c = make(), make(), make()
    a.advance_steps(6)
    assert a.sync()[0] == 0
    assert N.batch_run([b], 6) == 0 and N.batch_run([c], 6, persistent=True) == 0
    ua, ta = a.read_state()
    for s in (b, c):
        u, t = s.read_state()
        assert t == ta and np.array_equal(u, ua)
    # and on from there alone: the batched steps leave the step control as the solver's own do
    for s in (a, b, c):
        s.advance_steps(3)
        assert s.sync()[2] == 9
    assert np.array_equal(b.read_state()[0], a.read_state()[0])
    assert np.array_equal(c.read_state()[0], a.read_state()[0])


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_limiter_on_total_degree_spaces(k, bc):
    b = O.BC_PERIODIC if bc == "periodic" else O.BC_OUTFLOW
    p = O.Problem(dim=2, nx=31, ny=9, k=k, basis=O.BASIS_P, eq=O.EQ_EULER, bc=(b,) * 4, positivity=1)
    s = N.Solver(dim=2, nx=31, ny=9, k=k, basis=N.BASIS_P, eq=N.EQ_EULER, positivity=1,
                 bc=(N.BC_PERIODIC if bc == "periodic" else N.BC_OUTFLOW,) * 4)
    rough = I.random_modal_state(p.shape, 60 + k, [(0.5, 1.0), (-0.2, 0.2), (-0.2, 0.2), (0.6, 1.4)], high_scale=1.0,
                                 decay=0.8)
    u0 = O.positivity(p, rough)                        # an admissible start, a third to two thirds limited
    assert (np.abs(u0 - rough).max((0, 1)) > 0).sum() > 50
    s.write_state(u0)
    s.advance_steps(6)
    assert s.sync()[0] == 0
    ug, _ = s.read_state()
    uo, _, _ = O.advance(p, u0, 0.0, INF, 6)
    assert rel_l1(p, ug, uo) <= 1e-10                  # the bar of the limiter's other parity tests
