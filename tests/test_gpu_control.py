"""Host-side control of a solve: how many steps dg_advance_to enqueues, and the launches that are counted."""
import numpy as np
import pytest

from paper_2407_19169_gb300 import _native as N

pytestmark = pytest.mark.gpu


def test_advance_to_with_a_growing_step_enqueues_few_idle_steps():
    # a spike of 500 in one cell collapses: the first step size says 4000 steps, some 410 are taken
    s = N.Solver(dim=1, nx=200, k=2, eq=N.EQ_BURGERS, bc=(N.BC_PERIODIC,) * 4)
    u = np.zeros(s.shape)
    u[0, 0] = 1.0
    u[0, 0, 100] = 500.0
    s.write_state(u)
    l0 = s.kernel_launches()
    steps = s.advance_to(0.8 / 200)
    assert steps > 200
    # a 1D step is one launch; no chunk is longer than four times the steps before it
    assert s.kernel_launches() - l0 <= 2 * steps


@pytest.mark.parametrize("eq,rate", [(N.EQ_BURGERS, 1), (N.EQ_ADVECTION, 1), (N.EQ_EULER, 2)])
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("precision,convert", [(N.PREC_FP64, 0), (N.PREC_FP32_MIXED, 1)])
def test_launches_of_a_written_state(dim, eq, rate, precision, convert):
    # the conversion to the FP32 form's storage and the rate: Euler first brackets it, then evaluates
    s = N.Solver(dim=dim, nx=16, ny=16 if dim == 2 else 1, k=1, eq=eq, bc=(N.BC_PERIODIC,) * 4, precision=precision)
    u = np.zeros(s.shape)
    u[:, 0] = 0.0 if eq == N.EQ_EULER else 1.0
    if eq == N.EQ_EULER:
        u[0, 0], u[-1, 0] = 1.0, 2.5
    for _ in range(2):
        l0 = s.kernel_launches()
        s.write_state(u)
        assert s.kernel_launches() - l0 == convert + rate
