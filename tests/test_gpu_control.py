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
