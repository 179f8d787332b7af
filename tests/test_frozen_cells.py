"""Frozen cells: how many a handle takes."""
import numpy as np
import pytest

from paper_2007_05718_gb300 import lbrt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [lbrt.LB_RT_F32, lbrt.LB_RT_F16_DEV])
def test_more_than_2_27_frozen_cells(cuda, storage):
    """lb_rt_set_frozen takes any int count.  One direction, two sites: the list
    names site 0 over and over (always with the same value) and site 1 at its
    very end, where 32 threads a cell have passed 2^32."""
    n = (1 << 27) + 1
    cells = np.zeros(n, np.int64)
    values = np.full((n, 1), 3.0, np.float32)
    cells[-1], values[-1] = 1, 8.0
    h = lbrt.lb_rt_create(3, 2, 1, 1, dirs=[[0.0, 0.0, 1.0]], storage=storage,
                          collision=lbrt.LB_RT_EXPLICIT)
    try:
        lbrt.lb_rt_set_state(h, np.ones((1, 1, 1, 2), np.float32))
        lbrt.lb_rt_set_frozen(h, cells, values)
        lbrt.lb_rt_step(h, 1)
        I = np.zeros((1, 1, 1, 2), np.float32)
        lbrt.lb_rt_get_populations(h, I)
    finally:
        lbrt.lb_rt_destroy(h)
    assert I.ravel().tolist() == [3.0, 8.0]
