"""Diagnostics of a batch in which a box refuses: the boxes before it are filled in, as if the
boxes were asked one by one."""
import numpy as np
import pytest

from paper_1507_02518_gb300 import lb

pytestmark = pytest.mark.gpu


def test_boxes_before_a_refusing_one_are_filled():
    batch = lb.Batch([{"n": 16, "nu": 1e-3, "urms": 0.04}] * 3, storage="f32", scheme="pull")
    u = np.zeros((3, 16, 16, 16))
    u[0] = 0.01
    for k in range(3):
        lb.lb_init_field(batch.box(k), None, u.ctypes.data, False)
    box = batch.box(1)
    lb.lb_set_kernel(box, "staged")
    lb.lb_set_wait_budget(box, 200000, True)  # its copies never come: the wait runs out
    lb.lb_step(box, 1)
    for call in range(2):  # the time-out itself, then the state that it left
        out = (lb.lb_diag * 3)()
        for d in out:
            d.nodes = -1
        assert lb.load().lb_batch_diagnostics(batch.handle, out) == lb.LB_ERR_TIMEOUT
        assert out[0].nodes == 16 ** 3
        assert abs(out[0].mass - 16 ** 3) <= 16 ** 3 * 27 * 2.0 ** -24
        assert out[2].nodes == -1
        assert b"box 1" in lb.load().lb_batch_last_error(batch.handle)
