"""Calls that mix groups of instances, chained single steps and checks, bitwise
against single steps that are waited for."""
import numpy as np
import pytest

from gpu_helpers import lib
from test_gpu_calls import _context, _state

pytestmark = pytest.mark.gpu

CASES = [("cylindrical", True, (64, 4, 256), 5, "fp32"), ("ellipsoidal", False, (48, 4, 301), 5, "fp16_shifted"),
         ("cylindrical", True, (17, 3, 41), 2, "fp64")]


def _waited_for(L, call, steps):
    c = _context(L, *call)
    for _ in range(steps):
        c.lb_step(1)
        c.stream.synchronize()
    s = _state(c)
    c.close()
    return s


@pytest.mark.parametrize("call", CASES, ids=lambda c: f"{c[0]}-{'x'.join(map(str, c[2]))}-b{c[3]}-{c[4]}")
@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
def test_checks_groups_and_single_steps(call, batch):
    """Checks every 7 steps cut calls into groups and single steps."""
    L = lib()
    c = _context(L, *call)
    b = L.LBBatch([c]) if batch else None
    (b.lb_batch_set_option if batch else c.lb_set_option)(L.LB_OPT_CHECK_EVERY, 7)
    for n in (5, 11, 1, 2, 9):
        b.lb_batch_step(n) if batch else c.lb_step(n)
    assert np.array_equal(_state(c), _waited_for(L, call, 28))
    if batch:
        b.close()
    c.close()
