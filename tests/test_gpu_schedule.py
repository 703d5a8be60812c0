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


REPLAYED = CASES + [("cylindrical", True, (16, 4, 32), 70, "bf16_shifted"), ("cylindrical", True, (16, 4, 32), 1, "fp32"),
                    ("ellipsoidal", False, (16, 4, 33), 2, "fp16_shifted")]


@pytest.mark.parametrize("call", REPLAYED, ids=lambda c: f"{c[0]}-{'x'.join(map(str, c[2]))}-b{c[3]}-{c[4]}")
@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
def test_replayed_long_calls(call, batch):
    """From either buffer, twice, and with launched steps in between."""
    L = lib()
    c = _context(L, *call)
    b = L.LBBatch([c]) if batch else None
    (b.lb_batch_set_option if batch else c.lb_set_option)(L.LB_OPT_USE_GRAPH, 1)
    for n in (289, 256, 3, 300):
        b.lb_batch_step(n) if batch else c.lb_step(n)
    assert np.array_equal(_state(c), _waited_for(L, call, 848))
    if batch:
        b.close()
    c.close()


def test_a_callers_capture_takes_a_long_call():
    """With LB_OPT_USE_GRAPH, on a stream that the caller captures."""
    import torch
    L = lib()
    c = _context(L, *CASES[0])
    c.lb_set_option(L.LB_OPT_USE_GRAPH, 1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=c.stream, capture_error_mode="thread_local"):
        c.lb_step(260)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(_state(c), _waited_for(L, CASES[0], 260))
    c.close()


@pytest.mark.parametrize("call", [("cylindrical", True, (64, 4, 256), 8, "fp32"),
                                  ("cylindrical", True, (64, 4, 256), 1, "fp64")], ids=["groups", "chained"])
def test_a_long_call_returns_before_its_steps(call):
    """LB_OPT_USE_GRAPH keeps the caller free: under 0.3 of the steps' time is
    spent in the call (launched one by one nine tenths in the groups, three
    quarters in the chained launches, whose queue holds 1000; replayed a few
    percent)."""
    import time

    import torch
    L = lib()
    c = _context(L, *call)
    c.lb_set_option(L.LB_OPT_USE_GRAPH, 1)
    held = []
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        c.lb_step(4000)
        h = time.perf_counter() - t
        torch.cuda.synchronize()
        held.append(h / (time.perf_counter() - t))
    assert min(held) < 0.3
    c.close()


@pytest.mark.parametrize("plan", [False, True], ids=["one", "groups"])
def test_replayed_pairs_of_the_tma_and_half_force_kernels(plan):
    """Calls that replay a captured pair of steps -- the TMA kernel, the
    half-force variant -- from either buffer and across an lb_init that changes
    the kernel, against single steps that are waited for."""
    L = lib()
    spec = L.ChannelSpec("cylindrical", 1.0, 1.0 / 0.975, 48, 4, 256)
    batch = 6 if plan else 1
    outs = []
    for graph in (1, 0):
        c = L.LBContext(spec, batch=batch, precision="fp32")
        c.lb_set_option(L.LB_OPT_USE_GRAPH, graph)
        states = []
        for forcing, kernel in ((0, 2), (2, 2), (2, 1), (0, 2), (0, 1)):
            c.lb_set_option(L.LB_OPT_STEP_KERNEL, kernel)
            c.lb_init([L.make_params(0.6 + 0.05 * i, 1e-5, forcing, 1 + i, 1e-3, False) for i in range(batch)])
            for n in (1, 37, 8, 3):
                if graph:
                    c.lb_step(n)
                else:
                    for _ in range(n):
                        c.lb_step(1)
                        c.stream.synchronize()
            states.append(_state(c))
        outs.append(states)
        c.close()
    assert all(np.array_equal(a, b) for a, b in zip(*outs))
    assert not np.array_equal(outs[0][0], outs[0][1])      # the variant is another step


def test_small_fp64_steps_leave_each_other_their_sms():
    """Contexts whose blocks fit the SMs one by one take about the time of one:
    1.07 for two of 24 blocks, 1.0 for one of 49 against one of 24 (1.46 and 1.4
    while the blocks of several steps to come waited on the SMs)."""
    import time

    import torch
    L = lib()

    def us(blocks, contexts):
        cs = [L.LBContext(L.ChannelSpec("cylindrical", 1.0, 1.05, blocks, 1, 128), batch=1, precision="fp64")
              for _ in range(contexts)]
        for c in cs:
            c.lb_init([L.make_params(0.8, 1e-6, False, 1, 1e-4, False)])
        best = 1e9
        for _ in range(8):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for c in cs:
                c.lb_step(100)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        for c in cs:
            c.close()
        return best * 1e4

    one = us(24, 1)
    assert us(49, 1) < 1.2 * one
    assert us(24, 2) < 1.25 * one


def test_tma_step_between_four_walls_costs_what_two_do():
    """8 channels of 64 x 4 x 256: 39 us a step with walls on x3 too, 34 without
    (100 with the wall rule evaluated node by node)."""
    import time

    import torch
    L = lib()
    best = {}
    for metric, periodic3 in (("ellipsoidal", False), ("cylindrical", True)):
        c = L.LBContext(L.ChannelSpec(metric, 1.0, 1.025, 64, 4, 256, periodic3=periodic3), batch=8, precision="fp32")
        c.lb_set_option(L.LB_OPT_STEP_KERNEL, 2)
        c.lb_init([L.make_params(0.8, 1e-6, False, 1, 1e-4, False)] * 8)
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            t = time.perf_counter()
            c.lb_step(50)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        best[metric] = min(times)
        c.close()
    assert best["ellipsoidal"] < 1.6 * best["cylindrical"]
