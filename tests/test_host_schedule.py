"""Which launches a call makes, and on which streams: the host side over a
stand-in runtime (host_library.py)."""
import ctypes

import numpy as np
import pytest

from host_library import Host, build_host_library, launches, take_log  # noqa: F401
from paper_1411_3133_gb300 import lbgm as L

SWEEP = ("cylindrical", (64, 4, 256), 5, "fp32")  # five instances of 21.5 MB: groups of one


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return build_host_library(str(tmp_path_factory.mktemp("host")))


class Batch:
    def __init__(self, lib, members):
        self.lib, self.members, self.h = lib, members, ctypes.c_void_p()
        arr = (ctypes.c_void_p * len(members))(*[m.ctx for m in members])
        assert lib.lb_batch_create(arr, len(members), ctypes.byref(self.h)) == L.LB_OK

    def option(self, opt, value):
        assert self.lib.lb_batch_set_option(self.h, opt, value) == L.LB_OK

    def step(self, n):
        assert self.lib.lb_batch_step(self.h, n) == L.LB_OK, self.lib.lb_batch_last_error(self.h)

    def close(self):
        self.lib.lb_batch_destroy(self.h)


def _whole(log, instances):
    """Launches that take every instance at once (the steps outside groups)."""
    return sum(x["count"] == instances for x in log)


@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
@pytest.mark.parametrize("precision", ["fp32", "fp16_shifted"])
def test_checks_do_not_end_the_groups(lib, precision, batch):
    """With a check every 100 steps, a call from step 97 takes 3 steps one by
    one and the others in groups."""
    c = Host(lib, *SWEEP[:3], precision)
    b = Batch(lib, [c]) if batch else None
    for on in filter(None, (c, b)):
        on.option(L.LB_OPT_CHECK_EVERY, 100)
    take = b.step if batch else c.step
    take(97)
    assert _whole(launches(lib), 5) == 0
    take(203)
    log = launches(lib)
    assert _whole(log, 5) == 3
    assert sum(x["count"] for x in log) == 203 * 5
    assert np.array_equal(c.counts(), [300] * 5)
    take(2)
    take(1)
    assert _whole(launches(lib), 5) == 3 and np.array_equal(c.counts(), [303] * 5)
    if batch:
        b.close()
    c.close()


@pytest.mark.parametrize("steps,kernel", [(8, 1), (2, 2)])
def test_autotuner_times_what_a_call_runs(lib, steps, kernel):
    """Node costs at which one launch over all instances is slower than the TMA
    kernel and the groups are faster than both: trials of 4 and more steps see
    the groups, shorter ones (whose calls run without) do not."""
    lib.fake_set_costs(2.0, 0.5e-4, 1e-4, 50e6, 0.8e-4)
    c = Host(lib, *SWEEP)
    best, trials, n = L.lb_tune(), (L.lb_tune * 16)(), ctypes.c_int()
    c.ok(lib.lb_autotune(c.ctx, steps, ctypes.byref(best), trials, 16, ctypes.byref(n)))
    take_log(lib)
    assert n.value == 10 and (best.schedule == 2) == (kernel == 2)
    assert np.array_equal(c.counts(), [10 * (steps + 1)] * 5)
    c.step(8)
    assert {x["kind"] for x in launches(lib)} == {"tma" if kernel == 2 else "f32"}
    c.close()
    lib.fake_set_costs(2.0, 1e-4, 1e-4, 1e18, 1e-4)


@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
def test_streams_of_the_groups_are_like_the_owners(lib, batch):
    """On the context's device, whatever device is current at the first long
    call (which stays current), and with its stream's priority."""
    c = Host(lib, *SWEEP, priority=-3)
    b = Batch(lib, [c]) if batch else None
    take = b.step if batch else c.step
    if not batch:
        lib.fake_set_device(1)
    take(4)
    made = [x for x in take_log(lib) if x["kind"] == "create"]
    assert len(made) == 3 and {(x["device"], x["priority"]) for x in made} == {(0, -3)}
    assert lib.fake_device() == (0 if batch else 1)
    lib.fake_set_device(0)
    if batch:
        b.close()
    c.close()


# groups of one instance; several instances a group; one chained launch a step
LONG = [(("cylindrical", (64, 4, 256), 5, "fp32"), 5), (("cylindrical", (16, 4, 32), 70, "fp16_shifted"), 3),
        (("cylindrical", (64, 4, 256), 1, "fp64"), 1)]


@pytest.mark.parametrize("spec,chunks", LONG, ids=["groups", "small", "chained"])
@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
def test_long_calls_are_replayed(lib, spec, chunks, batch):
    """LB_OPT_USE_GRAPH: of a call of 2000 steps a few are launched by the
    caller, the rest in graphs made once per chunk and first buffer; the graphs
    follow the launch options, and nobody's capture is interrupted."""
    c = Host(lib, *spec)
    b = Batch(lib, [c]) if batch else None
    on, take = (b, b.step) if batch else (c, c.step)
    on.option(L.LB_OPT_USE_GRAPH, 1)
    if batch and spec[2] > 16:
        chunks = 5  # at most 16 instances a launch
    total = 0

    def call(n, made, threads=128):
        nonlocal total
        take(n)
        total += n
        log = take_log(lib)
        steps = [x for x in log if "count" in x]
        assert sum(x["count"] for x in steps) == n * spec[2] and {x["threads"] for x in steps} == {threads}
        assert sum(x["kind"] == "instantiate" for x in log) == made
        assert np.array_equal(c.counts(), [total] * spec[2])
        return [x for x in steps if not x["replay"]]

    take_log(lib)
    assert len(call(2000, chunks)) <= 31 * chunks
    assert len(call(2000, 0)) <= 31 * chunks
    call(1001, chunks)     # an odd number of steps first: the other buffer
    call(333, 0)
    call(1000, 0)
    on.option(L.LB_OPT_BLOCK_THREADS, 64)
    call(320, chunks, 64)
    assert all(not x["replay"] for x in call(20, 0, 64))       # short calls are launched
    lib.fake_capture(c.stream, 1)
    take(2000)             # goes into the caller's own graph
    lib.fake_capture(c.stream, 0)
    assert not [x for x in take_log(lib) if x["kind"] == "instantiate"]
    if batch:
        b.close()
    c.close()


def test_replays_follow_the_parameters(lib):
    """lb_init may switch to the half-force kernel and back."""
    c = Host(lib, *SWEEP)
    c.option(L.LB_OPT_USE_GRAPH, 1)
    for old_forcing, kind in ((0, "f32"), (2, "shift32"), (0, "f32")):
        c.init(old_forcing)
        take_log(lib)
        c.step(320)
        assert {x["kind"] for x in launches(lib)} == {kind}
        assert np.array_equal(c.counts(), [320] * 5)
    c.close()


def _channel(metric, nr, ntheta, n3, periodic3=True):
    from oracle.geometry import Channel
    return Channel(metric, 1.0, 1.0 / 0.975, nr, ntheta, n3, periodic3=periodic3)


@pytest.mark.parametrize("steps", [1, 3, 4, 20])
@pytest.mark.parametrize("precision", ["fp32", "fp16_shifted", "fp64"])
def test_bench_counts_the_launches(lib, precision, steps):
    """bench.step_launches (its gpu_launches) against the launches of the
    library: uniform contexts, and batches of unlike channels."""
    import bench
    for ch, batch in ((_channel("cylindrical", 64, 4, 256), 24), (_channel("ellipsoidal", 64, 4, 256, False), 7),
                      (_channel("cylindrical", 16, 4, 32), 70), (_channel("cylindrical", 96, 8, 400), 3)):
        c = Host(lib, ch.metric, (ch.nr, ch.ntheta, ch.n3), batch, precision, ch.periodic3)
        take_log(lib)
        c.step(steps)
        assert len(launches(lib)) == steps * bench.step_launches([ch] * batch, precision, steps)
        c.close()
    chs = [_channel("cylindrical", 32 + 16 * (i % 3), 4, 128 + 37 * i) for i in range(7)] + \
        [_channel("ellipsoidal", 64, 4, 200 + 31 * i, False) for i in range(19)]
    stream = lib.fake_stream(0)
    members = [Host(lib, ch.metric, (ch.nr, ch.ntheta, ch.n3), 1, precision, ch.periodic3, stream=stream) for ch in chs]
    b = Batch(lib, members)
    take_log(lib)
    b.step(steps)
    assert len(launches(lib)) == steps * bench.step_launches(chs, precision, steps, 16)
    b.close()
    for m in members:
        m.close()


@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
@pytest.mark.parametrize("precision,instances,threads,chained",
                         [("fp64", 3, 128, True), ("fp64", 4, 128, False), ("fp64", 9, 128, False),
                          ("fp64", 10, 128, True), ("fp64", 9, 64, True), ("fp64", 3, 64, False),
                          ("fp32", 6, 128, True), ("fp16_shifted", 8, 128, True)])
def test_fp64_steps_of_one_block_per_sm_are_not_chained(lib, precision, instances, threads, chained, batch):
    """16 x 4 x 32 nodes: 16 blocks of 128 an instance, 152 SMs. Between a third
    of them and all, two blocks of a chained FP64 step meet on one SM."""
    c = Host(lib, "cylindrical", (16, 4, 32), instances, precision)
    b = Batch(lib, [c]) if batch else None
    (b or c).option(L.LB_OPT_BLOCK_THREADS, threads)
    for n in (1, 12):
        take_log(lib)
        (b or c).step(n)
        log = launches(lib)
        assert len(log) == n and {x["chained"] for x in log} == {int(chained)}
    if batch:
        b.close()
    c.close()


@pytest.mark.parametrize("metric,n3", [("cylindrical", 401), ("cylindrical", 8), ("flat", 256)])
def test_walls_on_x3_cost_no_memory(lib, metric, n3):
    """2-byte storage: a channel walled on x3 holds 5 rows of the stream table an
    i_r layer instead of one, 4 x 416 bytes, and more source keys (x3 classes);
    not a row for every pair of nodes, 208 bytes a node of the cross-section."""
    alloc_t, free_t = (dict(L.lb_allocator._fields_)[k] for k in ("alloc", "free"))
    libc = ctypes.CDLL(None)
    libc.malloc.restype, libc.malloc.argtypes = ctypes.c_void_p, [ctypes.c_size_t]
    libc.free.argtypes = [ctypes.c_void_p]
    held = {}
    for periodic3 in (True, False):
        total = [0]

        def grab(n, stream, user):
            total[0] += n
            return libc.malloc(n)

        a = L.lb_allocator(alloc=alloc_t(grab), free=free_t(lambda p, n, stream, user: libc.free(p)))
        desc = L.make_desc(1.0, 1.0 / 0.975, 130, 1, n3, periodic3=periodic3)
        c = ctypes.c_void_p()
        assert lib.lb_create_geometry(L.METRICS[metric], ctypes.byref(desc), 3, L.PRECISIONS["fp16_shifted"],
                                      ctypes.c_void_p(lib.fake_stream(0)), ctypes.byref(a), ctypes.byref(c)) == L.LB_OK
        held[periodic3] = total[0]
        lib.lb_destroy(c)
    assert held[False] <= held[True] + 3 * 130 * 4 * 416 + 7 * 7 * 7 * 176


def test_long_tiles_leave_two_blocks_per_sm(lib):
    """LB_OPT_TILE_BLOCKS 4 in blocks of 128 nodes: 512 an instance of 65536 (64 x 4
    x 256), so tiles of one block (4 would be 128 of them for 152 SMs); 10 instances
    of 16384 on their own, one launch of 1280, take tiles of 4 (320)."""
    for batch, size, n, tile in ((5, (64, 4, 256), 8, 128), (10, (32, 4, 128), 1, 512)):
        c = Host(lib, "cylindrical", size, batch, "fp32")
        b = Batch(lib, [c])
        b.option(L.LB_OPT_TILE_BLOCKS, 4)
        take_log(lib)
        b.step(n)
        assert {x["tile"] for x in launches(lib)} == {tile}
        b.close()
        c.close()
