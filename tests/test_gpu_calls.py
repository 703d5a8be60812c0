"""What one call of several steps does against the same steps one by one (the
groups of instances kept in L2, chained launches), and the surrogate's gradients
at the edges of its tiles."""
import numpy as np
import pytest

from gpu_helpers import lib
from mlp_reference import grads
from test_gpu_mlp import _inputs, _net

pytestmark = pytest.mark.gpu


def _context(L, metric, periodic3, size, batch, precision, stream=None):
    spec = L.ChannelSpec(metric, 1.0, 1.0 / 0.975, *size, periodic3=periodic3)
    c = L.LBContext(spec, batch=batch, precision=precision, stream=stream)
    c.lb_init([L.make_params(0.6 + 0.05 * i, 1e-5, False, 1 + i, 1e-3, False) for i in range(batch)])
    return c


def _state(c):
    buf = np.zeros(c.lb_state_bytes(), np.uint8)
    return c.lb_get_state(buf).copy()


# one instance a group and several; a last group with one instance less; batches
# below the groups' size (one chained launch a step)
CALLS = [("cylindrical", True, (64, 4, 256), 5, "fp32"), ("cylindrical", True, (64, 4, 256), 7, "fp16_shifted"),
         ("ellipsoidal", False, (48, 4, 301), 5, "bf16_shifted"), ("cylindrical", True, (64, 4, 250), 3, "fp64"),
         ("ellipsoidal", False, (16, 4, 33), 2, "fp32"), ("cylindrical", True, (16, 4, 32), 1, "fp16_shifted"),
         ("cylindrical", True, (17, 3, 41), 2, "fp64")]


@pytest.mark.parametrize("n", [4, 9])
@pytest.mark.parametrize("call", CALLS, ids=lambda c: f"{c[0]}-{'x'.join(map(str, c[2]))}-b{c[3]}-{c[4]}")
def test_a_call_of_n_steps_is_n_calls(call, n):
    """Bitwise, also with two calls in a row (the parity of n)."""
    L = lib()
    a, b = _context(L, *call), _context(L, *call)
    for _ in range(2):
        a.lb_step(n)
        for _ in range(n):
            b.lb_step(1)
    assert np.array_equal(_state(a), _state(b))
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp16_shifted", "fp64"])
def test_a_batch_call_is_the_members_steps(precision):
    """Work lists of unlike channels in groups, against lb_step on each."""
    import torch
    L = lib()
    st = torch.cuda.Stream()
    specs = [("cylindrical", True, (64, 4, 256), 2), ("ellipsoidal", False, (48, 4, 301), 2),
             ("cylindrical", True, (48, 6, 224), 1), ("cylindrical", True, (16, 4, 33), 2)]
    members = [_context(L, *s, precision, stream=st) for s in specs]
    alone = [_context(L, *s, precision) for s in specs]
    batch = L.LBBatch(members)
    batch.lb_batch_step(5)
    batch.lb_batch_step(4)
    for m, c in zip(members, alone):
        c.lb_step(9)
        assert np.array_equal(_state(m), _state(c))
    batch.close()
    for c in members + alone:
        c.close()


@pytest.mark.parametrize("rows", [1, 31, 65, 130])
@pytest.mark.parametrize("shape", [(1, 5, 3, 2), (3, 33, 4, 2), (4, 65, 3, 6), (2, 260, 3, 2)],
                         ids=lambda s: f"width{s[1]}")
def test_gradients_at_tile_edges(shape, rows):
    """A sum of k products in FP32 is off by at most k 2^-24 of the sum of their
    magnitudes: 1.6e-5 for the longest (260), over three or four layers and with
    magnitudes adding to a few times the largest gradient below 1e-4 of it."""
    import torch
    NF, W, D, NP = shape
    net = _net(shape)
    p0 = net.get_params()
    mean, std = np.array([1.0, 0.0, 0.1, 0.0], np.float32), np.array([0.5, 0.5, 0.1, 0.5], np.float32)
    net.set_output_scale(mean, std)
    x, y = _inputs(rows, 2, NP)
    net.train_step(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), 1e-3)
    _, g = grads(p0.astype(np.float64), x, y, mean, std, NF, W, D)
    assert np.abs(net.get_grads() - g).max() <= 1e-4 * np.abs(g).max()
    net.close()
