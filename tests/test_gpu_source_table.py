"""The step's gather at the sizes where it switches form: axes of 7 and 8
nodes (every node near a wall, one inside), theta shorter and longer than the
classes of the source table, odd and even x3 (the pairs of 2-byte storage),
x3 a few nodes around one warp's and two warps' worth -- with bounce-back and
equilibrium walls, x3 periodic and walled, against the FP64 oracle."""
import numpy as np
import pytest

from gpu_helpers import Twin, lib, max_rel
from oracle.geometry import Channel
from paper_1411_3133_gb300.workloads import noise_field

pytestmark = pytest.mark.gpu

SIZES = [(7, 1, 7), (8, 2, 8), (7, 6, 9), (9, 7, 31), (8, 8, 33), (7, 3, 63), (7, 4, 64), (8, 5, 66), (7, 4, 129)]
KINDS = [("cylindrical", True, "bounceback"), ("cylindrical", True, "equilibrium"), ("flat", False, "bounceback"),
         ("ellipsoidal", False, "bounceback"), ("ellipsoidal", False, "equilibrium"),
         ("ellipsoidal", True, "bounceback")]


def _twin(kind, size, precision):
    metric, periodic3, wall = kind
    ro = 1.0 if metric == "flat" else 1.05
    ch = Channel(metric, 0.0 if metric == "flat" else 1.0, ro, *size, b=0.9 if metric == "ellipsoidal" else 1.0,
                 periodic3=periodic3, wall=wall)
    params = [dict(tau=0.7, G=2e-4, seed=3, amp=1e-2), dict(tau=0.9, G=1e-4, seed=4, amp=1e-2, old=True)]
    tw = Twin(ch, params, precision)
    tw.ctx.lb_init(tw.lparams)
    for p, s in zip(params, tw.sims):
        s.init_rest(noise_field(p["seed"], tw.N, p["amp"]))
    return tw


@pytest.mark.parametrize("size", SIZES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kind", KINDS, ids=lambda k: f"{k[0]}-{'per' if k[1] else 'wall'}-{k[2]}")
def test_fp64_against_oracle(kind, size):
    """1e-12 of the largest value, as the other FP64 parity tests: 4 steps of
    arithmetic on numbers of order 1."""
    tw = _twin(kind, size, "fp64")
    tw.step(4)
    fo = np.stack([s.f for s in tw.sims])
    assert max_rel(tw.lib_f(), fo, np.abs(fo).max()) <= 1e-12
    tw.close()


@pytest.mark.parametrize("precision,eps", [("fp16_shifted", 2.0 ** -11), ("bf16_shifted", 2.0 ** -8)])
@pytest.mark.parametrize("size", SIZES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kind", KINDS, ids=lambda k: f"{k[0]}-{'per' if k[1] else 'wall'}-{k[2]}")
def test_2byte_against_oracle(kind, size, precision, eps):
    """Stored deviations g = (f - r) / w: each of the start and 3 steps rounds
    g once, by eps |g|; a step passes an error on with |1 - omega| <= 1 plus
    omega times the equilibrium's response, in all below a factor 4 (the
    largest row sum of the linearised collision at these taus is under that),
    so after 3 steps an error in g is below eps max|g| (1 + 4 + 16 + 64)."""
    tw = _twin(kind, size, precision)
    tw.step(3)
    from oracle import lattice as OL
    w = OL.W[None, :, None]
    fo = np.stack([s.f for s in tw.sims])
    rest = 1.0 / np.asarray(tw.geo["sqrtg"]).reshape(-1)[0]
    g_max = np.abs((fo - w * rest) / w).max()
    assert max_rel(tw.lib_f() / w, fo / w, 1.0) <= 85 * eps * g_max
    tw.close()


@pytest.mark.parametrize("precision,eps", [("fp16_shifted", 2.0 ** -11), ("bf16_shifted", 2.0 ** -8)])
@pytest.mark.parametrize("size", SIZES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("kind", KINDS, ids=lambda k: f"{k[0]}-{'per' if k[1] else 'wall'}-{k[2]}")
def test_2byte_step_velocity_by_velocity(kind, size, precision, eps):
    """One step from the stored state itself, deviations g = f / w - 1 from the
    rest state: every population is off by one rounding of its own g, eps |g|,
    and by the FP32 arithmetic before it, some 700 operations on numbers of
    order 1: below 1000 x 2^-24. A population from a wrong node or of the wrong
    direction is off by the noise's own g, 0.03 and more."""
    from oracle import lattice as OL
    L = lib()
    tw = _twin(kind, size, precision)
    tw.ctx.lb_set_option(L.LB_OPT_STORAGE_REFERENCE, 0)
    tw.ctx.lb_init(tw.lparams)
    for s, f in zip(tw.sims, tw.lib_f()):
        s.f = f.copy()
    tw.step(1)
    w = OL.W[None, :, None]
    g = np.stack([s.f for s in tw.sims]) / w - 1.0
    assert (np.abs(tw.lib_f() / w - 1.0 - g) <= eps * np.abs(g) + 1000 * 2.0 ** -24).all()
    tw.close()
