"""Observables of fields that hold an infinity or a NaN: what the sums over the
nodes give, and nothing of it in the other instances."""
import numpy as np
import pytest

from gpu_helpers import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr,ntheta,n3", [(7, 2, 5), (9, 3, 70)])
@pytest.mark.parametrize("node", [0.02, 0.5])  # before and after the other rows of its warp
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan], ids=str)
@pytest.mark.parametrize("component", [0, 1, 2])
def test_vortex_amplitudes_and_speed(nr, ntheta, n3, node, bad, component):
    """vortex_amp is the rms of u^r (an infinity gives infinity, a NaN NaN),
    vortex_amp_x3 that of u^r less its row mean (NaN with either), max_speed
    leaves NaN out. Finite ones to 1e-12: sums of some thousand terms."""
    import torch
    L = lib()
    n = nr * ntheta * n3
    rng = np.random.default_rng(5)
    rho = 1.0 + 0.01 * rng.standard_normal((3, n))
    u = 0.1 * rng.standard_normal((3, 3, n))
    u[1, component, int(node * n)] = bad
    desc = L.make_desc(1.0, 1.1, nr, ntheta, n3)
    got = L.lb_diagnostics_noalloc("cylindrical", desc, [0.8] * 3, torch.from_numpy(rho).cuda(),
                                   torch.from_numpy(u).cuda())
    rows = u[:, 0].reshape(3, nr * ntheta, n3)
    with np.errstate(invalid="ignore"):
        amp = np.sqrt((rows ** 2).reshape(3, -1).mean(axis=1))
        x3 = np.sqrt(((rows - rows.mean(axis=2, keepdims=True)) ** 2).reshape(3, -1).mean(axis=1))
        speed = np.sqrt(np.nanmax((u ** 2).sum(axis=1), axis=1))
    for b in range(3):
        assert got[b]["vortex_amp"] == pytest.approx(amp[b], rel=1e-12, nan_ok=True)
        assert got[b]["vortex_amp_x3"] == pytest.approx(x3[b], rel=1e-12, nan_ok=True)
        assert got[b]["max_speed"] == pytest.approx(speed[b], rel=1e-12)
        assert got[b]["nonfinite"] == (b == 1)
