"""Performance cases: the passes a user of this library has it run.

A channel case advances a state by some tens of time steps and reads the
state back (as a sweep does between two samples, or before a checkpoint); a
sample case reads the observables between two such runs; a train case takes
minibatch steps of the surrogate network. Every case goes through the Python
binding (LBContext, LBBatch, LBMlp), with the options the sweeps set.

`exact` recomputes a pass in FP64 with plain torch, from the formulas of the
paper's Sec. II (equilibrium, improved forcing, BGK) and Sec. III-IV (metrics,
observables): no code of the package is used there.
"""
import math

import numpy as np
import torch

CS2 = 1.0 - math.sqrt(0.4)
PRECISION_BYTES = {"fp64": 8, "fp32": 4, "fp16_shifted": 2, "bf16_shifted": 2}
STATE_DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16_shifted": torch.float16,
               "bf16_shifted": torch.bfloat16}
FLOPS_PER_UPDATE = 700  # about what one D3Q41 collision with forcing needs


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _channel(name, metric, nr, ntheta, n3, instances, precision, steps, tau=0.55, wall="bounceback",
             periodic3=True, eta=0.975, b=1.0, ri=1.0, rescaled=False, forcing=0, speed=0.1):
    c = dict(kind="channel", metric=metric, nr=nr, ntheta=ntheta, n3=n3, instances=instances, precision=precision,
             steps=steps, tau=tau, wall=wall, periodic3=periodic3, eta=eta, b=b, ri=ri, rescaled=rescaled,
             forcing=forcing, speed=speed)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the Dean-number sweep of the narrow cylinder, 24 instances in one context (bench's default workload)
        _channel("sweep_fp32", "cylindrical", 64, 4, 256, 24, "fp32", 48),
        # the same sweep in 2-byte storage (the combined sweep)
        _channel("sweep_fp16", "cylindrical", 64, 4, 256, 24, "fp16_shifted", 80),
        # the plain FP64 sweep, which takes its instances one after another
        _channel("channel_fp64", "cylindrical", 64, 4, 256, 1, "fp64", 24),
        # 24 four-wall double-curved channels of Sec. IV.B (bench's ellipsoid workload), both storages it is run in
        _channel("fourwall_fp32", "ellipsoidal", 64, 4, 256, 24, "fp32", 48, periodic3=False, b=0.9, ri=1 / 0.81,
                 rescaled=True),
        _channel("fourwall_fp16", "ellipsoidal", 64, 4, 256, 24, "fp16_shifted", 60, periodic3=False, b=1.1,
                 ri=1 / 1.21, rescaled=True),
        # channels of mixed metric and ragged size in one lb_batch (config of the mixed surrogate's training runs
        # and of bench's mixed workload), both storages
        dict(kind="mixed", name="mixed_fp32", instances=24, precision="fp32", steps=40, n3_lo=128, n3_hi=512),
        dict(kind="mixed", name="mixed_bf16", instances=24, precision="bf16_shifted", steps=12, n3_lo=128, n3_hi=512),
        # the paper's own walls: 16 Dean numbers of the wide cylinder, one theta node (continuation runs)
        _channel("eqwall_fp32", "cylindrical", 129, 1, 256, 16, "fp32", 48, tau=0.9, wall="equilibrium", eta=0.8),
        # the theta-resolved double-curved channel over the paper's 64 theta nodes
        _channel("theta_fp32", "ellipsoidal_theta", 65, 64, 128, 2, "fp32", 20, tau=1.0, wall="equilibrium", eta=0.9,
                 b=0.8),
        # the smallest channel in use (smoke, parity): a handful of blocks, launches count
        _channel("small_fp32", "cylindrical", 16, 4, 32, 1, "fp32", 20, tau=0.8),
        # the observables and the convergence monitor between two runs of a sweep
        dict(kind="sample", name="sample_fp32", metric="cylindrical", nr=64, ntheta=4, n3=256, instances=24,
             precision="fp32", wall="bounceback", periodic3=True, eta=0.975, b=1.0, ri=1.0, rescaled=False,
             tau=0.55, forcing=0, speed=0.1),
        # four minibatch steps of the 5 x 256 surrogate, late in its learning-rate schedule
        dict(kind="train", name="train_5x256", plain=2, fourier=4, width=256, depth=5, batch=4096, batches=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel"] * 7 + ["mixed", "sample", "train"])
    if kind == "train":
        return dict(kind="train", plain=rng.choice([2, 6]), fourier=rng.randint(1, 12), width=rng.choice([64, 128, 200, 256]),
                    depth=rng.randint(3, 5), batch=_log_int(rng, 500, 16384), batches=rng.randint(1, 4))
    if kind == "mixed":
        return dict(kind="mixed", instances=rng.randint(2, 24), precision=rng.choice(["fp32", "fp16_shifted", "bf16_shifted"]),
                    steps=rng.randint(5, 20), n3_lo=rng.randint(40, 128), n3_hi=rng.randint(129, 400))
    metric = rng.choice(["cylindrical", "cylindrical", "ellipsoidal", "ellipsoidal", "flat", "ellipsoidal_theta"])
    precision = rng.choice(["fp32", "fp32", "fp16_shifted", "bf16_shifted", "fp64"])
    if metric == "ellipsoidal_theta" and precision not in ("fp32", "fp64"):
        precision = "fp32"
    wall = rng.choice(["bounceback", "bounceback", "equilibrium"])
    periodic3 = metric in ("cylindrical", "flat") or rng.random() < 0.4
    nr, ntheta, n3 = rng.randint(12, 130), rng.choice([1, 1, 3, 4, 4, 8, 16]), _log_int(rng, 24, 400)
    nodes = nr * ntheta * n3
    instances = min(24, max(1, _log_int(rng, 20_000, 1_500_000) // nodes))
    steps = max(3, min(24 if precision == "fp64" else 48, int((1e7 if precision == "fp64" else 6e7) / (nodes * instances))))
    if precision == "bf16_shifted":
        steps = min(steps, 12)
    ell = metric.startswith("ellipsoidal")
    # Sec. IV.B's rescaled spacings with bounce-back walls; the unscaled channels of Sec. IV run at tau near 1
    rescaled = ell and wall == "bounceback"
    ri, b = (1.0, 1.0) if not ell else rng.choice([(1.0, rng.uniform(0.8, 1.2)), (rng.uniform(0.8, 1.4), 1.0)])
    c = _channel(None, metric, nr, ntheta, n3, instances, precision, steps,
                 tau=round(rng.uniform(0.9 if ell and not rescaled else 0.55, 1.0), 3), wall=wall, periodic3=periodic3,
                 eta=rng.choice([0.9, 0.975] if ell else [0.8, 0.9, 0.975]), b=round(b, 3), ri=round(ri, 3),
                 rescaled=rescaled, forcing=rng.choice([0, 0, 0, 1]), speed=round(rng.uniform(0.02, 0.12), 3))
    # keep the channel's phi range (+-n3 h / 2) well inside the poles
    if ell and 0.5 * n3 / nr * (1 / c["eta"] - 1) * (1.0 if rescaled else ri) > 0.4:
        c["eta"] = round(1 / (1 + 0.8 * nr / n3 / ri), 4)
    if kind == "sample":
        c.update(kind="sample")
        c.pop("steps")
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda")


def _mixed(c, seed):
    """The channels of a mixed case: alternately a cylinder and a double-curved channel (Sec. IV.B)."""
    rng = np.random.default_rng(99)  # the sizes belong to the case, the fields to the seed
    out = []
    for i in range(c["instances"]):
        nr, n3 = int(rng.choice([32, 48, 64])), int(rng.integers(c["n3_lo"], c["n3_hi"] + 1))
        ratio = float(math.exp(rng.uniform(math.log(0.25), math.log(4.0))))
        one = dict(c, kind="channel", nr=nr, ntheta=4, n3=n3, instances=1, tau=0.55, wall="bounceback", forcing=0,
                   speed=0.08)
        if i % 2 == 0:
            one.update(metric="cylindrical", periodic3=True, eta=0.975, ri=1.0, b=1.0, rescaled=False)
        else:
            one.update(metric="ellipsoidal", periodic3=False, ri=ratio, b=1.0 / math.sqrt(ratio),
                       eta=ratio / (ratio + 1 / 40.0), rescaled=True)
        out.append((one, seed * 1000 + i))
    return out


def _geometry(c):
    """Radii, spacings and the node coordinates of a channel (Sec. III, IV, IV.B)."""
    ri = c["ri"]
    ro = ri / c["eta"]
    eq = c["wall"] == "equilibrium"
    h = (ro - ri) / (c["nr"] - 1 if eq else c["nr"])
    st, s3 = (1.0 / (c["b"] * ri), 1.0 / ri) if c["rescaled"] else (1.0, 1.0)
    f64 = dict(dtype=torch.float64, device=_device())
    r = ri + (torch.arange(c["nr"], **f64) + (0.0 if eq else 0.5)) * h
    on_walls = eq and not c["periodic3"]
    k = torch.arange(c["n3"], **f64)
    x3 = (k - 0.5 * (c["n3"] - 1) if on_walls else k + 0.5 - 0.5 * c["n3"]) * h * s3
    th = (torch.arange(c["ntheta"], **f64) + 0.5 - 0.5 * c["ntheta"]) * h * st
    return ri, ro, h, st, s3, r, th, x3


def _metric(c):
    """(g_ij physical, scaled g'_ij, h Gamma'^i_jk) at every node: (3, 3, N), (3, 3, N), {(i, j, k): (N,)}."""
    ri, ro, h, st, s3, r, th, x3 = _geometry(c)
    R, T, P = (t.reshape(-1) for t in torch.meshgrid(r, th, x3, indexing="ij"))
    g = torch.zeros(3, 3, R.numel(), dtype=torch.float64, device=R.device)
    gam = {}
    if c["metric"] == "flat":
        g[0, 0] = g[1, 1] = g[2, 2] = 1.0
    elif c["metric"] == "cylindrical":
        g[0, 0], g[1, 1], g[2, 2] = 1.0, R * R, 1.0
        gam = {(0, 1, 1): -R, (1, 0, 1): 1 / R, (1, 1, 0): 1 / R}
    else:
        # position (r cos phi cos theta, b r cos phi sin theta, r sin phi): g = J^T J
        if c["metric"] == "ellipsoidal":
            T = torch.zeros_like(T)
        b, cp, sp, ct, sn = c["b"], torch.cos(P), torch.sin(P), torch.cos(T), torch.sin(T)
        o = torch.zeros_like(R)
        J = torch.stack([torch.stack([cp * ct, -R * cp * sn, -R * sp * ct]),
                         torch.stack([b * cp * sn, b * R * cp * ct, -b * R * sp * sn]),
                         torch.stack([sp, o, R * cp])])
        g = torch.einsum("ain,ajn->ijn", J, J)
        gam = {(0, 1, 1): -R * cp * cp, (0, 2, 2): -R, (1, 0, 1): 1 / R, (1, 1, 0): 1 / R, (2, 0, 2): 1 / R,
               (2, 2, 0): 1 / R, (1, 1, 2): -sp / cp, (1, 2, 1): -sp / cp, (2, 1, 1): sp * cp}
    s = (1.0, st, s3)
    gs = torch.stack([torch.stack([g[i, j] * s[i] * s[j] for j in range(3)]) for i in range(3)])
    gam = {(i, j, k): h * v * s[j] * s[k] / s[i] for (i, j, k), v in gam.items()}
    return g, gs, gam


def _fields(c, seed):
    """Start of every instance: rho' = 1 / sqrt(g) and a developed flow -- a near-laminar streamwise profile, a pair
    of wavy Dean vortices a tenth as fast and noise -- as a warm-started run has; (rho (B, N), u (B, 3, N))."""
    B, nr, nt, n3 = c["instances"], c["nr"], c["ntheta"], c["n3"]
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    f64 = dict(dtype=torch.float64, device=dev)
    _, gs, _ = _metric(c)
    sg = torch.sqrt(torch.linalg.det(gs.permute(2, 0, 1)))
    x = ((torch.arange(nr, **f64) + 0.5) / nr).view(1, nr, 1, 1)
    t = (2 * math.pi * torch.arange(nt, **f64) / nt).view(1, 1, nt, 1)
    zf = ((torch.arange(n3, **f64) + 0.5) / n3).view(1, 1, 1, n3)
    ph = (2 * math.pi * torch.rand(B, 2, generator=gen, **f64)).view(B, 2, 1, 1, 1)
    amp = c["speed"] * (0.6 + 0.4 * torch.rand(B, generator=gen, **f64)).view(B, 1, 1, 1)
    cap = torch.ones_like(zf) if c["periodic3"] else 4 * zf * (1 - zf)
    cells = max(1, round(n3 / (2 * nr)))
    wave = 2 * math.pi * cells * zf + 0.3 * torch.cos(t + ph[:, 1])
    u = torch.empty(B, 3, nr, nt, n3, **f64)
    u[:, 0] = 0.1 * amp * torch.sin(math.pi * x) ** 2 * cap * torch.cos(wave + ph[:, 0])
    u[:, 1] = amp * 4 * x * (1 - x) * cap * (1 + 0.1 * torch.sin(math.pi * x) * torch.sin(wave + ph[:, 0]))
    u[:, 2] = -0.05 * amp * torch.sin(2 * math.pi * x) * cap * torch.sin(wave + ph[:, 0])
    u += 1e-4 * (2 * torch.rand(u.shape, generator=gen, **f64) - 1)
    rho = (1.0 / sg).expand(B, -1) * (1 + 1e-4 * (2 * torch.rand(B, nr * nt * n3, generator=gen, **f64) - 1))
    nu = (c["tau"] - 0.5) * CS2
    force = [float(8 * nu * a / nr ** 2) for a in amp.reshape(-1).tolist()]
    return rho.contiguous(), u.reshape(B, 3, -1).contiguous(), force


def _context(c, seed, stream=None):
    from paper_1411_3133_gb300 import lbgm as L
    ri, ro, h, st, s3, _, _, _ = _geometry(c)
    spec = L.ChannelSpec(c["metric"], ri, ro, c["nr"], c["ntheta"], c["n3"], b=c["b"], periodic3=c["periodic3"],
                         dtheta_scale=st, d3_scale=s3, wall=c["wall"])
    ctx = L.LBContext(spec, batch=c["instances"], precision=c["precision"], stream=stream)
    ctx.lb_set_option(L.LB_OPT_USE_GRAPH, 1)
    rho, u, force = _fields(c, seed)
    torch.cuda.synchronize()  # the fields are made on torch's stream, read on the context's
    ctx.lb_init_fields([L.make_params(c["tau"], G, c["forcing"]) for G in force], rho, u, on_device=True)
    return ctx


def _state_buffer(c):
    n = c["instances"] * 41 * c["nr"] * c["ntheta"] * c["n3"]
    return torch.empty(n, dtype=STATE_DTYPE[c["precision"]], device=_device())


def _train_data(c, seed):
    """Minibatches of (parameters, r, z) rows with smooth normalised fields, and a partly trained net's weights."""
    gen = torch.Generator().manual_seed(int(seed))
    xs, ys = [], []
    for _ in range(c["batches"]):
        x = torch.rand(c["batch"], c["plain"] + 1, generator=gen)
        r, z = x[:, -2], x[:, -1]
        d = x[:, 0]
        y = torch.stack([1 + 0.01 * r, 0.01 * d * torch.sin(3 * r) * torch.cos(2 * math.pi * z), 0.1 * r * (1 - r) * (1 + d),
                         0.01 * d * torch.cos(3 * r) * torch.sin(2 * math.pi * z)], dim=1)
        xs.append(x.float())
        ys.append(y.float())
    fan = [c["plain"] + 2 * c["fourier"]] + [c["width"]] * (c["depth"] - 1) + [4]
    params = []
    for fi, fo in zip(fan[:-1], fan[1:]):
        params += [(2 * torch.rand(fo * fi, generator=gen) - 1) * math.sqrt(6.0 / fi), 0.1 * torch.randn(fo, generator=gen)]
    return xs, ys, torch.cat(params).float(), fan


Y_MEAN, Y_STD, LEARNING_RATE = (1.0, 0.0, 0.03, 0.0), (0.01, 0.005, 0.02, 0.005), 1e-4


def prepare(case, seed):
    from paper_1411_3133_gb300 import lbgm as L
    kind = case["kind"]
    if kind == "channel":
        return dict(kind=kind, ctx=_context(case, seed), steps=case["steps"], out=_state_buffer(case))
    if kind == "mixed":
        stream = torch.cuda.Stream()
        parts = _mixed(case, seed)
        ctxs = [_context(c, s, stream) for c, s in parts]
        batch = L.LBBatch(ctxs)
        batch.lb_batch_set_option(L.LB_OPT_USE_GRAPH, 1)
        return dict(kind=kind, batch=batch, ctxs=ctxs, steps=case["steps"], out=[_state_buffer(c) for c, _ in parts])
    if kind == "sample":
        n = 3 * case["instances"] * case["nr"] * case["ntheta"] * case["n3"]
        u_prev = torch.zeros(n, dtype=torch.float64, device=_device())
        torch.cuda.synchronize()
        return dict(kind=kind, ctx=_context(case, seed), u_prev=u_prev)
    xs, ys, params, _ = _train_data(case, seed)
    net = L.LBMlp(n_fourier=case["fourier"], width=case["width"], depth=case["depth"], max_batch=case["batch"],
                  n_plain=case["plain"])
    net.set_output_scale(Y_MEAN, Y_STD)
    net.set_params(params.numpy())
    return dict(kind=kind, net=net, xs=[x.cuda() for x in xs], ys=[y.cuda() for y in ys])


def run(state):
    kind = state["kind"]
    if kind == "channel":
        state["ctx"].lb_step(state["steps"])
        return state["ctx"].lb_get_state(state["out"], on_device=True)
    if kind == "mixed":
        state["batch"].lb_batch_step(state["steps"])
        return [c.lb_get_state(o, on_device=True) for c, o in zip(state["ctxs"], state["out"])]
    if kind == "sample":
        d = state["ctx"].lb_diagnostics()
        change, umax = state["ctx"].lb_velocity_change(state["u_prev"])
        return dict({k: np.array([x[k] for x in d]) for k in OBSERVABLES}, change=change, umax=umax, u=state["u_prev"])
    n = len(state["xs"])
    for i in range(n):
        loss = state["net"].train_step(state["xs"][i], state["ys"][i], LEARNING_RATE, want_loss=i == n - 1)
    return dict(loss=loss, grads=state["net"].get_grads())


OBSERVABLES = ("mass_rho_prime", "mass_physical", "mean_v_theta", "dean", "mean_vorticity", "vortex_amp",
               "vortex_amp_x3", "max_speed", "nonfinite")


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Every time step reads and writes 41 populations per node."""
    if case["kind"] == "train":
        fan = [case["plain"] + 2 * case["fourier"]] + [case["width"]] * (case["depth"] - 1) + [4]
        products = sum(a * b for a, b in zip(fan[:-1], fan[1:]))
        first = fan[0] * fan[1]
        flops = 2.0 * case["batch"] * (3 * products - first) * case["batches"]
        row = 4.0 * (case["plain"] + 1 + 4) * case["batch"]
        return {"bytes": case["batches"] * (row + 28.0 * products), "flops": flops}
    if case["kind"] == "mixed":
        parts = [work(dict(c, steps=case["steps"])) for c, _ in _sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nodes = float(case["instances"] * case["nr"] * case["ntheta"] * case["n3"])
    s = PRECISION_BYTES[case["precision"]]
    if case["kind"] == "sample":
        return {"bytes": nodes * (41 * s + 2 * 24), "flops": nodes * 300}
    return {"bytes": case["steps"] * nodes * 82 * s, "flops": case["steps"] * nodes * FLOPS_PER_UPDATE}


def _sizes(case):
    return _mixed(case, 0)


# ---------------------------------------------------------------------------
# the same passes in FP64, from the paper's formulas
# ---------------------------------------------------------------------------
def _velocities():
    """D3Q41 of Table I, c and -c next to each other, with its weights."""
    s10 = math.sqrt(10.0)
    w = {"rest": 2 / 2025 * (5045 - 1507 * s10), "100": 37 / (5 * s10) - 91 / 40, "110": (55 - 17 * s10) / 50,
         "111": (233 * s10 - 730) / 1600, "300": (295 - 92 * s10) / 16200, "333": (130 - 41 * s10) / 129600}
    half = [((1, 0, 0), "100"), ((0, 1, 0), "100"), ((0, 0, 1), "100"), ((1, 1, 0), "110"), ((1, -1, 0), "110"),
            ((1, 0, 1), "110"), ((1, 0, -1), "110"), ((0, 1, 1), "110"), ((0, 1, -1), "110"), ((1, 1, 1), "111"),
            ((1, 1, -1), "111"), ((1, -1, 1), "111"), ((1, -1, -1), "111"), ((3, 0, 0), "300"), ((0, 3, 0), "300"),
            ((0, 0, 3), "300"), ((3, 3, 3), "333"), ((3, 3, -3), "333"), ((3, -3, 3), "333"), ((3, -3, -3), "333")]
    cs, ws = [(0, 0, 0)], [w["rest"]]
    for v, k in half:
        cs += [v, tuple(-x for x in v)]
        ws += [w[k], w[k]]
    return cs, ws


def _sources(c, cs):
    """Flat index (population * N + node) each streamed population is read from: periodic axes wrapped; bounce-back
    walls halfway outside the end nodes reverse a population's whole velocity, possibly several times in one step;
    equilibrium walls take what lies beyond them from the wall node of the line."""
    dims = (c["nr"], c["ntheta"], c["n3"])
    walled = (True, False, not c["periodic3"])
    N = dims[0] * dims[1] * dims[2]
    x = torch.meshgrid(*[torch.arange(n, device=_device()) for n in dims], indexing="ij")
    x = [t.reshape(-1) for t in x]
    out = torch.empty(len(cs), N, dtype=torch.int64, device=_device())
    for l, cv in enumerate(cs):
        if c["wall"] == "equilibrium" or l == 0:
            y = [(x[a] - cv[a]).clamp(0, dims[a] - 1) if walled[a] else (x[a] - cv[a]) % dims[a] for a in range(3)]
            out[l] = l * N + (y[0] * dims[1] + y[1]) * dims[2] + y[2]
            continue
        # walk back in half-node units along the line; |c| components are 0 or one common length
        length = max(abs(v) for v in cv)
        sign = [(v > 0) - (v < 0) for v in cv]
        pos = [2 * t for t in x]
        turn = torch.ones_like(x[0])  # +1 walking against c, -1 along it
        folds = torch.zeros_like(x[0])
        for _ in range(2 * length):
            # a half-node step that would end on a wall (odd coordinates -1, 2 n - 1) is taken, then the walk turns
            hit = torch.zeros_like(x[0], dtype=torch.bool)
            for a in range(3):
                pos[a] = pos[a] - turn * sign[a]
                if walled[a] and sign[a]:
                    hit |= (pos[a] <= -1) | (pos[a] >= 2 * dims[a] - 1)
            turn = torch.where(hit, -turn, turn)
            folds += hit
        y = [torch.div(p, 2, rounding_mode="floor") if walled[a] else torch.div(p, 2, rounding_mode="floor") % dims[a]
             for a, p in enumerate(pos)]
        pop = torch.where(folds % 2 == 1, (l - 1) // 2 * 2 + 2 - (l - 1) % 2, l)
        out[l] = pop * N + (y[0] * dims[1] + y[1]) * dims[2] + y[2]
    return out


def _equilibrium(rho, u, D, cs, ws):
    """f^eq (B, 41, N) of Sec. II for rho (B, N), u (3 of (B, N)), Delta (3, 3, N)."""
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    trD = D[0, 0] + D[1, 1] + D[2, 2]
    Du = [D[i, 0] * u[0] + D[i, 1] * u[1] + D[i, 2] * u[2] for i in range(3)]
    V = [CS2 * (trD * u[i] + 2 * Du[i]) + uu * u[i] for i in range(3)]
    e0 = 1 - (CS2 * trD + uu) / (2 * CS2)
    f = torch.empty(rho.shape[0], len(cs), rho.shape[1], dtype=rho.dtype, device=rho.device)
    for l, c in enumerate(cs):
        uc = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
        cDc = sum(c[i] * c[j] * D[i, j] for i in range(3) for j in range(3))
        Vc = c[0] * V[0] + c[1] * V[1] + c[2] * V[2]
        f[:, l] = ws[l] * rho * (e0 + uc / CS2 + cDc / (2 * CS2) + uc * uc / (2 * CS2 ** 2) + cDc * uc / (2 * CS2 ** 2)
                                 + uc ** 3 / (6 * CS2 ** 3) - Vc / (2 * CS2 ** 2))
    return f


def _moments(f, cs):
    rho = f.sum(dim=1)
    j = [torch.zeros_like(rho) for _ in range(3)]
    for l, c in enumerate(cs):
        for i in range(3):
            if c[i]:
                j[i] += c[i] * f[:, l]
    return rho, [t / rho for t in j]


def _collide(f, c, D, ginv, gam, force, tau, kappa, cs, ws, wall_node):
    """One BGK collision with the improved forcing on streamed populations f (B, 41, N)."""
    rho, u = _moments(f, cs)
    feq = _equilibrium(rho, u, D, cs, ws)
    S = {}
    for i in range(3):
        for j in range(i, 3):
            t = torch.zeros_like(rho)
            for l, cv in enumerate(cs):
                if cv[i] * cv[j]:
                    t += cv[i] * cv[j] * f[:, l]
            pi = t - rho * (CS2 * ginv[i, j] + u[i] * u[j])
            S[i, j] = S[j, i] = rho * (CS2 * D[i, j] + u[i] * u[j]) + kappa * pi
    trA = S[0, 0] + S[1, 1] + S[2, 2]
    out = torch.empty_like(f)
    for l, cv in enumerate(cs):
        F = [ginv[i, 1] * force for i in range(3)]
        for (i, j, k), g in gam.items():
            if cv[j] * cv[k]:
                F[i] = F[i] - g * (cv[j] * cv[k])
        uc = cv[0] * u[0] + cv[1] * u[1] + cv[2] * u[2]
        Fc = cv[0] * F[0] + cv[1] * F[1] + cv[2] * F[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        Ac = [cv[0] * S[i, 0] + cv[1] * S[i, 1] + cv[2] * S[i, 2] for i in range(3)]
        cAc = cv[0] * Ac[0] + cv[1] * Ac[1] + cv[2] * Ac[2]
        FAc = F[0] * Ac[0] + F[1] * Ac[1] + F[2] * Ac[2]
        # Hermite coefficients rho F, a1 F + F a1 and A2 F + ... of the forcing term, orders 1 to 3
        Fl = ws[l] * (rho * Fc / CS2 + rho * (uc * Fc / CS2 ** 2 - uF / CS2)
                      + Fc * (cAc / CS2 - trA) / (2 * CS2 ** 2) - FAc / CS2 ** 2)
        out[:, l] = f[:, l] - (f[:, l] - feq[:, l]) / tau + Fl
    if wall_node is not None:
        rest = _equilibrium(rho, [torch.zeros_like(rho)] * 3, D, cs, ws)
        out = torch.where(wall_node, rest, out)
    return out


def _wall_nodes(c):
    if c["wall"] != "equilibrium":
        return None
    m = torch.zeros(c["nr"], c["ntheta"], c["n3"], dtype=torch.bool, device=_device())
    m[0] = m[-1] = True
    if not c["periodic3"]:
        m[:, :, 0] = m[:, :, -1] = True
    return m.reshape(-1)


def _exact_channel(c, seed):
    cs, ws = _velocities()
    rho, u, force = _fields(c, seed)
    _, gs, gam = _metric(c)
    ginv = torch.linalg.inv(gs.permute(2, 0, 1)).permute(1, 2, 0)
    D = ginv - torch.eye(3, dtype=torch.float64, device=ginv.device)[:, :, None]
    force = torch.tensor(force, dtype=torch.float64, device=ginv.device)[:, None]
    kappa = 0.0 if c["forcing"] == 1 else 1 - 1 / (2 * c["tau"])
    f = _equilibrium(rho, [u[:, i] for i in range(3)], D, cs, ws)
    src, wall = _sources(c, cs).reshape(-1), _wall_nodes(c)
    B, N = rho.shape
    for _ in range(c["steps"]):
        f = f.reshape(B, -1)[:, src].reshape(B, 41, N)
        f = _collide(f, c, D, ginv, gam, force, c["tau"], kappa, cs, ws, wall)
    if PRECISION_BYTES[c["precision"]] == 2:
        # stored: the deviation from the equilibrium of the row's mean fields, over the weight
        shape = (B, -1, c["nr"], c["ntheta"], c["n3"])
        over = (3,) if c["metric"] == "ellipsoidal" else (3, 4)
        mean = torch.cat([rho[:, None], u], dim=1).reshape(shape).mean(dim=over, keepdim=True).expand(
            -1, -1, -1, c["ntheta"], c["n3"]).reshape(B, 4, N)
        r = _equilibrium(mean[:, 0].contiguous(), [mean[:, i].contiguous() for i in (1, 2, 3)], D, cs, ws)
        f = (f - r) / torch.tensor(ws, dtype=torch.float64, device=f.device)[None, :, None]
    return f.reshape(-1)


def _exact_sample(c, seed):
    cs, ws = _velocities()
    rho, u, _ = _fields(c, seed)
    g, gs, _ = _metric(c)
    ginv = torch.linalg.inv(gs.permute(2, 0, 1)).permute(1, 2, 0)
    D = ginv - torch.eye(3, dtype=torch.float64, device=ginv.device)[:, :, None]
    f = _equilibrium(rho, [u[:, i] for i in range(3)], D, cs, ws)
    B, N = rho.shape
    f = f.reshape(B, -1)[:, _sources(c, cs).reshape(-1)].reshape(B, 41, N)
    rho, v = _moments(f, cs)
    u_out = torch.stack(v, dim=1)
    w = u_out.clone()
    wall = _wall_nodes(c)
    if wall is not None:
        w[:, :, wall] = 0.0  # the wall nodes' velocity is the wall's
    shape = (B, c["nr"], c["ntheta"], c["n3"])
    cell = (c["nr"], c["ntheta"], c["n3"])
    det = torch.linalg.det(gs.permute(2, 0, 1))
    speed = torch.sqrt(gs[1, 1])
    area = torch.sqrt(g[0, 0] * g[2, 2] - g[0, 2] ** 2) if c["metric"] != "flat" else torch.ones_like(det)
    weight = torch.sqrt(g[1, 1])
    eq = c["wall"] == "equilibrium"

    def slope(a, axis, walled):
        a = a.movedim(axis, 0)
        if not walled:
            d = 0.5 * (a.roll(-1, 0) - a.roll(1, 0))
        else:
            d = torch.empty_like(a)
            d[1:-1] = 0.5 * (a[2:] - a[:-2])
            d[0] = 0.5 * (-3 * a[0] + 4 * a[1] - a[2]) if eq else a[0] + a[1] / 3
            d[-1] = 0.5 * (3 * a[-1] - 4 * a[-2] + a[-3]) if eq else -(a[-1] + a[-2] / 3)
        return d.movedim(0, axis)

    ur, uz = w[:, 0].reshape(shape), w[:, 2].reshape(shape)
    om = (slope(ur, 3, not c["periodic3"]) - slope(uz, 1, True)).abs() * weight.reshape(cell)
    fl = ur - ur.mean(dim=3, keepdim=True)
    mean_v = (speed * w[:, 1] * area).sum(dim=1) / area.sum()
    ri, ro, h, *_ = _geometry(c)
    R = ri if c["metric"] == "cylindrical" else ri * c["b"] ** 2
    nu = (c["tau"] - 0.5) * CS2
    dean = mean_v * ((ro - ri) / h) / nu * math.sqrt((ro - ri) / R) if c["metric"] != "flat" else mean_v * 0
    out = dict(mass_rho_prime=rho.sum(dim=1), mass_physical=(det * rho).sum(dim=1), mean_v_theta=mean_v, dean=dean,
               mean_vorticity=om.reshape(B, -1).sum(dim=1) / area.sum(), vortex_amp=ur.reshape(B, -1).square().mean(dim=1).sqrt(),
               vortex_amp_x3=fl.reshape(B, -1).square().mean(dim=1).sqrt(), max_speed=w.square().sum(dim=1).sqrt().amax(dim=1),
               change=u_out.abs().amax(dim=(1, 2)), umax=u_out.abs().amax(dim=(1, 2)), u=u_out.reshape(-1))
    return dict({k: v.cpu().numpy() if k != "u" else v for k, v in out.items()}, nonfinite=np.zeros(B))


def _exact_train(c, seed):
    xs, ys, params, fan = _train_data(c, seed)
    dev = _device()
    w = params.double().to(dev)
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    mean, std = (torch.tensor(t, dtype=torch.float32, device=dev).double() for t in (Y_MEAN, Y_STD))
    k = torch.arange(1, c["fourier"] + 1, device=dev, dtype=torch.float64)
    for step, (x, y) in enumerate(zip(xs, ys), 1):
        x, y = x.double().to(dev), y.double().to(dev)
        a = 2 * math.pi * x[:, -1:] * k
        h = torch.cat([x[:, :-1], torch.stack([torch.sin(a), torch.cos(a)], dim=2).flatten(1)], dim=1)
        # the products take the weights rounded to BF16; the gradient is that of the rounded weights
        leaves, at = [], 0
        for fi, fo in zip(fan[:-1], fan[1:]):
            W = w[at:at + fi * fo].float().bfloat16().double().reshape(fo, fi).requires_grad_()
            b = w[at + fi * fo:at + fi * fo + fo].clone().requires_grad_()
            at += fi * fo + fo
            leaves += [W, b]
            z = h @ W.T + b
            h = z if fo == 4 and len(leaves) == 2 * (len(fan) - 1) else z * torch.sigmoid(z)
        loss = (h - (y - mean) / std).square().mean()
        grads = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss, leaves)])
        m, v = 0.9 * m + 0.1 * grads, 0.999 * v + 0.001 * grads * grads
        w = w - LEARNING_RATE * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    return dict(loss=float(loss), grads=grads.detach().cpu().numpy())


def exact(case, seed):
    if case["kind"] == "channel":
        return _exact_channel(case, seed)
    if case["kind"] == "mixed":
        return [_exact_channel(dict(c, steps=case["steps"]), s) for c, s in _mixed(case, seed)]
    if case["kind"] == "sample":
        return _exact_sample(case, seed)
    return _exact_train(case, seed)
