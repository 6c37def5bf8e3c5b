"""The work that a user of this package has it do, as measurable cases.

Five families, each through the package's Python entry points:

* ``heat``   receding-horizon solves of the 1D / 2D nonlinear heat problems
             (``nmpc.Solver``): single instances, ragged and uniform batches,
             float32 lower layer (mixed) or float64, Jacobi or red-black;
* ``plate``  the pinned-actuator plate with input bounds (``plate.PlateSolver``);
* ``wave``   the damped nonlinear string / membrane (``wave.WaveSolver``);
* ``net_forward`` / ``net_backward``  the network of the learned warm start
             (``mlp.MLP``): controls for a batch of plant states, and the
             gradients of a training step.

A solve's case makes the problem data (initial fields, references) from the
seed, keeps the handle and the device arrays as a control program does, and
one pass solves every instance from the cold start and returns the whole
primal-dual solution with each instance's status.

``exact`` restates each family in 64-bit torch on whole arrays (the same
iteration and stopping rule; the network without any 16-bit rounding).
"""
import math
import types

import numpy as np
import torch

from paper_2004_02484_gb300 import mlp, nmpc, plate, wave

TOL = 1e-6


def listed():
    return [
        # one small string-like heat problem: the smallest call, a controller's
        # single instance (latency and launches)
        dict(name="heat1d_single", family="heat", dim=1, batch=1, mx=32, my=1, horizon=20, n_act=2,
             ragged=False, mixed=True, redblack=False, tol=TOL),
        # 1024 different 1D instances, sizes M 32..256, N 10..60, 1..4 inputs
        dict(name="heat1d_ragged_1024", family="heat", dim=1, batch=1024, mx=256, my=1, horizon=60,
             n_act=4, ragged=True, mixed=True, redblack=False, tol=TOL),
        # one 64x64 plate-like heat problem, N = 50, 8 actuators: a single
        # controller's ordinary solve
        dict(name="heat2d_64_single", family="heat", dim=2, batch=1, mx=64, my=64, horizon=50,
             n_act=8, ragged=False, mixed=True, redblack=False, tol=TOL),
        # the batch from which the learned warm start's training targets come
        dict(name="heat2d_64_batch128", family="heat", dim=2, batch=128, mx=64, my=64, horizon=50,
             n_act=8, ragged=False, mixed=True, redblack=False, tol=1e-7),
        # the largest: 64 instances of 256x256, N = 100, 16 actuators, the
        # red-black upper layer (the benchmark's first step)
        dict(name="heat2d_256_batch64", family="heat", dim=2, batch=64, mx=256, my=256, horizon=100,
             n_act=16, ragged=False, mixed=True, redblack=True, tol=TOL),
        # the default precision (everything in float64) on an odd, not square grid
        dict(name="heat2d_97x61_fp64", family="heat", dim=2, batch=4, mx=97, my=61, horizon=30,
             n_act=4, ragged=False, mixed=False, redblack=False, tol=TOL),
        # the paper's experiment: one 13x13 plate, N = 20, bounds and barrier
        dict(name="plate_single_fp64", family="plate", batch=1, m=13, horizon=20, mixed=False,
             redblack=False),
        # 1024 plates at once, default precision
        dict(name="plate_batch1024_fp64", family="plate", batch=1024, m=13, horizon=20, mixed=False,
             redblack=False),
        # second-order problems: 256 membranes of 32x32 in float64, 256
        # strings with the float32 lower layer and the red-black upper layer
        dict(name="wave_membranes256_fp64", family="wave", dim=2, batch=256, m=32, horizon=10,
             n_act=2, neumann=False, mixed=False, redblack=False),
        dict(name="wave_strings256_mixed", family="wave", dim=1, batch=256, m=64, horizon=20,
             n_act=2, neumann=False, mixed=True, redblack=True),
        # the learned start's network: the closed loop's 64 states forward, and
        # one training batch of 256 backward
        dict(name="net_forward_64", family="net_forward", batch=64, n_in=8192, hidden=512, n_out=1600),
        dict(name="net_backward_256", family="net_backward", batch=256, n_in=8192, hidden=512,
             n_out=6800),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["heat1d", "heat1d", "heat2d", "heat2d", "heat2d_fp64", "plate", "wave1d",
                       "wave2d", "net_forward", "net_backward"])
    if kind == "heat1d":
        return dict(family="heat", dim=1, batch=_log(rng, 1, 1024), mx=rng.randint(32, 256), my=1,
                    horizon=rng.randint(10, 60), n_act=rng.randint(1, 4), ragged=rng.random() < 0.5,
                    mixed=True, redblack=rng.random() < 0.3, tol=TOL)
    if kind == "heat2d":
        mx, my, n = rng.randint(24, 256), rng.randint(24, 256), rng.randint(10, 100)
        return dict(family="heat", dim=2, batch=_log(rng, 1, max(1, min(128, 50_000_000 // (mx * my * n)))),
                    mx=mx, my=my, horizon=n, n_act=rng.choice([4, 8, 16]), ragged=False, mixed=True,
                    redblack=rng.random() < 0.5, tol=TOL)
    if kind == "heat2d_fp64":
        mx, my, n = rng.randint(16, 100), rng.randint(16, 100), rng.randint(10, 50)
        return dict(family="heat", dim=2, batch=_log(rng, 1, 8), mx=mx, my=my, horizon=n, n_act=4,
                    ragged=False, mixed=False, redblack=rng.random() < 0.3, tol=TOL)
    if kind == "plate":
        return dict(family="plate", batch=_log(rng, 1, 1024), m=rng.randint(9, 15),
                    horizon=rng.randint(8, 20), mixed=rng.random() < 0.4, redblack=rng.random() < 0.5)
    if kind in ("wave1d", "wave2d"):
        dim = 1 if kind == "wave1d" else 2
        return dict(family="wave", dim=dim, batch=_log(rng, 1, 256),
                    m=rng.randint(24, 96) if dim == 1 else rng.randint(12, 32),
                    horizon=rng.randint(6, 20 if dim == 1 else 10), n_act=2,
                    neumann=rng.random() < 0.3, mixed=rng.random() < 0.5,
                    redblack=rng.random() < 0.5)
    if kind == "net_forward":
        return dict(family=kind, batch=_log(rng, 1, 256), n_in=8 * rng.randint(64, 1024),
                    hidden=64 * rng.randint(4, 8), n_out=8 * rng.randint(50, 850))
    return dict(family=kind, batch=8 * _log(rng, 2, 32), n_in=8 * rng.randint(64, 1024),
                hidden=64 * rng.randint(4, 8), n_out=8 * rng.randint(50, 850))


# ---------------------------------------------------------------------------
# Inputs, from the seed alone (plain numpy on the host, as problem data comes)
# ---------------------------------------------------------------------------
def _grid(m):
    return np.arange(1, m + 1) / (m + 1.0)


def _near(p, m):
    """Interior cell nearest to coordinate p."""
    return int(min(max(round(p * (m + 1) - 1.0), 0), m - 1))


def _sines(rng, mx, my):
    k = np.arange(1, 5)[:, None] * np.pi
    return (np.sin(k * _grid(my)).T @ (0.1 * rng.standard_normal((4, 4))) @ np.sin(k * _grid(mx))).ravel()


def _heat_instances(case, seed):
    rng = np.random.default_rng([seed, 1])
    sizes = np.random.default_rng([case["batch"], 7])  # a ragged batch's own sizes, whatever the seed
    out = []
    for _ in range(case["batch"]):
        mx, my, n, n_act, r = case["mx"], case["my"], case["horizon"], case["n_act"], 0.01
        if case["ragged"]:
            mx = int(sizes.integers(32, max(33, mx + 1)))
            n = int(sizes.integers(min(10, n), n + 1))
            n_act = int(sizes.integers(1, n_act + 1))
            r = float(10.0 ** sizes.uniform(-3.0, -1.0))
        if case["dim"] == 1:
            act = [_near((a + 0.5) / n_act, mx) for a in range(n_act)]
            x0, ref, h = rng.random(mx), 0.8 * np.sin(np.pi * _grid(mx)), 1e-4
        else:
            ny = 2 if n_act < 16 else 4
            act = [_near((b + 0.5) / ny, my) * mx + _near((a + 0.5) / (n_act // ny), mx)
                   for b in range(ny) for a in range(n_act // ny)]
            cx, cy, amp = 0.3 + 0.4 * rng.random(), 0.3 + 0.4 * rng.random(), 0.5 + rng.random()
            x0, h = _sines(rng, mx, my), 2e-5
            d2 = (_grid(mx)[None, :] - cx) ** 2 + (_grid(my)[:, None] - cy) ** 2
            ref = (amp * np.exp(-d2 / (2 * 0.15 ** 2))).ravel()
        out.append(types.SimpleNamespace(
            dim=case["dim"], mx=mx, my=my, horizon=n, h=h, act=np.asarray(act, dtype=np.int32), q=1.0,
            r=r, qf=10.0, gamma=h * r, k0=0.1, k1=0.5, act_gain=32.0, x0=x0, ref=ref))
    return out


def _plate_instances(case, seed):
    rng = np.random.default_rng([seed, 2])
    m, n = case["m"], case["horizon"]
    xs = np.linspace(0.0, 1.0, m)
    idx = [int(round(f * (m - 1))) for f in (1 / 12, 4 / 12, 8 / 12, 11 / 12)]
    act = np.asarray([iy * m + ix for iy in idx for ix in idx], dtype=np.int32)
    is_act = np.zeros(m * m, dtype=bool)
    is_act[act] = True
    rc, tz = 8960.0 * 386.0, 0.01
    cosm = np.cos(np.arange(4)[:, None] * np.pi * xs)
    out = []
    for b in range(case["batch"]):
        field = 300.0 + (cosm.T @ (10.0 * rng.standard_normal((4, 4))) @ cosm)
        prof = xs if b % 2 == 0 else np.abs(2.0 * xs - 1.0)
        ref = np.tile(350.0 + 300.0 * prof, (m, 1)).ravel()
        out.append(types.SimpleNamespace(
            dim=2, m=m, bc="neumann", horizon=n, h=5.0, act=act, k0=400.0 / rc, k1=0.0,
            beta=2.0 / (rc * tz), t_amb=300.0, gamma_r=2.0 * 0.5 * 5.67e-8 / (rc * tz), q=1.0, r=0.1,
            qf=0.0, gamma=0.5, tau=100.0, u_lo=300.0, u_hi=700.0, x0=field.ravel()[~is_act],
            x_ref=ref[~is_act], u_ref=ref[is_act]))
    return out


def _wave_instances(case, seed):
    rng = np.random.default_rng([seed, 3])
    m, n, dim = case["m"], case["horizon"], case["dim"]
    coords = np.linspace(0.0, 1.0, m) if case["neumann"] else _grid(m)
    near = [int(np.argmin(np.abs(coords - (k + 0.5) / case["n_act"]))) for k in range(case["n_act"])]
    act = near if dim == 1 else [a * m + b for a in near for b in near]
    modes = np.sin(np.arange(1, 5)[:, None] * np.pi * coords)
    out = []
    for _ in range(case["batch"]):
        if dim == 1:
            w0 = 0.1 * rng.standard_normal(4) @ modes
            ref = 0.2 * np.exp(-(coords - 0.5) ** 2 / (2 * 0.15 ** 2))
        else:
            w0 = (modes.T @ (0.1 * rng.standard_normal((4, 4))) @ modes).ravel()
            d2 = (coords[None, :] - 0.5) ** 2 + (coords[:, None] - 0.5) ** 2
            ref = (0.2 * np.exp(-d2 / (2 * 0.15 ** 2))).ravel()
        out.append(types.SimpleNamespace(
            dim=dim, m=m, bc="neumann" if case["neumann"] else "dirichlet", horizon=n, h=0.06 / 20,
            act=np.asarray(act, dtype=np.int32), a=1.0, b=1.0, c=1.0, kappa=10.0, gain=10.0, q=1.0,
            qv=0.1, r=0.01, qf=10.0, gamma=0.01 * 0.06 / 20, x0=np.concatenate([w0, np.zeros_like(w0)]),
            w_ref=ref, u_ref=np.zeros(len(act))))
    return out


def _widths(case):
    return [case["n_in"]] + 3 * [case["hidden"]] + [case["n_out"]]


def _net_inputs(case, seed):
    """Parameters (a layer's weights [out, in] then its biases), inputs, targets."""
    rng = np.random.default_rng([seed, 4])
    w, parts = _widths(case), []
    for i, o in zip(w[:-1], w[1:]):
        parts.append((2.0 * rng.random(i * o, dtype=np.float32) - 1.0) / np.float32(math.sqrt(i)))
        parts.append(0.01 * rng.standard_normal(o, dtype=np.float32))
    x = rng.standard_normal((case["batch"], w[0]), dtype=np.float32)
    t = rng.standard_normal((case["batch"], w[-1]), dtype=np.float32)
    return np.concatenate(parts), x, t


# ---------------------------------------------------------------------------
# One case
# ---------------------------------------------------------------------------
def prepare(case, seed):
    family = case["family"]
    if family in ("net_forward", "net_backward"):
        net = mlp.MLP(_widths(case), case["batch"])
        p, x, t = _net_inputs(case, seed)
        net.set_params(p)
        return dict(family=family, net=net, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda())
    opts = dict(precision=nmpc.NMPC_MIXED if case["mixed"] else nmpc.NMPC_FP64, max_iter=5000,
                variant=nmpc.NMPC_VARIANT_REDBLACK if case["redblack"] else nmpc.NMPC_VARIANT_JACOBI)
    if family == "heat":
        solver = nmpc.Solver(_heat_instances(case, seed), tol=case["tol"], **opts)
    elif family == "plate":
        solver = plate.PlateSolver(_plate_instances(case, seed), tol=TOL, **opts)
    else:
        solver = wave.WaveSolver(_wave_instances(case, seed), tol=TOL, **opts)
    return dict(family=family, solver=solver)


def run(state):
    if state["family"] == "net_forward":
        net = state["net"]
        y = torch.empty((state["x"].shape[0], net.widths[-1]), dtype=torch.float32, device="cuda")
        net.forward(state["x"], y)
        return {"y": y}
    if state["family"] == "net_backward":
        net = state["net"]
        loss = net.backward(state["x"], state["t"])
        return {"loss": np.float32(loss), "grads": net.get_grads()}
    s = state["solver"]
    _, stats = s.solve()
    x, u, lam = s.state()
    return {"x": x, "u": u, "lam": lam, "status": np.array([e.status for e in stats], dtype=np.int32)}


# Iterations that these problems take to the stopping rule, roughly: what a
# solve's arithmetic is counted with.
def _iterations(case):
    if case["family"] == "heat":
        n = 170 if case["dim"] == 1 else 140 if case["mx"] * case["my"] <= 128 * 128 else 220
    else:
        n = 110
    return n * 0.6 if case["redblack"] else n


def work(case):
    """A solve reads each instance's fields once and writes its trajectories
    once; an iteration's arithmetic is counted per grid point and stage (the
    residual, the coefficients, n_u_it + 1 = 3 lower-layer applications)."""
    family = case["family"]
    if family in ("net_forward", "net_backward"):
        w, b = _widths(case), case["batch"]
        params = sum(i * o + o for i, o in zip(w[:-1], w[1:]))
        flops = 2.0 * b * params
        if family == "net_forward":
            return {"bytes": 2.0 * params + 4.0 * b * (w[0] + w[-1]), "flops": flops}
        return {"bytes": 6.0 * params + 4.0 * b * (w[0] + w[-1]), "flops": 3.0 * flops}
    if family == "heat":
        scale = 0.35 if case["ragged"] else 1.0
        points, per = scale * case["batch"] * case["mx"] * case["my"], 170.0
        fields, traj = 2.0, 2.0
    elif family == "plate":
        points, per, fields, traj = float(case["batch"] * case["m"] ** 2), 220.0, 2.0, 2.0
    else:
        points, per, fields, traj = float(case["batch"] * case["m"] ** case["dim"]), 300.0, 3.0, 4.0
    return {"bytes": 8.0 * points * (fields + traj * case["horizon"]),
            "flops": per * points * case["horizon"] * _iterations(case)}


# ---------------------------------------------------------------------------
# 64-bit restatements
# ---------------------------------------------------------------------------
def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64,
                           device="cuda" if torch.cuda.is_available() else "cpu")


def _col(insts, name, dims):
    return _dev(np.array([float(getattr(i, name)) for i in insts])).reshape((-1,) + (1,) * dims)


def _iterate(step, S, tol, max_iter, batch):
    """Upper-layer iterations until every instance's ||K||_inf <= tol; an
    instance stays at the first iterate that passed.  step(S) gives the
    norms [batch] and the next iterate."""
    live = torch.ones(batch, dtype=torch.bool, device=S[0].device)
    status = torch.full((batch,), 3, dtype=torch.int32, device=S[0].device)
    for _ in range(max_iter + 1):
        r, new = step(S)
        done = live & (r <= tol)
        status[done] = 1
        live = live & ~done
        if not bool(live.any()):
            break
        S = tuple(torch.where(live.reshape((-1,) + (1,) * (a.dim() - 1)), b, a) for a, b in zip(S, new))
    return S, status


def _flat(t, masks):
    """Packed per instance: the entries inside each instance's own sizes."""
    return t[masks]


def _exact_heat(case, seed, n_lo=2, n_u_it=2):
    insts = _heat_instances(case, seed)
    B, N = len(insts), max(i.horizon for i in insts)
    mx, my, A = max(i.mx for i in insts), max(i.my for i in insts), max(len(i.act) for i in insts)
    h, q, r, qf, gamma, k0, k1, b0 = (_col(insts, n, 3) for n in
                                      ("h", "q", "r", "qf", "gamma", "k0", "k1", "act_gain"))
    cx = _dev([(i.mx + 1.0) ** 2 for i in insts]).reshape(B, 1, 1, 1)
    cy = _dev([(i.my + 1.0) ** 2 if i.dim == 2 else 0.0 for i in insts]).reshape(B, 1, 1, 1)
    dco = 2.0 * (cx + cy)

    def pad(name):
        f = np.zeros((B, 1, my, mx))
        for b, i in enumerate(insts):
            f[b, 0, :i.my, :i.mx] = getattr(i, name).reshape(i.my, i.mx)
        return _dev(f)

    x0, ref = pad("x0"), pad("ref")
    cell = torch.zeros((B, 1, my, mx), dtype=torch.float64, device=x0.device)
    stage = torch.zeros((B, N, 1, 1), dtype=torch.float64, device=x0.device)
    last = torch.zeros_like(stage)
    act = torch.zeros((B, A), dtype=torch.int64, device=x0.device)
    am = torch.zeros((B, 1, A), dtype=torch.float64, device=x0.device)
    for b, i in enumerate(insts):
        cell[b, 0, :i.my, :i.mx] = 1.0
        stage[b, :i.horizon] = 1.0
        last[b, i.horizon - 1] = 1.0
        act[b, :len(i.act)] = _dev(i.act // i.mx * mx + i.act % i.mx).long()
        am[b, 0, :len(i.act)] = 1.0
    on = cell * stage
    idx = act[:, None, :].expand(B, N, A)
    even = (torch.arange(N, device=x0.device) % 2 == 0).reshape(1, N, 1, 1)

    def nb(v):
        p = torch.nn.functional.pad(v, (1, 1, 1, 1))
        return cx * (p[:, :, 1:-1, :-2] + p[:, :, 1:-1, 2:]) + cy * (p[:, :, :-2, 1:-1] + p[:, :, 2:, 1:-1])

    def scatter(u):
        z = torch.zeros((B, N, my * mx), dtype=torch.float64, device=u.device)
        return z.scatter_add_(2, idx, u * am).reshape(B, N, my, mx)

    def gather(v):
        return v.reshape(B, N, my * mx).gather(2, idx) * am

    h1, r1, b1, g1 = h[..., 0], r[..., 0], b0[..., 0], gamma[..., 0]

    def rows(X, U, L, Xn, Ln):
        prev = torch.cat([x0, Xn[:, :-1]], 1)
        nxt = torch.cat([Ln[:, 1:], torch.zeros_like(Ln[:, :1])], 1)
        nxt = torch.where(last > 0, h * qf * (X - ref), nxt)
        phi = k0 * (X + 0.5 * k1 * X * X) * on
        mu = nb(L) - dco * L
        dphi = k0 * (1.0 + k1 * X)
        K1 = (prev - X + h * (nb(phi) - dco * phi + b0 * scatter(U))) * on
        K3 = (nxt - L + h * (q * (X - ref) + dphi * mu)) * on
        return K1, h1 * (r1 * U + b1 * gather(L)) * am * stage[..., 0], K3, mu, dphi

    def step(S):
        X, U, L = S
        K1, K2, K3, mu, dphi = rows(X, U, L, X, L)
        norm = torch.stack([k.abs().flatten(1).amax(1) for k in (K1, K2, K3)]).amax(0)
        dg = -1.0 - h * dco * dphi
        axx = h * (q + k0 * k1 * mu) + last * h * qf
        auu = h1 * r1 + g1

        def p_inv(b4, b5):
            v5 = b4 / dg
            for _ in range(n_lo - 1):
                v5 = (b4 - h * nb(dphi * v5 * on)) / dg
            b5 = b5 - axx * v5
            v4 = b5 / dg
            for _ in range(n_lo - 1):
                v4 = (b5 - h * dphi * nb(v4 * on)) / dg
            return v4 * on, v5 * on

        def direction(K1, K3):
            v3 = torch.zeros_like(U)
            for _ in range(n_u_it):
                y, _ = p_inv(h * b0 * scatter(v3) - K1, -K3)
                v3 = (K2 + h1 * b1 * gather(y)) / auu * am
            v4, v5 = p_inv(K1 - h * b0 * scatter(v3), K3)
            return v5, v3, v4

        dX, dU, dL = direction(K1, K3)
        if not case["redblack"]:
            return norm, (X - dX, U - dU, L - dL)
        Xe, Le = torch.where(even, X - dX, X), torch.where(even, L - dL, L)
        K1, _, K3, _, _ = rows(X, U, L, Xe, Le)
        eX, eU, eL = direction(K1, K3)
        return norm, (torch.where(even, Xe, X - eX), U - torch.where(even[..., 0], dU, eU),
                      torch.where(even, Le, L - eL))

    S = (x0 * on, torch.zeros((B, N, A), dtype=torch.float64, device=x0.device), torch.zeros_like(x0 * on))
    (X, U, L), status = _iterate(step, S, case["tol"], 5000, B)
    keep, keep_u = (on > 0).expand_as(X), ((am > 0) & (stage[..., 0] > 0)).expand_as(U)
    return {"x": _flat(X, keep), "u": _flat(U, keep_u), "lam": _flat(L, keep), "status": status}


def _lap1(m, neumann):
    L = -2.0 * np.eye(m) + np.eye(m, k=1) + np.eye(m, k=-1)
    if neumann:  # mirrored fictitious points
        L[0, 1], L[m - 1, m - 2] = 2.0, 2.0
    return L * ((m - 1.0) ** 2 if neumann else (m + 1.0) ** 2)


def _exact_plate(case, seed, n_lo=2, n_u_it=2):
    insts = _plate_instances(case, seed)
    B, N, m = len(insts), case["horizon"], case["m"]
    p = insts[0]
    L1 = _dev(_lap1(m, True))
    act = torch.as_tensor(p.act, device=L1.device).long()
    isact = torch.zeros(m * m, dtype=torch.bool, device=L1.device)
    isact[act] = True
    st = ~isact
    on = st.double().reshape(m, m)
    Ld = L1.diag()[:, None] + L1.diag()[None, :]
    lap = lambda v: L1 @ v + v @ L1.T  # noqa: E731
    lapt = lambda v: L1.T @ v + v @ L1  # noqa: E731

    def full(rows, vals, base=None):
        f = torch.zeros(rows.shape[:-1] + (m * m,), dtype=torch.float64, device=L1.device) if base is None else base
        f[..., vals] = rows
        return f

    def grid(f):
        return f.reshape(f.shape[:-1] + (m, m))

    h, k0, beta, ta, gr, tau = p.h, p.k0, p.beta, p.t_amb, p.gamma_r, p.tau
    x0 = grid(full(_dev(np.stack([i.x0 for i in insts]))[:, None], st))
    xref = grid(full(_dev(np.stack([i.x_ref for i in insts]))[:, None], st))
    uref = _dev(np.stack([i.u_ref for i in insts]))[:, None]
    even = (torch.arange(N, device=L1.device) % 2 == 0).reshape(1, N, 1, 1)

    def at(v):
        return v.flatten(-2)[..., act]

    def step(S):
        X, U, L = S  # X, L on the grid, zero at the actuator points
        W = grid(full(U, act, X.flatten(-2).clone()))
        prev = torch.cat([x0, X[:, :-1]], 1)
        nxt = torch.cat([L[:, 1:], torch.zeros_like(L[:, :1])], 1)
        ltl = lapt(L)
        K1 = (prev - X + h * (k0 * lap(W) - beta * (X - ta) - gr * (X ** 4 - ta ** 4))) * on
        K3 = (nxt - L + h * (p.q * (X - xref) + k0 * ltl - (beta + 4 * gr * X ** 3) * L)) * on
        lo, hi = U - p.u_lo, p.u_hi - U
        K2 = h * (p.r * (U - uref) - tau / lo + tau / hi + k0 * at(ltl))
        norm = torch.stack([k.abs().flatten(1).amax(1) for k in (K1, K2, K3)]).amax(0)
        dg = h * (Ld * k0 - beta - 4 * gr * X ** 3) - 1.0
        axx = h * (p.q - 12 * gr * X ** 2 * L)
        auu = h * (p.r + tau / lo ** 2 + tau / hi ** 2) + p.gamma

        def p_inv(b4, b5):
            v5 = b4 / dg * on
            for _ in range(n_lo - 1):
                v5 = (b4 - h * k0 * (lap(v5) - Ld * v5)) / dg * on
            b5 = b5 - axx * v5
            v4 = b5 / dg * on
            for _ in range(n_lo - 1):
                v4 = (b5 - h * k0 * (lapt(v4) - Ld * v4)) / dg * on
            return v4, v5

        def fu(v3):
            return h * lap(grid(full(k0 * v3, act))) * on

        def direction(K1, K3):
            v3 = torch.zeros_like(U)
            for _ in range(n_u_it):
                y, _ = p_inv(fu(v3) - K1, -K3)
                v3 = (K2 + h * k0 * at(lapt(y))) / auu
            v4, v5 = p_inv(K1 - fu(v3), K3)
            return v5, v3, v4

        dX, dU, dL = direction(K1, K3)
        if case["redblack"]:
            ex = torch.where(even, dX, torch.zeros_like(dX))
            el = torch.where(even, dL, torch.zeros_like(dL))
            K1o = K1 - torch.cat([torch.zeros_like(ex[:, :1]), ex[:, :-1]], 1)
            K3o = K3 - torch.cat([el[:, 1:], torch.zeros_like(el[:, :1])], 1)
            oX, oU, oL = direction(K1o, K3o)
            dX, dL, dU = torch.where(even, dX, oX), torch.where(even, dL, oL), torch.where(even[..., 0], dU, oU)
        # the largest step that keeps 0.5% of every bound's slack
        lim = torch.where(dU > 0, 0.995 * lo / dU, torch.where(dU < 0, -0.995 * hi / dU, torch.ones_like(dU)))
        a = lim.flatten(1).amin(1).clamp(max=1.0).reshape(B, 1, 1)
        return norm, (X - a[..., None] * dX, U - a * dU, L - a[..., None] * dL)

    X0 = x0.expand(B, N, m, m).clone()
    S = (X0, torch.full((B, N, len(p.act)), 500.0, dtype=torch.float64, device=L1.device), torch.zeros_like(X0))
    (X, U, L), status = _iterate(step, S, TOL, 5000, B)
    return {"x": X.flatten(-2)[..., st].reshape(-1), "u": U.reshape(-1),
            "lam": L.flatten(-2)[..., st].reshape(-1), "status": status}


def _exact_wave(case, seed, n_lo=2, n_u_it=2):
    insts = _wave_instances(case, seed)
    B, N, m, dim = len(insts), case["horizon"], case["m"], case["dim"]
    p, ng = insts[0], m ** dim
    L1 = _dev(_lap1(m, case["neumann"]))
    act = torch.as_tensor(p.act, device=L1.device).long()
    h, ia, kap = p.h, 1.0 / p.a, p.kappa

    def lap(v, M=L1):
        if dim == 1:
            return v @ M.T
        g = v.reshape(v.shape[:-1] + (m, m))
        return (M @ g + g @ M.T).flatten(-2)

    def lapt(v):
        return lap(v, L1.T)

    d1 = L1.diag()
    Ld = d1 if dim == 1 else (d1[:, None] + d1[None, :]).reshape(-1)
    x0 = _dev(np.stack([i.x0 for i in insts]))[:, None]
    wref = _dev(np.stack([i.w_ref for i in insts]))[:, None]
    last = torch.zeros((1, N, 1), dtype=torch.float64, device=L1.device)
    last[:, -1] = 1.0
    even = (torch.arange(N, device=L1.device) % 2 == 0).reshape(1, N, 1)

    def scatter(u):
        z = torch.zeros(u.shape[:-1] + (ng,), dtype=torch.float64, device=u.device)
        z[..., act] = u
        return z

    def step(S):
        X, U, L = S
        W, V, LW, LV = X[..., :ng], X[..., ng:], L[..., :ng], L[..., ng:]
        prev = torch.cat([x0, X[:, :-1]], 1)
        nxt = torch.cat([L[:, 1:], torch.zeros_like(L[:, :1])], 1)
        term = last * h * p.qf * (W - wref)
        g = (p.c * lap(W) - p.b * V - kap * W ** 3 + p.gain * scatter(U)) * ia
        K1 = prev - X + h * torch.cat([V, g], -1)
        K3 = nxt - L + torch.cat([term + h * (p.q * (W - wref) + (p.c * lapt(LV) - 3 * kap * W * W * LV) * ia),
                                  h * (p.qv * V + LW - p.b * ia * LV)], -1)
        K2 = h * (p.r * U + p.gain * ia * LV[..., act])
        norm = torch.stack([k.abs().flatten(1).amax(1) for k in (K1, K2, K3)]).amax(0)
        ed = -(1.0 + h * p.b * ia) + h * h * (p.c * Ld - 3 * kap * W * W) * ia
        axw = h * (p.q - 6 * kap * W * LV * ia) + last * h * p.qf
        fu, auu = h * p.gain * ia, h * p.r + p.gamma

        def sweeps(b, op):
            v = b / ed
            for _ in range(n_lo - 1):
                v = (b - h * h * p.c * ia * (op(v) - Ld * v)) / ed
            return v

        def p_inv(b4, b5):
            b6, b7 = b4[..., :ng], b4[..., ng:]
            v7 = sweeps(b7 + h * (p.c * lap(b6) - 3 * kap * W * W * b6) * ia, lap)
            v6 = h * v7 - b6
            b8, b9 = b5[..., :ng] - axw * v6, b5[..., ng:] - h * p.qv * v7
            v9 = sweeps(b9 + h * b8, lapt)
            v8 = h * (p.c * lapt(v9) - 3 * kap * W * W * v9) * ia - b8
            return torch.cat([v8, v9], -1), torch.cat([v6, v7], -1)

        def fuv(v3):
            s = fu * scatter(v3)
            return torch.cat([torch.zeros_like(s), s], -1)

        def direction(K1, K3):
            v3 = torch.zeros_like(U)
            for _ in range(n_u_it):
                y, _ = p_inv(fuv(v3) - K1, -K3)
                v3 = (K2 + fu * y[..., ng:][..., act]) / auu
            v4, v5 = p_inv(K1 - fuv(v3), K3)
            return v5, v3, v4

        dX, dU, dL = direction(K1, K3)
        if case["redblack"]:
            ex = torch.where(even, dX, torch.zeros_like(dX))
            el = torch.where(even, dL, torch.zeros_like(dL))
            oX, oU, oL = direction(K1 - torch.cat([torch.zeros_like(ex[:, :1]), ex[:, :-1]], 1),
                                   K3 - torch.cat([el[:, 1:], torch.zeros_like(el[:, :1])], 1))
            dX, dL, dU = torch.where(even, dX, oX), torch.where(even, dL, oL), torch.where(even, dU, oU)
        return norm, (X - dX, U - dU, L - dL)

    X0 = x0.expand(B, N, 2 * ng).clone()
    S = (X0, torch.zeros((B, N, len(p.act)), dtype=torch.float64, device=L1.device), torch.zeros_like(X0))
    (X, U, L), status = _iterate(step, S, TOL, 5000, B)
    return {"x": X.reshape(-1), "u": U.reshape(-1), "lam": L.reshape(-1), "status": status}


def _exact_net(case, seed):
    p, x, t = _net_inputs(case, seed)
    w, o, layers = _widths(case), 0, []
    for i, k in zip(w[:-1], w[1:]):
        layers.append((_dev(p[o:o + i * k].reshape(k, i)).requires_grad_(),
                       _dev(p[o + i * k:o + i * k + k]).requires_grad_()))
        o += i * k + k
    a = _dev(x)
    for n, (W, b) in enumerate(layers):
        a = a @ W.T + b
        if n < len(layers) - 1:
            a = torch.nn.functional.gelu(a)
    if case["family"] == "net_forward":
        return {"y": a.detach()}
    loss = ((a - _dev(t)) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grads": torch.cat([g.grad.reshape(-1) for l in layers for g in l])}


def exact(case, seed):
    family = case["family"]
    if family in ("net_forward", "net_backward"):
        return _exact_net(case, seed)
    if family == "heat":
        # about 150 whole-array operations an iteration: too long for the largest
        if case["batch"] * case["mx"] * case["my"] * case["horizon"] > 60_000_000:
            return None
        return _exact_heat(case, seed)
    return _exact_plate(case, seed) if family == "plate" else _exact_wave(case, seed)
