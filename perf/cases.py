"""The work whose speed is watched: what a program that uses this package has it do.

A case is a dict of plain values.  ``prepare`` draws its inputs on the GPU from the seed alone
(the channel, traffic and load targets of the package's own configurations, instances.py),
``run`` makes one pass through the public entry points, ``work`` says what a pass cannot do
without and ``exact`` gives the outputs in 64 bits from plain torch.

Kinds of work (the key "kind"):
  cost      path gains -> rates -> cost and the regularisation eps (build_cost_from_gains)
  solve     Algorithm 1 on a cost matrix, FP32 log domain (solve_cost), cold or warm-started
  lowp      Algorithm 1 on a stored 16-bit kernel (solve_lowp)
  f64       Algorithm 1 in FP64 (solve_f64)
  batch     many ragged instances in one planned launch (Batch.run)
  adaptive  Algorithm 2: outer steps of solve and load shift in one launch (adaptive)
  serve     time instances of resident, drifting, warm-started cells (Server)
"""
import math

import torch

from paper_1805_01559_gb300 import binding, instances

_CTX = None


def _ctx():
    """The library context: a program makes one for its device and keeps it."""
    global _CTX
    if _CTX is None:
        _CTX = binding.Context(0)
    return _CTX


# ------------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------------
def _cost(I, J):
    return {"kind": "cost", "I": I, "J": J, "eps_rel": 0.05}


def _solve(I, J, eps_rel=0.05, warm=False, padded=True, hotspot=False):
    return {"kind": "solve", "I": I, "J": J, "eps_rel": eps_rel, "tol": 1e-6, "warm": warm, "padded": padded,
            "hotspot": hotspot}


def _lowp(I, J, fmt="bf16"):
    return {"kind": "lowp", "I": I, "J": J, "eps_rel": 0.05, "tol": 1e-3, "fmt": fmt}


def listed():
    return [
        # Setting up one small cell (the 1000 x 50 configuration): launches and host time count.
        dict(_cost(1000, 50), name="cost_1000x50"),
        # Rates, cost and median of the large 4 km^2 instance, the first part of its step.
        dict(_cost(50000, 800), name="cost_50000x800"),
        # The smallest solve a controller makes: 1 km^2, 50 RRHs.
        dict(_solve(1000, 50), name="solve_1000x50"),
        # A new time instance of a small serving cell, started from the potentials of the last.
        dict(_solve(5000, 128, warm=True), name="solve_5000x128_warm"),
        # A cell of no round size, its cost as build_cost returns it (rows not 16-byte aligned).
        dict(_solve(12347, 1021, padded=False), name="solve_12347x1021_packed"),
        # The large instance of the eps sweep, hot spots and capacity targets.
        dict(_solve(50000, 800, eps_rel=0.03, hotspot=True), name="solve_50000x800"),
        # More RRHs than a warp's row holds.
        dict(_solve(100000, 1536, hotspot=True), name="solve_100000x1536"),
        # The huge instance, the kernel stored in BF16.
        dict(_lowp(400000, 4096), name="lowp_bf16_400000x4096"),
        # The small configuration in the FP64 form.
        {"kind": "f64", "I": 1000, "J": 50, "eps_rel": 0.05, "tol": 1e-6, "name": "f64_1000x50"},
        # Independent ragged cells, I from 2,000 to 60,000 and J from 64 to 1,024.
        {"kind": "batch", "n": 48, "shapes": 0, "eps_rel": 0.05, "tol": 1e-6, "name": "batch_48_ragged"},
        # Algorithm 2 on a mid-size cell.
        {"kind": "adaptive", "I": 20000, "J": 400, "outer": 10, "eps_rel": 0.1, "tol": 1e-6,
         "name": "adaptive_20000x400"},
        # One request of each of twelve resident cells whose devices have moved on.
        {"kind": "serve", "n": 12, "shapes": 0, "dt": 0.1, "eps_rel": 0.05, "tol": 1e-6, "name": "serve_12_cells"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cost", "solve", "solve", "solve", "lowp", "batch", "adaptive", "serve", "f64"])
    if kind == "cost":
        return _cost(_log_int(rng, 300, 50000), _log_int(rng, 12, 800))
    if kind == "solve":
        I = _log_int(rng, 500, 100000)
        J = _log_int(rng, 20, 1536)
        return _solve(I, J, eps_rel=math.exp(rng.uniform(math.log(0.01), math.log(0.1))), warm=rng.random() < 0.3,
                      padded=rng.random() < 0.7, hotspot=rng.random() < 0.5)
    if kind == "lowp":
        return _lowp(_log_int(rng, 10000, 400000), _log_int(rng, 300, 4096), rng.choice(["bf16", "f16"]))
    if kind == "batch":
        return {"kind": "batch", "n": _log_int(rng, 4, 48), "shapes": rng.randrange(1, 1 << 20), "eps_rel": 0.05,
                "tol": 1e-6}
    if kind == "adaptive":
        return {"kind": "adaptive", "I": _log_int(rng, 1000, 20000), "J": _log_int(rng, 20, 400),
                "outer": rng.randint(4, 10), "eps_rel": 0.1, "tol": 1e-6}
    if kind == "serve":
        return {"kind": "serve", "n": _log_int(rng, 2, 12), "shapes": rng.randrange(1, 1 << 20), "dt": 0.1,
                "eps_rel": 0.05, "tol": 1e-6}
    return {"kind": "f64", "I": _log_int(rng, 200, 1500), "J": _log_int(rng, 10, 70), "eps_rel": 0.05, "tol": 1e-6}


def _shapes(case):
    """(I, J) of a batch's instances or a server's cells; case["shapes"] picks them."""
    if case["kind"] == "batch":
        return [(I, J) for I, J, _ in instances.config3_shapes(case["n"], case["shapes"])]
    return [(min(I, 20000), J) for I, J, _ in instances.serving_cell_shapes(case["n"], case["shapes"])]


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------
_DEV = "cuda"
_ROWS = 16384  # rows drawn together


def _gen(seed, *more):
    s = seed
    for m in more:
        s = (s * 1000003 + int(m) + 1) % (1 << 62)
    return torch.Generator(device=_DEV).manual_seed(s)


def _rand(gen, *shape, dtype=torch.float64):
    return torch.rand(*shape, generator=gen, device=_DEV, dtype=dtype)


def _randn(gen, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=gen, device=_DEV, dtype=dtype)


def _layout(gen, I, J, side, hotspot):
    """Device and RRH positions: RRHs on a jittered grid, devices uniform or 40% in 5 hot spots."""
    r = max(1, math.isqrt(J))
    c = -(-J // r)
    k = torch.arange(J, device=_DEV)
    jit = 0.5 * _rand(gen, J, 2) - 0.25
    rrh = torch.stack([(k % c + 0.5 + jit[:, 0]) * (side / c), (k // c + 0.5 + jit[:, 1]) * (side / r)], dim=1)
    dev = side * _rand(gen, I, 2)
    if hotspot:
        n = int(round(0.4 * I))
        centre = side * _rand(gen, 5, 2)
        which = (_rand(gen, n) * 5).long().clamp_(max=4)
        spot = centre[which] + 0.05 * side * _randn(gen, n, 2, dtype=torch.float64)
        spot = torch.remainder(spot, 2 * side)  # back inside by reflection
        spot = torch.where(spot > side, 2 * side - spot, spot)
        dev = torch.cat([spot, dev[n:]])[torch.randperm(I, generator=gen, device=_DEV)]
    return dev, rrh


def _path_gains(dev, rrh, shadow):
    """Linear gains of the path-loss model, in the type of `shadow` (dB)."""
    dev, rrh = dev.to(shadow.dtype), rrh.to(shadow.dtype)
    dx = dev[:, None, 0] - rrh[None, :, 0]
    dy = dev[:, None, 1] - rrh[None, :, 1]
    d2 = (dx * dx + dy * dy).clamp_(min=instances.D_MIN_M ** 2)
    db = d2.log10_().mul_(5.0 * instances.PL_EXPONENT).add_(shadow).add_(instances.PL0_DB)
    return torch.pow(10.0, db.mul_(-0.1))


def _cost_of(G):
    """C = 1/(mu R) from gains at unit power: R = W log2(1 + SINR), every other RRH interfering."""
    own = G.double()
    interf = own.sum(dim=1, keepdim=True) + instances.noise_power_w() - own
    sinr = own / interf if G.dtype == torch.float64 else G / interf.float()
    return math.log(2.0) / (instances.MU_PER_BIT * instances.W_HZ * torch.log1p(sinr))


def _traffic(gen, I, sigma):
    lam = torch.exp(sigma * _randn(gen, I, dtype=torch.float64))
    return (lam / lam.sum()).float()


def _target(gen, J, capacity):
    kappa = 0.5 + _rand(gen, J) if capacity else torch.ones(J, device=_DEV, dtype=torch.float64)
    return (kappa / kappa.sum()).float()


def _padded(I, J, pad):
    return torch.empty((I, -(-J // 4) * 4 if pad else J), dtype=torch.float32, device=_DEV)[:, :J]


def _instance(seed, I, J, eps_rel, hotspot=False, padded=True, dt=None):
    """C, p, q, eps of one instance (and with dt the cost of the same devices dt earlier)."""
    gen = _gen(seed, I, J)
    side = 1000.0 * (1 if J < 300 else 2 if J < 1100 else 4)
    dev, rrh = _layout(gen, I, J, side, hotspot)
    p, q = _traffic(gen, I, 1.5 if hotspot else 1.0), _target(gen, J, hotspot)
    C, before = _padded(I, J, padded), None if dt is None else _padded(I, J, True)
    step = 10.0 * dt * _randn(gen, I, 2, dtype=torch.float64) if dt is not None else None
    for a in range(0, I, _ROWS):
        b = min(I, a + _ROWS)
        shadow = _randn(gen, b - a, J) * instances.SHADOW_DB
        C[a:b] = _cost_of(_path_gains(dev[a:b], rrh, shadow))
        if dt is not None:
            before[a:b] = _cost_of(_path_gains(dev[a:b] + step[a:b], rrh, shadow))
    eps = eps_rel * C[: min(I, 4096)].median().item()
    return C, p, q, eps, before


def _cells(case, seed):
    """Positions, velocities, shadowing, traffic and targets of a server's drifting cells."""
    out = []
    for n, (I, J) in enumerate(_shapes(case)):
        gen = _gen(seed, n, I, J)
        side = 1000.0
        dev, rrh = _layout(gen, I, J, side, False)
        speed, way = 1.0 + 29.0 * _rand(gen, I), 2.0 * math.pi * _rand(gen, I)
        vel = torch.stack([speed * torch.cos(way), speed * torch.sin(way)], dim=1)
        shadow = _randn(gen, I, J) * instances.SHADOW_DB
        rows = min(I, 2048)
        eps = case["eps_rel"] * _cost_of(_path_gains(dev[:rows], rrh, shadow[:rows])).median().item()
        out.append({"I": I, "J": J, "side": side, "dev": dev, "rrh": rrh.float(), "vel": vel, "shadow": shadow,
                    "p": _traffic(gen, I, 1.0), "q": _target(gen, J, False), "eps": eps})
    return out


def prepare(case, seed):
    kind = case["kind"]
    ctx = _ctx()
    s = {"kind": kind, "ctx": ctx, "case": case}
    if kind == "cost":
        gen = _gen(seed, case["I"], case["J"])
        dev, rrh = _layout(gen, case["I"], case["J"], 1000.0 if case["J"] < 300 else 2000.0, False)
        s["G"] = _path_gains(dev, rrh, _randn(gen, case["I"], case["J"]) * instances.SHADOW_DB)
        s["P"] = torch.full((case["J"],), instances.P_TX_W, device=_DEV)
    elif kind == "solve":
        s["C"], s["p"], s["q"], s["eps"], before = _instance(seed, case["I"], case["J"], case["eps_rel"],
                                                             case["hotspot"], case["padded"],
                                                             0.1 if case["warm"] else None)
        if case["warm"]:  # the potentials of the time instance before
            s["g0"] = _sinkhorn64(before, s["p"], s["q"], s["eps"], case["tol"])[1]
            s["g"] = torch.empty_like(s["g0"])
    elif kind == "lowp":
        s["C"], s["p"], s["q"], s["eps"], _ = _instance(seed, case["I"], case["J"], case["eps_rel"], True)
        s["fmt"] = binding.OT_KERNEL_BF16 if case["fmt"] == "bf16" else binding.OT_KERNEL_F16
    elif kind == "f64":
        C, p, q, s["eps"], _ = _instance(seed, case["I"], case["J"], case["eps_rel"], False, False)
        s["C"], s["p"], s["q"] = C.double(), p.double() / p.double().sum(), q.double() / q.double().sum()
    elif kind == "adaptive":
        s["C"], s["p"], _, s["eps"], _ = _instance(seed, case["I"], case["J"], case["eps_rel"])
        s["delta"] = 0.05 / case["J"]
    elif kind == "batch":
        # the potentials and loads of the instances lie in one tensor each
        shapes = _shapes(case)
        nI, nJ = sum(I for I, _ in shapes), sum(J for _, J in shapes)
        f, g, rho = (torch.zeros(n, dtype=torch.float64, device=_DEV) for n in (nI, nJ, nJ))
        inst, a, b = [], 0, 0
        for n, (I, J) in enumerate(shapes):
            C, p, q, eps, _ = _instance(seed * 1009 + n, I, J, case["eps_rel"])
            inst.append(binding.Instance(C=C, p=p, q=q, eps=eps, tol=case["tol"], f=f[a:a + I], g=g[b:b + J],
                                         rrh_load=rho[b:b + J]))
            a, b = a + I, b + J
        s["f"], s["g"], s["rho"], s["batch"] = f, g, rho, ctx.batch(inst)
    elif kind == "serve":
        s["server"] = ctx.server(max_J=1024)
        s["ids"] = []
        for c in _cells(case, seed):
            ones = torch.full((c["J"],), instances.P_TX_W)
            cid = s["server"].add_cell(c["I"], c["J"], c["eps"], ones.numpy(), c["p"].cpu().numpy(),
                                       c["q"].cpu().numpy(), instances.MU_PER_BIT, instances.noise_power_w(),
                                       instances.W_HZ, tol=case["tol"], dev_xy=c["dev"].cpu().numpy(),
                                       dev_v=c["vel"].cpu().numpy(), rrh_xy=c["rrh"].cpu().numpy(),
                                       shadow_db=c["shadow"].cpu().numpy(), side_m=c["side"])
            s["ids"].append((cid, c["I"], c["J"]))
    return s


def run(s):
    kind, ctx, case = s["kind"], s["ctx"], s["case"]
    if kind == "cost":
        return ctx.build_cost_from_gains(s["G"], s["P"], instances.noise_power_w(), instances.W_HZ,
                                         instances.MU_PER_BIT, eps_rel=case["eps_rel"])
    if kind == "solve":
        if case["warm"]:
            r = ctx.solve_cost(s["C"], s["p"], s["q"], s["eps"], tol=case["tol"], warm_g=s["g0"], g=s["g"])
        else:
            r = ctx.solve_cost(s["C"], s["p"], s["q"], s["eps"], tol=case["tol"])
        return r.f, r.g, r.rrh_load, r.transport_cost
    if kind == "lowp":
        r = ctx.solve_lowp(s["C"], s["p"], s["q"], s["eps"], tol=case["tol"], fmt=s["fmt"])
        return r.f, r.g, r.rrh_load, r.transport_cost
    if kind == "f64":
        r = ctx.solve_f64(s["C"], s["p"], s["q"], s["eps"], tol=case["tol"])
        return r.f, r.g, r.rrh_load, r.transport_cost
    if kind == "adaptive":
        r = ctx.adaptive(s["C"], s["p"], s["eps"], s["delta"], case["outer"], tol=case["tol"])
        return r.f, r.g, r.q, r.rrh_load
    if kind == "batch":
        res = s["batch"].run()
        return s["f"], s["g"], s["rho"], sum(r.transport_cost for r in res)
    server = s["server"]
    for cid, _, _ in s["ids"]:
        server.submit(cid, dt=case["dt"])
    server.drain()
    return [server.cell_state(cid, I, J) for cid, I, J in s["ids"]]


# ------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _sweeps(case):
    """Iterations these instances take, by the regularisation and the start."""
    n = 17.0 * (0.1 / case["eps_rel"]) ** 0.38 if case["tol"] < 1e-4 else 9.0
    return 0.5 * n if case.get("warm") or case["kind"] == "serve" else n


def work(case):
    """Each input read once and each output written once; per cell and iteration an exponent
    (4 operations), the exponential, a row and a column sum (6 flops more with the update)."""
    kind = case["kind"]
    if kind == "cost":
        n = case["I"] * case["J"]
        return {"bytes": 8 * n, "flops": 12 * n}
    if kind in ("batch", "serve"):
        n = sum(I * J for I, J in _shapes(case))
        ends = sum(12 * I + 20 * J for I, J in _shapes(case))
        per = 4 if kind == "batch" else 8
    else:
        n = case["I"] * case["J"]
        ends = 12 * case["I"] + 20 * case["J"]
        per = 8 if kind == "f64" else 4
    its = _sweeps(case) * (0.45 * case["outer"] if kind == "adaptive" else 1.0)
    return {"bytes": per * n + ends, "flops": 10 * n * its}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits, by plain torch
# ------------------------------------------------------------------------------------------------
def _sinkhorn64(C, p, q, eps, tol, max_iter=2000, g0=None):
    """Algorithm 1: a-update then b-update until the row residual of the plan is at most
    tol (1 - 2^-5), the margin below tol at which the solvers stop.  (f, g, loads, cost)."""
    I, J = C.shape
    mass = p.double().sum()
    p, q = p.double() / mass, q.double() / q.double().sum()
    g = torch.zeros(J, dtype=torch.float64, device=_DEV) if g0 is None else g0.double()
    f = torch.empty(I, dtype=torch.float64, device=_DEV)
    T = torch.empty((I, J), dtype=torch.float64, device=_DEV)  # pi_ij / p_i after the first iteration
    top = torch.full((J,), -math.inf, dtype=torch.float64, device=_DEV)
    for a in range(0, I, _ROWS):
        x = (g - C[a:a + _ROWS].double()) / eps
        f[a:a + _ROWS] = eps * (torch.log(p[a:a + _ROWS]) - torch.logsumexp(x, dim=1))
        T[a:a + _ROWS] = x + f[a:a + _ROWS, None] / eps
        top = torch.maximum(top, T[a:a + _ROWS].amax(dim=0))
    col = torch.zeros(J, dtype=torch.float64, device=_DEV)
    for a in range(0, I, _ROWS):
        col += torch.exp(T[a:a + _ROWS] - top).sum(dim=0)
    dg = torch.log(q) - torch.log(col) - top
    g = g + eps * dg
    for a in range(0, I, _ROWS):
        T[a:a + _ROWS] = torch.exp(T[a:a + _ROWS] + dg - torch.log(p[a:a + _ROWS])[:, None])
    u, v = torch.ones_like(f), torch.ones_like(g)
    for k in range(1, max_iter + 1):
        Tv = T @ v
        if k == max_iter or (p * (u * Tv - 1).abs()).sum().item() <= tol * (1 - 2.0 ** -5):
            break
        u = 1 / Tv
        v = q / (T.t() @ (p * u))
    w = p * u
    rho = torch.zeros(J, dtype=torch.float64, device=_DEV)
    for a in range(0, I, _ROWS):
        rho += (C[a:a + _ROWS].double() * T[a:a + _ROWS]).t() @ w[a:a + _ROWS]
    rho = mass * rho * v
    return f + eps * (torch.log(u) + torch.log(mass)), g + eps * torch.log(v), rho, rho.sum().item()


def _exact_adaptive(s, case):
    q = s["p"].double().sum() / case["J"] * torch.ones(case["J"], dtype=torch.float64, device=_DEV)
    g = None
    for k in range(case["outer"]):
        f, g, rho, _ = _sinkhorn64(s["C"], s["p"], q.float(), s["eps"], case["tol"], g0=g)
        if k + 1 < case["outer"]:
            j = int(rho.argmax())
            d = s["delta"] if s["delta"] < q[j].item() else 0.5 * q[j].item()
            move = torch.full_like(q, d / (case["J"] - 1))
            move[j] = -d
            q = q + move
    return f, g, q, rho


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for c in _cells(case, seed):
            x = torch.remainder(c["dev"] + c["vel"] * case["dt"], 2 * c["side"])
            x = torch.where(x > c["side"], 2 * c["side"] - x, x)
            C = _cost_of(_path_gains(x, c["rrh"].double(), c["shadow"].double()))
            out.append((C,) + _sinkhorn64(C, c["p"], c["q"], c["eps"], case["tol"])[:3])
        return out
    if kind == "batch":
        parts = []
        for n, (I, J) in enumerate(_shapes(case)):
            C, p, q, eps, _ = _instance(seed * 1009 + n, I, J, case["eps_rel"])
            parts.append(_sinkhorn64(C, p, q, eps, case["tol"]))
        return tuple(torch.cat([x[k] for x in parts]) for k in range(3)) + (sum(x[3] for x in parts),)
    s = prepare(case, seed)
    if kind == "cost":
        C = _cost_of(s["G"].double())
        x = C.reshape(-1).sort().values
        return C, case["eps_rel"] * 0.5 * (x[(x.numel() - 1) // 2] + x[x.numel() // 2]).item()
    if kind == "adaptive":
        return _exact_adaptive(s, case)
    return _sinkhorn64(s["C"], s["p"], s["q"], s["eps"], case["tol"], g0=s.get("g0"))
