"""The work that a user of this framework has it do, as cases to be timed.

`listed()` gives the cases, `draw(rng)` more of the same ranges, `prepare` what a
program holds before the call, `run` one pass through the public entry points,
`work` what a pass cannot do without and `exact` its outputs in 64 bits, from
plain torch and numpy.  Grids, swarms and records are those of the workloads in
synth.workloads(), of the benchmark and of the run file in tests/golden.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1905_12795_gb300 import binding as B
from paper_1905_12795_gb300 import synth

DEV = "cuda"

# centred weights c_0 .. c_R of the second derivative by space order
WEIGHTS = {
    2: (-2.0, 1.0),
    4: (-5 / 2, 4 / 3, -1 / 12),
    8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560),
    16: (-1077749 / 352800, 16 / 9, -14 / 45, 112 / 1485, -7 / 396, 112 / 32175, -2 / 3861,
         16 / 315315, -1 / 411840),
}


def listed():
    plain = dict(nx=461, nz=151, hx=20.0, hz=20.0, pad=40, order=8, T=3.0, f0=6.0, dt=0.0, vmin=1500.0,
                 vmax=4700.0, depth=20.0, kx=8, kz=4, mode=0)
    small = dict(nx=101, nz=101, hx=10.0, hz=10.0, pad=20, order=4, T=0.5, f0=10.0, dt=0.0, depth=20.0,
                 kx=8, kz=4, mode=0)
    fine = dict(nx=921, nz=301, hx=10.0, hz=10.0, pad=60, vmin=1500.0, vmax=4700.0, depth=20.0, dt=0.0,
                kx=8, kz=4, mode=0)
    return [
        # one shot of one model: a single modelling call, the smallest there is
        dict(small, name="model-101x101-one-shot", kind="models", vmin=1500.0, vmax=2625.0, M=1, S=1),
        # a whole swarm on the small grid: what a generation of the surrogate search models at first
        dict(small, name="swarm-101x101-P1024", kind="fitness", vmin=1200.0, vmax=3200.0, M=1024, S=1),
        # the plain search's generation, 32 particles by 16 shots
        dict(plain, name="swarm-461x151-P32-S16", kind="fitness", M=32, S=16),
        # one particle of the paper's own run file: anisotropic spacing, given time step, its level-wise
        # control grid under a water layer, 50 shots with sources and receivers at the surface
        dict(name="particle-369x375-levels-S50", kind="fitness", nx=369, nz=375, hx=25.0, hz=8.0, pad=40,
             order=8, T=4.0, f0=3.0, dt=0.00061, vmin=1500.0, vmax=4700.0, depth=0.0, kx=8, kz=4, mode=2,
             M=1, S=50),
        # a generation over two resolutions in one launch (half resolution, half frequency, longer record)
        dict(plain, name="swarm-two-grids-P16-S16x2", kind="uneven", M=16, S=16),
        # observed data on the fine grid, 17 Hz, before they are low-passed for the coarse inversion
        dict(fine, name="traces-921x301-S16", kind="traces", order=8, T=3.0, f0=17.0, M=1, S=16),
        # observed data of one band of the local inversion: its 16th-order operator on its fine grid
        dict(fine, name="traces-921x301-order16-S16", kind="traces", order=16, T=2.0, f0=4.6 / 2.5, M=1, S=16),
        # the local inversion's gradient: on the plain grid, and order 16 on the fine one
        dict(plain, name="gradient-461x151-S16", kind="gradient", M=1, S=16),
        dict(fine, name="gradient-921x301-order16-S4", kind="gradient", order=16, T=3.0, f0=11.5 / 2.5, M=1, S=4),
        # a generation's work of the surrogate: predict the swarm, six training steps of 1024
        dict(name="surrogate-K32-H256", kind="surrogate", P=1024, K=32, H=256, steps=6, batch=1024, pairs=6144,
             recent=4096),
        # one step of the swarm with its elitist mutation, and its new state
        dict(name="step-P1024-D32", kind="step", P=1024, K=32),
        # observed data low-passed below 6 Hz and moved from the fine grid's steps to the plain grid's
        dict(name="lowpass-S16-R461", kind="lowpass", S=16, nrec=461, nt_in=2826, nt_out=1414, T=3.0, fcut=6.0,
             half=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("models", "fitness", "fitness", "uneven", "traces", "traces", "gradient", "gradient",
                       "surrogate", "step", "lowpass"))
    if kind == "surrogate":
        P = rng.randint(200, 1024)
        return dict(kind=kind, P=P, K=rng.choice((8, 32, 45, 64, 142, 192)), H=rng.choice((64, 128, 192, 256)),
                    steps=rng.randint(1, 6), batch=_log(rng, 64, 1024), pairs=_log(rng, 1000, 6144),
                    recent=rng.choice((0, 1000, 4096)))
    if kind == "step":
        return dict(kind=kind, P=_log(rng, 16, 2048), K=_log(rng, 6, 192))
    if kind == "lowpass":
        nt_in = _log(rng, 400, 2826)
        return dict(kind=kind, S=_log(rng, 1, 16), nrec=_log(rng, 40, 461), nt_in=nt_in,
                    nt_out=int(nt_in / rng.uniform(1.0, 4.0)), T=rng.choice((1.0, 2.0, 3.0)),
                    fcut=rng.uniform(4.0, 12.0), half=rng.uniform(0.2, 0.5))
    # a modelling grid: sides over their logarithm, the record by its number of steps
    order = rng.choice((8, 8, 4, 2) if kind in ("models", "fitness", "uneven") else (8, 16, 16, 4))
    big = kind in ("traces", "gradient")
    nx, nz = _log(rng, 61, 921 if big else 461), _log(rng, 41, 301 if big else 231)
    if kind == "uneven":
        nx, nz = nx | 1, nz | 1
    h = rng.choice((8.0, 10.0, 12.5, 20.0, 25.0))
    c = dict(kind=kind, nx=nx, nz=nz, hx=h, hz=h, pad=rng.randint(10, 60 if big else 40), order=order, T=1.0,
             f0=1500.0 / (h * rng.uniform(10.0, 16.0)), dt=0.0, vmin=1500.0,
             vmax=rng.choice((2625.0, 3200.0, 4700.0)), depth=2 * h, kx=rng.randint(4, 12), kz=rng.randint(3, 8),
             mode=rng.choice((0, 0, 1, 2)) if kind == "fitness" else 0)
    c["T"] = round((_log(rng, 240, 1500) - 1.5) * _dt_rule(c), 6)
    points = (nx + 2 * c["pad"]) * (nz + 2 * c["pad"])
    nt = _axis(c)[1]
    if kind == "models":
        c.update(M=_log(rng, 1, 8), S=_log(rng, 1, 16))
    elif kind == "traces":
        c.update(M=1, S=_log(rng, 1, 16))
    elif kind == "gradient":
        c.update(M=1, S=_log(rng, 1, 16))
    else:
        c.update(M=_log(rng, 2, 256), S=_log(rng, 1, 16))
    # no more than 2e10 updates (a third of that on two grids, a tenth in a gradient's history)
    most = {"uneven": 1.2e10, "gradient": 2e9}.get(kind, 2e10)
    while c["M"] * c["S"] * points * nt > most and c["M"] * c["S"] > 1:
        k = "M" if c["M"] >= c["S"] else "S"
        c[k] = max(1, c[k] * 2 // 3)
    return c


# ---- geometry and inputs ---------------------------------------------------------------------------


def _dt_rule(c):
    """0.9 of the stability limit of the scheme."""
    w = WEIGHTS[c["order"]]
    rho = abs(w[0] + sum(2 * (-x if m & 1 else x) for m, x in enumerate(w) if m))
    return 0.9 * 2.0 / (c["vmax"] * math.sqrt(rho * (1 / c["hx"] ** 2 + 1 / c["hz"] ** 2)))


def _f32(x):
    return float(np.float32(x))


def _axis(c):
    """(dt, nt): dt as the 32-bit number that a grid holds."""
    T = _f32(c["T"])
    if c["dt"] > 0:
        return _f32(c["dt"]), int(round(T / _f32(c["dt"]))) + 1
    q = dict(c, vmax=_f32(c["vmax"]), hx=_f32(c["hx"]), hz=_f32(c["hz"]))
    nt = int(math.ceil(T / _dt_rule(q))) + 1
    return _f32(T / (nt - 1)), nt


def _half(c):
    """The second grid of a two-resolution generation: half of everything, a third longer record."""
    return dict(c, nx=(c["nx"] - 1) // 2 + 1, nz=(c["nz"] - 1) // 2 + 1, hx=2 * c["hx"], hz=2 * c["hz"],
                pad=c["pad"] // 2, f0=c["f0"] / 2, T=c["T"] * 4 / 3)


def _grids(c):
    return [_half(c), c] if c["kind"] == "uneven" else [c]


def _shots(c):
    """Source positions, and one receiver for each horizontal node."""
    return (synth.shot_line(c["S"], (c["nx"] - 1) * c["hx"], c["depth"]).astype(np.float32).astype(np.float64),
            synth.receiver_line(c["nx"], c["hx"], c["depth"]).astype(np.float32).astype(np.float64))


def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + k)
    return g


def _rand(seed, k, *shape, dtype=torch.float32):
    return torch.rand(*shape, generator=_gen(seed, k), device=DEV, dtype=dtype)


def _observed(c, seed):
    """Recorded traces [S][nt][nrec]: the direct wave and three reflections, as hyperbolas of Ricker
    wavelets with the amplitudes of a line source, and a little noise."""
    dt, nt = _axis(c)
    shots, rec = _shots(c)
    r = _rand(seed, 7, 3, 2, dtype=torch.float64).cpu().numpy()
    x = torch.tensor(rec[None, :, 0] - shots[:, :1], device=DEV, dtype=torch.float32)
    t = (torch.arange(1, nt + 1, device=DEV, dtype=torch.float32) * dt)[None, :, None]
    out = 0.01 * (_rand(seed, 8, c["S"], nt, len(rec)) - 0.5)
    top = 0.5 * (c["nz"] - 1) * c["hz"] / 1500.0
    for k in range(4):
        v = c["vmin"] if k == 0 else c["vmin"] + (c["vmax"] - c["vmin"]) * (0.3 + 0.5 * r[k - 1][0])
        t0 = 0.0 if k == 0 else (k + 0.5 * r[k - 1][1]) * top / 2
        arr = torch.sqrt(t0 * t0 + (x / v) ** 2)
        amp = (1.0 if k == 0 else 0.3 / k) * 0.2 / torch.sqrt(1 + 2 * math.pi * c["f0"] * arr)
        a = (math.pi * c["f0"] * (t - arr[:, None, :] - 1.0 / c["f0"])) ** 2
        out += amp[:, None, :] * (1 - 2 * a) * torch.exp(-a)
    return out.contiguous()


def _velocity(c, seed):
    """A model such as the search hands to the inversion: velocity growing with depth, smooth blocks on it."""
    z = torch.linspace(0, 1, c["nz"], device=DEV)[:, None]
    base = c["vmin"] + (0.85 * c["vmax"] - c["vmin"]) * z
    low = _rand(seed, 3, c["M"], 1, 5, 9) - 0.5
    bump = F.interpolate(low, size=(c["nz"], c["nx"]), mode="bilinear", align_corners=True)[:, 0]
    return (base + 0.5 * (c["vmax"] - c["vmin"]) * bump).clamp(c["vmin"], c["vmax"]).contiguous()


def _levels(c):
    """The level-wise control grid: depths, node counts, node positions, velocity of the 1-D model at each."""
    Lx, Lz = (c["nx"] - 1) * c["hx"], (c["nz"] - 1) * c["hz"]
    z, n, x, v1d = synth.level_layout(Lx, Lz, 4 * c["hz"], 1500.0, 0.75 * c["vmax"], c["f0"], 0.4)
    x, z = x.astype(np.float32), z.astype(np.float32)
    return np.minimum(z, np.float32(Lz)), n, np.minimum(x, np.float32(Lx)), np.repeat(v1d(z), n)


def _particles(c, seed):
    if c["mode"] != 2:
        return c["vmin"] + (c["vmax"] - c["vmin"]) * _rand(seed, 4, c["M"], c["kx"] * c["kz"])
    v = torch.tensor(_levels(c)[3], device=DEV, dtype=torch.float32)
    return (v * (0.75 + 0.6 * _rand(seed, 4, c["M"], len(v)))).contiguous()


def _surrogate_inputs(c, seed):
    K, H = c["K"], c["H"]
    lo, hi = 1200.0, 3200.0
    x = lo + (hi - lo) * _rand(seed, 4, c["pairs"] + c["P"], K)
    u = (x - lo) / (hi - lo) - _rand(seed, 5, K)
    misfit = torch.exp((u * u).mean(1).double() * 6.0 - 4.0 + 0.1 * _rand(seed, 6, len(x), dtype=torch.float64))
    w = []
    for i, (rows, cols) in enumerate(((H, K), (H, H), (1, H))):      # He-uniform weights, zero biases
        w.append(((2 * _rand(seed, 10 + i, rows, cols) - 1) * math.sqrt(6.0 / cols)).reshape(-1))
        w.append(torch.zeros(rows, device=DEV))
    return x[: c["pairs"]].contiguous(), misfit[: c["pairs"]].contiguous(), x[c["pairs"]:].contiguous(), torch.cat(w)


def _step_inputs(c, seed):
    P, D = c["P"], c["K"]
    f64 = dict(dtype=torch.float64)
    lo, hi = 1500.0, 4700.0
    x = lo + (hi - lo) * _rand(seed, 1, P, D, **f64)
    v = 800.0 * (2 * _rand(seed, 2, P, D, **f64) - 1)
    p = lo + (hi - lo) * _rand(seed, 3, P, D, **f64)
    misfit = torch.exp(3 * _rand(seed, 4, P, **f64))
    pf = torch.exp(3 * _rand(seed, 5, P, **f64)) * 0.9
    return x, v, p, pf, misfit, int(pf.argmin())


def _pso(c, seed):
    return B.EmpsoPso(c["P"], c["K"], 1.2, 2.9, 0.5, 0.3, 0.25, 10, 1, 12795 + seed)


STEP_K = 20     # generations done before the step: the elitist mutation is on


def prepare(case, seed):
    c = case
    if c["kind"] == "surrogate":
        ctx = B.Context([B.make_grid(101, 101, 10.0, 10.0, 20, 4, 0.5, 10.0, 1200.0, 3200.0)],
                        synth.receiver_line(101, 10.0, 20.0), _pso(c, seed), 1200.0, 3200.0)
        ctx.surrogate_init(hidden=c["H"], capacity=50000, lr=1e-3, seed=77 + seed)
        ctx.surrogate_set_policy(recent=c["recent"])
        x, misfit, swarm, w = _surrogate_inputs(c, seed)
        ctx.surrogate_add(x, misfit)
        ctx.surrogate_set(w)
        return dict(c=c, ctx=ctx, swarm=swarm, logphi=torch.zeros(c["P"], device=DEV), w=w.clone())
    if c["kind"] == "step":
        ctx = B.Context([B.make_grid(101, 101, 10.0, 10.0, 20, 4, 0.5, 10.0, 1200.0, 3200.0)],
                        synth.receiver_line(101, 10.0, 20.0), _pso(c, seed), 1500.0, 4700.0)
        x, v, p, pf, misfit, g = _step_inputs(c, seed)
        ctx.pso_set_state(x, v, p, pf, g, STEP_K)
        out = dict(x=x, v=v, p=p, pf=pf, order=torch.zeros(c["P"], dtype=torch.int32, device=DEV),
                   gk=torch.zeros(2, dtype=torch.int32, device=DEV))
        return dict(c=c, ctx=ctx, misfit=misfit, particles=torch.zeros(c["P"], c["K"], device=DEV), out=out)
    if c["kind"] == "lowpass":
        ctx = B.Context([B.make_grid(61, 41, 10.0, 10.0, 10, 8, 0.25, 15.0, 1500.0, 3000.0)],
                        synth.receiver_line(61, 10.0, 20.0))
        return dict(c=c, ctx=ctx, traces=_lowpass_input(c, seed),
                    out=torch.zeros(c["S"], c["nt_out"], c["nrec"], device=DEV))
    grids = _grids(c)
    made = [B.make_grid(g["nx"], g["nz"], g["hx"], g["hz"], g["pad"], g["order"], g["T"], g["f0"], g["vmin"],
                        g["vmax"], kx=g["kx"], kz=g["kz"], mode=min(g["mode"], 1), dt=g["dt"]) for g in grids]
    recs = [_shots(g)[1] for g in grids]
    ctx = B.Context(made, np.concatenate(recs))
    xz, begin, count, ids, weights, first = [], [], [], [], [], 0
    for i, (g, r) in enumerate(zip(grids, recs)):
        for s in _shots(g)[0]:
            xz.append(s)
            begin.append(first)
            count.append(len(r))
            ids.append(i)
            weights.append(2.0 if len(grids) > 1 and i == 0 else 1.0)
        first += len(r)
    s = dict(c=c, ctx=ctx, shots=B.make_shots(xz, begin, count, ids, weights))
    if c["mode"] == 2:
        z, n, x, _ = _levels(c)
        ctx.set_levels(0, z, n, x)
        ctx.set_water(0, 4 * c["hz"], 1500.0)
    if c["kind"] in ("fitness", "uneven"):
        s["particles"] = _particles(c, seed)
    else:
        s["vel"] = _velocity(c, seed)
    if c["kind"] == "traces":
        s["traces"] = torch.zeros(c["M"], c["S"], _axis(c)[1], c["nx"], device=DEV)
    else:
        s["d_obs"] = torch.cat([_observed(g, seed).reshape(-1) for g in grids])
    if c["kind"] == "gradient":
        s["grad"] = torch.zeros_like(s["vel"])
    s["misfit"] = torch.zeros(c["M"], dtype=torch.float64, device=DEV)
    return s


def run(state):
    s = state
    c, ctx = s["c"], s["ctx"]
    kind = c["kind"]
    if kind in ("fitness", "uneven"):
        ctx.eval_fitness(s["particles"], s["shots"], s["d_obs"], s["misfit"])
        return s["misfit"]
    if kind == "models":
        ctx.eval_models(s["vel"], s["shots"], s["d_obs"], s["misfit"])
        return s["misfit"]
    if kind == "traces":
        ctx.forward_traces(s["vel"], s["shots"], s["traces"])
        return s["traces"]
    if kind == "gradient":
        ctx.gradient(s["vel"], s["shots"], s["d_obs"], s["grad"])
        return s["grad"]
    if kind == "surrogate":
        ctx.surrogate_predict(s["swarm"], s["logphi"])
        ctx.surrogate_train(c["steps"], c["batch"])
        ctx.surrogate_get(s["w"])
        return {"logphi": s["logphi"], "params": s["w"]}
    if kind == "step":
        ctx.pso_step(s["misfit"], s["particles"])
        ctx.pso_get_state(**s["out"])
        return dict(s["out"], particles=s["particles"])
    ctx.lowpass(s["traces"], c["T"] / (c["nt_in"] - 1), s["out"], c["T"] / (c["nt_out"] - 1), c["fcut"], c["half"])
    return s["out"]


def work(case):
    c = case
    kind = c["kind"]
    if kind == "surrogate":
        K, H = c["K"], c["H"]
        net = K * H + H * H + H
        return {"bytes": 4.0 * (c["steps"] * c["batch"] * K + c["P"] * K + 8 * (net + 2 * H + 1)),
                "flops": 2.0 * net * (c["P"] + 3 * c["steps"] * c["batch"])}
    if kind == "step":
        n = c["P"] * c["K"]
        return {"bytes": 8.0 * (6 * n + 4 * c["P"]) + 4.0 * n, "flops": 60.0 * n}
    if kind == "lowpass":
        taps = min(c["nt_in"], 2 * c["half"] * (c["nt_in"] - 1) / c["T"])
        return {"bytes": 4.0 * c["S"] * c["nrec"] * (c["nt_in"] + c["nt_out"]),
                "flops": 2.0 * c["S"] * c["nrec"] * c["nt_out"] * taps}
    flops = bytes_ = 0.0
    for g in _grids(c):
        nt = _axis(g)[1]
        updates = float(c["M"] * c["S"]) * (g["nx"] + 2 * g["pad"]) * (g["nz"] + 2 * g["pad"]) * nt
        per = 3 * g["order"] + 8            # pair sums and products of both axes, centre, damped update
        flops += updates * (2 * per + 3 if kind == "gradient" else per)
        data = 4.0 * c["S"] * nt * g["nx"]
        bytes_ += data * (c["M"] if kind == "traces" else 1)
        if kind not in ("fitness", "uneven"):
            bytes_ += 4.0 * c["M"] * g["nx"] * g["nz"] * (2 if kind == "gradient" else 1)
        if kind == "gradient":              # the forward field's part of the gradient, written and read once
            bytes_ += 8.0 * updates
    return {"bytes": bytes_ + 8.0 * c["M"] * (1 + c["kx"] * c["kz"]), "flops": flops}


# ---- the same in 64 bits ---------------------------------------------------------------------------


def _spline(n, K, mode):
    """[n][K] weights of K even control nodes on n grid nodes: natural cubic spline, or linear."""
    H = (n - 1) / (K - 1)
    i = np.arange(n, dtype=np.float64)
    seg = np.clip(np.floor(i / H).astype(int), 0, K - 2)
    t = (i - seg * H) / H
    W = np.zeros((n, K))
    W[np.arange(n), seg] += 1 - t
    W[np.arange(n), seg + 1] += t
    if mode == 0 and K > 2:
        A = 4 * np.eye(K - 2) + np.eye(K - 2, k=1) + np.eye(K - 2, k=-1)
        D = np.zeros((K - 2, K))
        for j in range(K - 2):
            D[j, j:j + 3] = (6 / H ** 2, -12 / H ** 2, 6 / H ** 2)
        M = np.zeros((K, K))
        M[1:-1] = np.linalg.solve(A, D)
        u = 1 - t
        W += H * H / 6 * ((u ** 3 - u)[:, None] * M[seg] + (t ** 3 - t)[:, None] * M[seg + 1])
    return W


def _models64(c, g, seed):
    """The gridded models [M][nz][nx] on grid g."""
    if c["kind"] not in ("fitness", "uneven"):
        return _velocity(c, seed).double()
    p = _particles(c, seed).double()
    if c["mode"] != 2:
        Wx = torch.tensor(_spline(g["nx"], g["kx"], c["mode"]), device=DEV)
        Wz = torch.tensor(_spline(g["nz"], g["kz"], c["mode"]), device=DEV)
        v = torch.einsum("ja,pab,ib->pji", Wz, p.reshape(-1, g["kz"], g["kx"]), Wx)
        return v.clamp(g["vmin"], g["vmax"])
    lz, n, lx, _ = _levels(c)
    x, z = np.arange(c["nx"]) * c["hx"], np.arange(c["nz"]) * c["hz"]
    ends = np.concatenate([[0], np.cumsum(n)])
    out = []
    for q in p.cpu().numpy():
        lev = np.stack([np.interp(x, lx[a:b].astype(float), q[a:b]) for a, b in zip(ends, ends[1:])])
        out.append(np.stack([np.interp(z, lz.astype(float), lev[:, i]) for i in range(c["nx"])], axis=1))
    v = np.clip(np.stack(out), c["vmin"], c["vmax"])
    v[:, z <= 4 * c["hz"]] = 1500.0
    return torch.tensor(v, device=DEV)


class _Scheme:
    """The damped leapfrog scheme on one grid in 64 bits, for M models by S shots at once."""

    def __init__(self, g, vel, instances=None):
        self.g = g
        dev = dict(device=DEV, dtype=torch.float64)
        self.w = WEIGHTS[g["order"]]
        self.R = len(self.w) - 1
        self.dt, self.nt = _axis(g)
        pad = g["pad"]
        self.NX, self.NZ = g["nx"] + 2 * pad, g["nz"] + 2 * pad
        a = F.pad(vel[:, None], (pad, pad, pad, pad), mode="replicate")[:, 0] ** 2 * self.dt ** 2
        t = torch.zeros(self.NZ, self.NX, **dev)
        for n, h, ax in ((g["nx"], g["hx"], 0), (g["nz"], g["hz"], 1)):
            if pad == 0:
                continue
            i = torch.arange(n + 2 * pad, **dev)
            d = torch.clamp(torch.maximum(pad - i, i - (pad + n - 1)), min=0) / pad
            e = 3 * _f32(g["vmax"]) * math.log(1000.0) / (2 * pad * h) * d * d * self.dt / 2
            t = t + (e[None, :] if ax == 0 else e[:, None])
        self.f = 1 / (1 + t)
        self.back = (1 - t) * self.f
        self.a = a[:, None]                                     # [M][1][NZ][NX]
        self.ix, self.iz = 1 / g["hx"] ** 2, 1 / g["hz"] ** 2
        n = torch.arange(self.nt, **dev)
        b = (math.pi * g["f0"] * (n * self.dt - 1 / g["f0"])) ** 2
        self.wave = (1 - 2 * b) * torch.exp(-b)

    def corners(self, xz, stride):
        """Flat indices [n][4] and bilinear weights [n][4] of positions in metres."""
        g = self.g
        fx = torch.tensor(xz[:, 0] / g["hx"] + g["pad"], device=DEV)
        fz = torch.tensor(xz[:, 1] / g["hz"] + g["pad"], device=DEV)
        i = fx.floor().clamp(0, self.NX - 2)
        j = fz.floor().clamp(0, self.NZ - 2)
        ax, az = fx - i, fz - j
        k = (j * stride + i).long()
        return (torch.stack([k, k + 1, k + stride, k + stride + 1], 1),
                torch.stack([(1 - ax) * (1 - az), ax * (1 - az), (1 - ax) * az, ax * az], 1))

    def zeros(self, I):
        return torch.zeros(I[0], I[1], self.NZ + 2 * self.R, self.NX + 2 * self.R, device=DEV, dtype=torch.float64)

    def inner(self, u):
        R = self.R
        return u[..., R:R + self.NZ, R:R + self.NX]

    def laplacian(self, u, out):
        R, NZ, NX = self.R, self.NZ, self.NX
        torch.mul(self.inner(u), self.w[0] * (self.ix + self.iz), out=out)
        for m in range(1, R + 1):
            for s in (-m, m):
                out.add_(u[..., R:R + NZ, R + s:R + s + NX], alpha=self.w[m] * self.ix)
                out.add_(u[..., R + s:R + s + NZ, R:R + NX], alpha=self.w[m] * self.iz)
        return out

    def forward(self, shots, rec, keep=False, a=None):
        """Traces [M][S][nt][nrec], and with `keep` L u^n + s^n of every step."""
        a = self.a if a is None else a
        I = (a.shape[0], len(shots))
        u, um = self.zeros(I), self.zeros(I)
        lap = torch.empty(*I, self.NZ, self.NX, device=DEV, dtype=torch.float64)
        af, f2 = a * self.f, 2 * self.f
        k, w = self.corners(shots, self.NX)
        k, w = k.repeat(I[0], 1), (w / (self.g["hx"] * self.g["hz"])).repeat(I[0], 1)
        stride = self.NX + 2 * self.R
        rk, rw = self.corners(rec, stride)
        rk = (rk + self.R * stride + self.R).reshape(-1)
        tr = torch.empty(I[0] * I[1], self.nt, len(rec), device=DEV, dtype=torch.float64)
        kept = torch.empty(self.nt, *lap.shape, device=DEV, dtype=torch.float64) if keep else None
        for n in range(self.nt):
            self.laplacian(u, lap)
            lap.view(I[0] * I[1], -1).scatter_add_(1, k, w * self.wave[n])
            if keep:
                kept[n] = lap
            o = self.inner(um)
            o.mul_(-self.back).addcmul_(self.inner(u), f2).addcmul_(lap, af)
            u, um = um, u
            tr[:, n] = (u.view(I[0] * I[1], -1).index_select(1, rk).view(I[0] * I[1], -1, 4) * rw).sum(2)
        return tr.view(*I, self.nt, len(rec)), kept

    def gradient(self, vel, shots, rec, d_obs):
        tr, kept = self.forward(shots, rec, keep=True)
        res = (tr - d_obs)[0]                                   # one model: [S][nt][nrec]
        I = (1, len(shots))
        q, mu1, mu2 = self.zeros(I), None, None
        lap = torch.empty(*I, self.NZ, self.NX, device=DEV, dtype=torch.float64)
        mu1, mu2, G = torch.zeros_like(lap), torch.zeros_like(lap), torch.zeros_like(lap)
        af, f2 = self.a * self.f, 2 * self.f
        k, w = self.corners(rec, self.NX)
        for n in range(self.nt - 1, -1, -1):
            self.inner(q).copy_(mu1 * af)
            self.laplacian(q, lap)
            mu2.mul_(-self.back).addcmul_(mu1, f2).add_(lap)
            flat = mu2.view(len(shots), -1)
            flat.index_add_(1, k.reshape(-1), (res[:, n, :, None] * w).reshape(len(shots), -1))
            mu1, mu2 = mu2, mu1
            G.addcmul_(mu1 * self.f, kept[n])
        G = G.sum(1)                                            # over the shots
        p = self.g["pad"]
        if p:                                                   # the transpose of the edge extension
            G = torch.cat([G[..., :p + 1].sum(-1, keepdim=True), G[..., p + 1:-p - 1],
                           G[..., -p - 1:].sum(-1, keepdim=True)], -1)
            G = torch.cat([G[:, :p + 1].sum(1, keepdim=True), G[:, p + 1:-p - 1],
                           G[:, -p - 1:].sum(1, keepdim=True)], 1)
        return 2 * vel * self.dt ** 2 * G


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of counters (arrays or numbers) under a 64-bit key."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ k0, b & m32, (a >> np.uint64(32)) ^ c[3] ^ k1, a & m32]
    return c


def _step64(c, seed):
    x, v, p, pf, misfit, _ = (t.cpu().numpy() if torch.is_tensor(t) else t for t in _step_inputs(c, seed))
    P, D, k, s = c["P"], c["K"], STEP_K + 1, 12795 + seed
    lo, hi = 1500.0, 4700.0
    better = misfit < pf
    p[better], pf = x[better], np.where(better, misfit, pf)
    g = int(np.argmin(pf))
    order = np.argsort(misfit, kind="stable")
    worst = np.zeros(P, dtype=bool)
    worst[order[P - int(0.25 * P):]] = True
    i, d = np.arange(P)[:, None], np.arange(D)[None, :]

    def unit(purpose, word=0):
        return _philox(k, i, d, purpose, s)[word].astype(np.float64) * 2.0 ** -32 + 2.0 ** -33

    phi = 1.2 + 2.9
    chi = 2 / abs(2 - phi - math.sqrt(phi * phi - 4 * phi))
    vn = np.clip(chi * (v + 1.2 * unit(2) * (p - x) + 2.9 * unit(3) * (p[g] - x)), -0.5 * (hi - lo), 0.5 * (hi - lo))
    normal = np.sqrt(-2 * np.log(unit(5, 0))) * np.cos(2 * np.pi * unit(5, 1))
    mutant = p[g] + np.where(unit(4) < 0.3, 0.1 * (hi - lo) * normal, 0.0)
    w = worst[:, None]
    x = np.clip(np.where(w, mutant, x + vn), lo, hi)
    return dict(x=x, v=np.where(w, v, vn), p=p, pf=pf, order=order.astype(np.int32),
                gk=np.array([g, k], dtype=np.int32), particles=x)


def _surrogate64(c, seed):
    x, misfit, swarm, w = _surrogate_inputs(c, seed)
    K, H, n, key = c["K"], c["H"], c["pairs"], 77 + seed
    y = torch.log(misfit)
    mu, sd = y.mean(), torch.sqrt((y * y).mean() - y.mean() ** 2)
    w = w.double()

    def scaled(v):
        return 2 * (v.double() - 1200.0) / 2000.0 - 1

    def split(w):
        a = H * K
        b = a + H
        d = b + H * H
        return w[:a].view(H, K), w[a:b], w[b:d].view(H, H), w[d:d + H], w[d + H:d + 2 * H], w[d + 2 * H:]

    def net(w, v):
        W1, b1, W2, b2, w3, b3 = split(w)
        z1 = v @ W1.T + b1
        z2 = z1.relu() @ W2.T + b2
        return z1, z2, z2.relu() @ w3 + b3

    logphi = net(w, scaled(swarm))[2]                           # before any training: mean 0, deviation 1
    m, s2 = torch.zeros_like(w), torch.zeros_like(w)
    for step in range(c["steps"]):
        b = np.arange(c["batch"])
        r = _philox(step, b, 5, 7, key)[0]
        rows = (r * np.uint64(n)) >> np.uint64(32)
        if c["recent"] > 0:
            new = n - 1 - ((r * np.uint64(min(c["recent"], n))) >> np.uint64(32)).astype(np.int64)
            rows = np.where(b >= c["batch"] // 2, new, rows.astype(np.int64))
        rows = torch.tensor(rows.astype(np.int64), device=DEV)
        v, t = scaled(x[rows]), (y[rows] - mu) / sd
        W1, b1, W2, b2, w3, b3 = split(w)
        z1, z2, out = net(w, v)
        dy = (out - t) / c["batch"]
        d2 = dy[:, None] * w3 * (z2 > 0)
        d1 = (d2 @ W2) * (z1 > 0)
        g = torch.cat([(d1.T @ v).reshape(-1), d1.sum(0), (d2.T @ z1.relu()).reshape(-1), d2.sum(0),
                       (z2.relu() * dy[:, None]).sum(0), dy.sum()[None]])
        m, s2 = 0.9 * m + 0.1 * g, 0.999 * s2 + 0.001 * g * g
        w = w - 1e-3 * (m / (1 - 0.9 ** (step + 1))) / (torch.sqrt(s2 / (1 - 0.999 ** (step + 1))) + 1e-8)
    return {"logphi": logphi, "params": w}


def _lowpass_input(c, seed):
    """Traces with energy inside and far above the pass band."""
    t = torch.linspace(0, c["T"], c["nt_in"], device=DEV, dtype=torch.float64)[None, :, None]
    x = torch.arange(c["nrec"], device=DEV, dtype=torch.float64)[None, None, :]
    s = torch.arange(c["S"], device=DEV, dtype=torch.float64)[:, None, None]
    r = _rand(seed, 1, 4, dtype=torch.float64).cpu().numpy()
    out = 0.02 * (_rand(seed, 2, c["S"], c["nt_in"], c["nrec"]) - 0.5)
    for k, q in enumerate(r):
        a = (math.pi * 17.0 * (t - c["T"] * (0.15 + 0.2 * k) - 0.001 * (q + 0.5) * x * (1 + 0.1 * s))) ** 2
        out += (0.2 / (k + 1) * (1 - 2 * a) * torch.exp(-a)).float()
    return out.contiguous()


def _lowpass64(c, seed):
    dt_in, dt_out = c["T"] / (c["nt_in"] - 1), c["T"] / (c["nt_out"] - 1)
    m = torch.arange(c["nt_out"], device=DEV, dtype=torch.float64)[:, None] * dt_out
    n = torch.arange(c["nt_in"], device=DEV, dtype=torch.float64)[None, :] * dt_in
    u = (m - n) / c["half"]
    win = 0.42 + 0.5 * torch.cos(math.pi * u) + 0.08 * torch.cos(2 * math.pi * u)
    h = torch.where(u.abs() < 1, 2 * c["fcut"] * dt_in * torch.sinc(2 * c["fcut"] * (m - n)) * win, 0.0)
    return torch.matmul(h, _lowpass_input(c, seed).double())


def exact(case, seed):
    c = case
    if c["kind"] == "surrogate":
        return _surrogate64(c, seed)
    if c["kind"] == "step":
        return _step64(c, seed)
    if c["kind"] == "lowpass":
        return _lowpass64(c, seed)
    total = torch.zeros(c["M"], dtype=torch.float64, device=DEV)
    for i, g in enumerate(_grids(c)):
        shots, rec = _shots(g)
        vel = _models64(c, g, seed)
        sch = _Scheme(g, vel)
        if c["kind"] == "gradient":
            return sch.gradient(vel, shots, rec, _observed(g, seed).double())
        if c["kind"] == "traces":
            return sch.forward(shots, rec)[0]
        d = _observed(g, seed).double()
        weight = 2.0 if c["kind"] == "uneven" and i == 0 else 1.0
        part = max(1, int(4e7 / (sch.NX * sch.NZ * len(shots))))      # models at once
        for m in range(0, c["M"], part):
            tr = sch.forward(shots, rec, a=sch.a[m:m + part])[0]
            total[m:m + part] += weight * 0.5 * ((tr - d) ** 2).sum((1, 2, 3))
    return total
