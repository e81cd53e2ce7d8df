"""The work a user of this framework has it do, as cases to be timed and compared.

Each case goes through the public binding: whole solves and a control step of a
batch, the rollout of given controls in its forms (hard and soft separation,
noise, shared and per-particle wind, rolling window), its gradient, the wind
field, the weights with their resampling and selection, and the perturbation.
Sizes are those of the repository's workloads (2, 8, 12 and 24 aircraft, mixed
batches, the paper's standard problem) or lie between them.
"""
import math

import numpy as np
import torch

import paper_1506_02869_gb300 as tma
import scenarios as S

DEV = "cuda"


def listed():
    return [
        # the smallest control problem (2 aircraft): one solve, bound by latency and launches
        dict(name="solve_2ac", kind="solve", N=2, H=20, S=4, L=1024, M=8, J=10, grid="16x16x4", box=30, sep=0),
        # a receding-horizon solve of the 8-aircraft traffic, wind field on the fine grid included
        dict(name="solve_8ac", kind="solve", N=8, H=60, S=4, L=16384, M=32, J=8, grid="64x64x8", box=50, sep=0),
        # a solve with accepted random-walk moves (two more rollouts an iteration)
        dict(name="solve_rwmh", kind="solve", N=6, H=30, S=4, L=4096, M=8, J=4, grid="16x16x4", box=50, sep=1,
             move=1),
        # one control step of a batch of uneven scenarios: measured states in, graph, results out
        dict(name="batch_mpc", kind="batch", scen=12, L=2048, M=16, H=60, J=6, grid="16x16x4"),
        # the rollout inside late iterations of the 8-aircraft workload at its full size, hard separation
        dict(name="rollout_8ac", kind="rollout", N=8, H=60, S=4, L=65536, M=32, J=20, grid="64x64x8", box=50, sep=0,
             controls="late"),
        # dense traffic: 24 aircraft, long horizon, noise map, hard and soft separation
        dict(name="rollout_24ac", kind="rollout", N=24, H=120, S=4, L=8192, M=64, J=20, grid="64x64x8", box=50,
             sep=2, noise=True, controls="late"),
        # the paper's standard problem: short horizon, a wind field per particle, rolling window,
        # SampleSchedule draws
        dict(name="rollout_paper", kind="rollout", N=10, H=6, S=4, L=10240, M=256, J=50, grid="2x2x2", box=50, sep=1,
             wind_mode=1, sample_mode=1, rolling=True, controls="late"),
        # first iteration (uniform controls, many infeasible) at ragged sizes, three control segments
        dict(name="rollout_ragged", kind="rollout", N=13, H=45, S=3, L=5003, M=7, J=0, grid="17x16x5", box=50, sep=1,
             controls="first"),
        # the gradient of the soft cost on the 12-aircraft workload
        dict(name="grad_12ac", kind="grad", N=12, H=60, S=4, L=16384, M=16, J=20, grid="16x16x4", box=50, sep=1,
             controls="late"),
        # a wind field on the fine grid, handed to the caller
        dict(name="wind_64", kind="wind", N=8, H=60, S=4, L=256, M=16, J=0, grid="64x64x8", box=50, sep=0),
        # annealed weights, resampling and final selection over the dense traffic's full particle set
        dict(name="weights_24ac", kind="weights", N=24, L=262144, Lout=262144, J=10),
        # gather and perturbation of that particle set
        dict(name="move_24ac", kind="move", N=24, H=120, S=4, L=262144, M=1, J=10, grid="16x16x4", box=50, sep=2),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "batch", "rollout", "rollout", "rollout", "grad", "wind", "weights", "move"])
    grid = rng.choice(["16x16x4", "32x32x8", "64x64x8", "17x12x5"])
    if kind == "solve":
        sep = rng.choice([0, 1, 2])
        # Langevin moves turn the gradient's last bits into accept decisions: their gradient has its own cases
        move = rng.choice([0, 1]) if sep else 0
        return dict(kind=kind, N=rng.randint(2, 12), H=rng.randint(10, 60), S=rng.randint(1, 5),
                    L=_spread(rng, 512, 16384), M=rng.randint(4, 24), J=rng.randint(2, 8), grid="16x16x4", box=50,
                    sep=sep, move=move)
    if kind == "batch":
        return dict(kind=kind, scen=rng.randint(2, 12), L=_spread(rng, 256, 2048), M=rng.randint(2, 16),
                    H=rng.randint(10, 60), J=rng.randint(2, 6), grid="16x16x4")
    if kind in ("rollout", "grad"):
        c = dict(kind=kind, N=rng.randint(1, 32), H=rng.randint(5, 90), S=rng.randint(1, 5), L=_spread(rng, 200, 32768),
                 M=_spread(rng, 2, 40), J=rng.randint(0, 30), grid=grid, box=rng.choice([30, 50, 60]),
                 sep=rng.choice([0, 1, 2]), controls=rng.choice(["late", "first"]))
        while c["N"] * c["N"] * c["H"] * c["L"] * c["M"] > 6e9:
            c["L"] = max(200, c["L"] // 3)
            c["M"] = max(2, c["M"] // 2)
        if kind == "grad":
            return dict(c, N=min(c["N"], 24), sep=rng.choice([1, 2]), noise=rng.random() < 0.3)
        form = rng.random()
        if form < 0.2:
            return dict(c, grid="2x2x2", wind_mode=1, sample_mode=rng.choice([0, 1]), rolling=rng.random() < 0.5)
        return dict(c, noise=rng.random() < 0.3, rolling=rng.random() < 0.15)
    if kind == "wind":
        return dict(kind=kind, N=2, H=rng.randint(5, 90), S=4, L=256, M=rng.randint(2, 12), J=0, grid=grid, box=50, sep=0)
    if kind == "weights":
        L = _spread(rng, 500, 262144)
        return dict(kind=kind, N=rng.randint(1, 24), L=L, Lout=L if rng.random() < 0.7 else max(1, int(L * rng.uniform(0.3, 1))),
                    J=rng.randint(0, 30))
    return dict(kind=kind, N=rng.randint(1, 24), H=30, S=rng.randint(1, 5), L=_spread(rng, 500, 262144), M=1,
                J=rng.randint(0, 30), grid="16x16x4", box=50, sep=0)


# ------------------------------------------------------------------ inputs

def _grid(case):
    return tuple(int(v) for v in case["grid"].split("x"))


def _problem(case, seed):
    """The scenario of a case: seeded traffic (arrivals and departures) with the workloads' constants."""
    rng = np.random.default_rng(seed)
    N, box = case["N"], 1000.0 * case["box"]
    top = 6000.0 if case["box"] == 30 else 8000.0
    p = S.Problem(N=N, H=case["H"], L=case["L"], M=case["M"], J_max=case["J"] if case["kind"] == "solve" else 30,
                  S=min(case["S"], case["H"]), seed=seed * 7919 + 17, box_lo=(-box, -box, 0.0), box_hi=(box, box, top),
                  grid=_grid(case), z_max=top, sep_mode=case["sep"], wind_mode=case.get("wind_mode", 0),
                  sample_mode=case.get("sample_mode", 0), rolling=int(case.get("rolling", False)))
    n_arr = (N + 1) // 2
    p.aircraft = S._traffic(rng, n_arr, N - n_arr, ring=0.8 * box, z_top=top, sep_h=p.sep_h, sep_v=p.sep_v)
    if case.get("noise"):
        p.w_noise = 0.1
        p.popdense, p.pop_lo, p.pop_hi = S.popdense_grid(rng)
        p.pop_n = p.popdense.shape
    if p.rolling:
        # some aircraft enter within the horizon
        late = rng.random(N) < 0.3
        p.aircraft["t_enter"] = np.where(late, 5 + rng.integers(0, max(2, p.H // 2), N), 0)
        p.mpc_step = 5
    return p


def _controls(p, case, seed):
    """Controls [L][N][S][3]: the uniform draw of the first iteration, or the cloud of a late one (a
    moderate sequence per aircraft with the spread of a few perturbations around it)."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    lo = torch.tensor(p.ctrl_lo, device=DEV, dtype=torch.float32)
    hi = torch.tensor(p.ctrl_hi, device=DEV, dtype=torch.float32)
    shape = (p.L, p.N, p.S, 3)
    if case["controls"] == "first":
        return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV)
    scale = torch.tensor([0.2, 0.12, 0.06], device=DEV)
    mid = 0.5 * (hi - lo) * scale * (2 * torch.rand((1,) + shape[1:], generator=g, device=DEV) - 1)
    mid[..., 1] = mid[..., 1].abs()       # level or climbing: thrust stays positive
    sig = 0.7 * torch.tensor(p.move_sigma, device=DEV, dtype=torch.float32)
    return torch.minimum(torch.maximum(mid + sig * torch.randn(shape, generator=g, device=DEV), lo), hi)


def _costs(case, seed):
    """Mean costs [N][L] of an iteration: exponential, a tenth infeasible."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    c = torch.empty((case["N"], case["L"]), device=DEV).exponential_(0.5, generator=g)
    c[torch.rand(c.shape, generator=g, device=DEV) < 0.1] = math.inf
    return c


def _scenarios(case, seed):
    """The batch workload's scenarios: uneven aircraft counts (the case's own), seeded traffic."""
    rng, counts = np.random.default_rng(seed), np.random.default_rng(case["scen"]).integers(2, 33, case["scen"])
    base, out = S.config5(n_scen=1)[0], []
    for s, n in enumerate(int(v) for v in counts):
        p = S.shrink(base.copy(N=n, seed=seed * 7919 + 29, scenario_id=s, aircraft=None), L=case["L"], M=case["M"],
                     H=case["H"], J_max=case["J"], grid=_grid(case))
        p.aircraft = S._traffic(rng, (n + 1) // 2, n // 2, ring=45000.0, z_top=9000.0, sep_h=p.sep_h, sep_v=p.sep_v,
                                dep_r=(2000.0, 30000.0))
        out.append(p)
    return out


def _kappa(J):
    return math.floor(3 + 5 * math.exp(0.05 * J))


class _Batch:
    """Owns a batch handle."""

    def __init__(self, ps):
        self.h = tma.tma_batch_create(ps)

    def __del__(self):
        tma.tma_batch_destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind, seed=seed)
    if kind == "weights":
        N, L = case["N"], case["L"]
        lib = tma.lib()
        st.update(cbar=_costs(case, seed), wt=torch.empty((N, L), dtype=torch.float64, device=DEV),
                  anc=torch.empty((N, case["Lout"]), dtype=torch.int32, device=DEV),
                  deg=torch.zeros(1, dtype=torch.int32, device=DEV),
                  work=torch.empty(max(16, lib.tma_lse_resample_workspace(N, L)), dtype=torch.uint8, device=DEV),
                  best=torch.empty(1, dtype=torch.int64, device=DEV),
                  bsum=torch.empty(1, dtype=torch.float64, device=DEV),
                  ninf=torch.empty(1, dtype=torch.int32, device=DEV),
                  swork=torch.empty(max(16, lib.tma_select_workspace(L)), dtype=torch.uint8, device=DEV))
        return st
    if kind == "batch":
        ps = _scenarios(case, seed)
        x0 = np.concatenate([np.stack([p.aircraft[f] for f in ("x", "y", "z", "v", "chi", "m")], axis=1) for p in ps])
        st.update(batch=_Batch(ps), x0=x0, mpc=[p.mpc_step for p in ps], Ns=[p.N for p in ps], S=ps[0].S)
        return st
    p = _problem(case, seed)
    if kind == "move":
        g = torch.Generator(device=DEV).manual_seed(seed)
        u = torch.tensor(p.ctrl_lo, device=DEV) + torch.rand((p.L, p.N, p.S, 3), generator=g, device=DEV) * (
            torch.tensor(p.ctrl_hi, device=DEV) - torch.tensor(p.ctrl_lo, device=DEV))
        # ancestors as systematic resampling leaves them: increasing, many repeated
        anc = torch.randint(0, p.L, (p.N, p.L), generator=g, device=DEV, dtype=torch.int32)
        anc = (anc // 3 * 3).sort(dim=1).values.contiguous()
        st.update(solver=tma.Solver(p), u=u.float(), anc=anc, out=torch.empty_like(u.float()))
        return st
    st["solver"] = tma.Solver(p)
    if kind == "solve" and case.get("move"):
        st["solver"].set_move(case["move"], 0.5)
    if kind == "wind":
        st["W"] = torch.empty((p.M, p.H, math.prod(p.grid), 2), device=DEV)
    if kind in ("rollout", "grad"):
        st["u"] = _controls(p, case, seed)
        tma.tma_wind_field(st["solver"].h)       # the current field, as a control loop has it
    return st


def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "weights":
        tma.tma_lse_resample(st["cbar"], float(_kappa(case["J"])), st["seed"], 3, case["J"], 7, st["wt"], st["anc"],
                             st["deg"], st["work"])
        tma.tma_select(st["cbar"], st["best"], st["bsum"], st["ninf"], st["swork"])
        return {k: st[k] for k in ("wt", "anc", "best", "bsum", "ninf", "deg")}
    if kind == "batch":
        h = st["batch"].h
        tma.tma_batch_set_state(h, st["x0"], st["mpc"])
        tma.tma_batch_mpc(h, 1, True)
        r = tma.tma_batch_results(h, st["Ns"], st["S"])
        return {"best_u": np.concatenate(r["best_u"]), "cost": r["best_cost"], "best": r["best"],
                "states": np.concatenate(r["states"])}
    s = st["solver"]
    if kind == "solve":
        best_u, cost, _ = s.solve()
        return {"best_u": best_u, "cost": cost, "particles": s.particles()}
    if kind == "rollout":
        cbar, soft = s.rollout_cost(st["u"], case["J"], soft=case["sep"] != 0)
        return {"cbar": cbar, "soft": soft}
    if kind == "grad":
        cost, grad, cbar = s.rollout_grad(st["u"], case["J"], cbar=True)
        return {"cost": cost, "grad": grad, "cbar": cbar}
    if kind == "wind":
        return {"W": tma.tma_wind_field(s.h, st["W"])}
    tma.tma_move(s.h, st["u"], st["anc"], case["J"], st["out"])
    return {"u": st["out"]}


def work(case):
    kind = case["kind"]
    if kind == "weights":
        n = case["N"] * case["L"]
        return {"bytes": 4 * n + 8 * n + 4 * case["N"] * case["Lout"], "flops": 30 * n}
    if kind == "batch":
        n = sum(p.N for p in _scenarios(case, 1))
        units = n * case["L"] * case["M"] * case["H"] * case["J"]
        return {"bytes": 16 * n * case["L"] * case["J"], "flops": 300 * units}
    N, L, M, H, Sg = case["N"], case["L"], case["M"], case["H"], min(case["S"], case["H"])
    u = 12 * Sg * N * L
    if kind == "move":
        return {"bytes": 2 * u + 4 * N * L, "flops": 20 * 3 * Sg * N * L}
    P = math.prod(_grid(case))
    field = 8 * M * H * P
    if kind == "wind":
        nxy = P // _grid(case)[2]
        return {"bytes": field, "flops": M * H * P * 2 * (nxy + 30)}
    Mj = min(_kappa(case["J"]), M) if case.get("sample_mode") else M
    # one aircraft-step under one wind sample, with half of the pairs each
    unit = 175 + (8 if case["sep"] == 0 else 17) * (N - 1) / 2
    one = unit * N * L * Mj * H
    if kind == "rollout":
        return {"bytes": u + 4 * N * L * (2 if case["sep"] else 1) + (0 if case.get("wind_mode") else field), "flops": one}
    if kind == "grad":
        return {"bytes": 2 * u + 4 * N * L + field, "flops": 3 * one}
    # a solve: the field and J rollouts; accepted random-walk moves add two rollouts an iteration
    extra = {0: 0, 1: 2}[case.get("move", 0)] * (case["J"] - 1)
    return {"bytes": field + u * case["J"], "flops": one * (case["J"] + extra)}


# ------------------------------------------------------ the same in 64 bits

F64 = torch.float64
M32 = 0xFFFFFFFF


def _philox(key, c0, c1, c2, c3):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    k0, k1 = key & M32, (key >> 32) & M32
    c = list(torch.broadcast_tensors(*(torch.as_tensor(v, dtype=torch.int64, device=DEV) for v in (c0, c1, c2, c3))))
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _normals(a, b):
    u, v = (((x >> 9).to(F64) + 0.5) / 8388608.0 for x in (a, b))
    r = torch.sqrt(-2.0 * torch.log(u))
    return r * torch.cos(2 * math.pi * v), r * torch.sin(2 * math.pi * v)


def _key(p):
    return (p.seed + p.scenario_id * 0x9E3779B97F4A7C15) & 0xFFFFFFFFFFFFFFFF


def _correlation(p, grid):
    """Cholesky factors of the horizontal and vertical correlation (FP64)."""
    ax = [torch.linspace(p.box_lo[d], p.box_hi[d], grid[d], dtype=F64, device=DEV) for d in range(3)]
    x, y = (v.reshape(-1) for v in torch.meshgrid(ax[0], ax[1], indexing="ij"))
    d = torch.sqrt((x[:, None] - x[None]) ** 2 + (y[:, None] - y[None]) ** 2)
    dz = (ax[2][:, None] - ax[2][None]).abs()
    return torch.linalg.cholesky(torch.exp(-p.beta_xy * d)), torch.linalg.cholesky(torch.exp(-p.gam_z * dz))


def _wind64(p):
    """W[M][H][P][2]."""
    nz, nxy = p.grid[2], p.grid[0] * p.grid[1]
    Lxy, Lz = _correlation(p, p.grid)
    node = torch.arange(nxy * nz, device=DEV)[None, :]
    m = torch.arange(p.M, device=DEV)[:, None] << 8
    a = math.exp(-p.dt * p.lam_t)
    W = torch.empty((p.M, p.H, nxy * nz, 2), dtype=F64, device=DEV)
    B = None
    for k in range(p.H):
        w = _philox(_key(p), node, m, k | (3 << 24), p.mpc_step << 16)
        v = torch.stack(_normals(w[0], w[1]), -1).reshape(p.M, nxy, nz, 2)
        B = v if B is None else a * B + math.sqrt(1 - a * a) * v
        W[:, k] = torch.einsum("pq,mqzc->mpzc", Lxy, torch.einsum("zy,mqyc->mqzc", Lz, B)).reshape(p.M, -1, 2)
    return p.wind_sigma * W


def _wrapped(a):
    return (a - 2 * math.pi * torch.round(a / (2 * math.pi))).abs()


def _cell(p, n, lo, hi, v):
    f = (v.clamp(lo, hi) - lo) * ((n - 1) / (hi - lo))
    i = f.detach().floor().long().clamp(0, n - 2)
    return i, f - i


def _interpolate(p, Wk, x, y, z):
    """Trilinear wind: Wk [m][P][2], positions [m][N][L]."""
    g = p.grid
    ix, tx = _cell(p, g[0], p.box_lo[0], p.box_hi[0], x)
    iy, ty = _cell(p, g[1], p.box_lo[1], p.box_hi[1], y)
    iz, tz = _cell(p, g[2], p.box_lo[2], p.box_hi[2], z)
    row = torch.arange(Wk.shape[0], device=DEV)[:, None, None]
    out = 0.0
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                w = (tx if a else 1 - tx) * (ty if b else 1 - ty) * (tz if c else 1 - tz)
                out = out + w[..., None] * Wk[row, ((ix + a) * g[1] + iy + b) * g[2] + iz + c]
    return out


def _rollout64(p, u, J, ms, W):
    """Per-sample costs (hard, soft) [m][N][L] of the samples `ms` (a tensor) for controls u[L][N][S][3]."""
    N, L, H = p.N, u.shape[0], p.H
    ac = {f: torch.as_tensor(p.aircraft[f].astype(np.float64), device=DEV)[None, :, None] for f in p.aircraft.dtype.names}
    full = (len(ms), N, L)
    el, ei, em = torch.arange(L, device=DEV)[None, None], torch.arange(N, device=DEV)[None, :, None], ms[:, None, None]
    x, y, z, v, chi = (ac[f].expand(full) for f in ("x", "y", "z", "v", "chi"))
    fuel, soft, sA, sB, sC, sN = (torch.zeros(full, dtype=F64, device=DEV) for _ in range(6))
    zero = torch.zeros(full, dtype=torch.bool, device=DEV)
    dead, landed, viol = zero, zero, zero
    arrival = ac["type"] == 0
    k_in = (ac["t_enter"] - p.mpc_step).clamp(0, H) if p.rolling else ac["t_enter"] * 0
    Ha = (H - k_in).clamp_min(1)
    out = k_in >= H
    key, mpc = _key(p), p.mpc_step
    if p.wind_mode:
        lxy, lz = _correlation(p, (2, 2, 2))
        Q = p.wind_sigma * torch.kron(lxy, lz)
        a = math.exp(-p.dt * p.lam_t)
        B = None
    if p.popdense is not None:
        pop = torch.as_tensor(np.asarray(p.popdense, np.float64), device=DEV)
    z0 = z
    for k in range(H):
        s = k * p.S // H
        uw, uh, ua = (u[:, :, s, c].T[None] for c in range(3))
        fly = ~dead & ~landed & ~out & (k >= k_in)
        mass = ac["m"] - fuel
        sg = uh / v
        ok = sg.abs() <= math.sin(p.gamma_max)
        cg = torch.sqrt((1 - sg * sg).clamp_min(1e-12))
        tp = uw * v / (9.80665 * cg)
        ok = ok & (tp.abs() < math.tan(p.phi_max))
        rho = 1.225 * (1 - 2.2558e-5 * z).clamp_min(1e-30) ** 4.2559
        qS = 0.5 * ac["S"] * rho * v * v
        CL = mass * 9.80665 * cg * torch.sqrt(1 + tp * tp) / qS
        T = mass * (ua + 9.80665 * sg) + qS * (ac["CD0"] + ac["CD2"] * CL * CL)
        ok = ok & (T >= ac["Tmin"]) & (T <= ac["Tmax"])
        dead = dead | (fly & ~ok)
        fly = fly & ok
        if p.wind_mode:
            v8 = []
            for r in range(4):
                w = _philox(key, el, 4 * em + r, k | (9 << 24), mpc << 16)
                v8 += [torch.stack(_normals(w[0], w[1]), -1), torch.stack(_normals(w[2], w[3]), -1)]
            v8 = torch.stack(v8, -2)[:, 0]                               # [m][L][8][2]
            B = v8 if B is None else a * B + math.sqrt(1 - a * a) * v8
            f = (torch.einsum("nj,mljc->mlnc", Q, B))[:, None]
            t = [((q - p.box_lo[d]) / (p.box_hi[d] - p.box_lo[d])).clamp(0, 1) for d, q in enumerate((x, y, z))]
            wind = 0.0
            for n in range(8):
                wt = (t[0] if n & 4 else 1 - t[0]) * (t[1] if n & 2 else 1 - t[1]) * (t[2] if n & 1 else 1 - t[2])
                wind = wind + wt[..., None] * f[..., n, :]
        else:
            wind = _interpolate(p, W[ms, k], x, y, z)
        if k % 2 == 0:
            words = _philox(key, el, ei | (em << 8), k >> 1, J | (mpc << 16))
        n = _normals(*words[2 * (k % 2):2 * (k % 2) + 2])
        x1 = x + p.dt * (v * cg * torch.cos(chi) + wind[..., 0] + p.turb_sigma * n[0])
        y1 = y + p.dt * (v * cg * torch.sin(chi) + wind[..., 1] + p.turb_sigma * n[1])
        f1 = fuel + p.dt * ac["Cf1"] * (1 + v / ac["Cf2"]) * T
        new = (x1, y1, z + p.dt * uh, v + p.dt * ua, chi + p.dt * uw, f1)
        x, y, z, v, chi, fuel = (torch.where(fly, b, c) for b, c in zip(new, (x, y, z, v, chi, fuel)))
        good = (z >= p.z_min) & (z <= p.z_max) & (v >= p.v_min) & (v <= p.v_max) & (ac["m"] - fuel >= ac["m_empty"])
        dead = dead | (fly & ~good)
        fly = fly & good
        r = torch.sqrt((x * x + y * y).clamp_min(1e-12))
        th = torch.atan2(y, x)
        sn = torch.sin(th.abs())
        small = th.abs() < 1e-6
        ratio = torch.where(small, 1 + th * th / 6, th.abs() / torch.maximum(torch.where(small, 1.0, sn), 0.25 * th.abs()).clamp_min(1e-12))
        beta = torch.atan2(z, r * ratio)
        land = fly & arrival & (r <= p.P_runway) & (beta <= p.P_beta) & (x > 0) & (th.abs() <= p.P_chi) & (
            _wrapped(chi - math.pi) <= p.P_chi) & (v <= p.P_vs)
        landed = landed | land
        act = fly & ~land
        sA = sA + act * torch.where(arrival, _wrapped(chi - math.pi - 2 * th), _wrapped(th - ac["theta_F"]))
        sB = sB + act * torch.where(arrival, (beta - p.beta_f).abs(), (ac["Z"] - z).abs())
        sC = sC + act * (v - ac["v_D"]).abs()
        if p.w_noise:
            h = (1 - (z / p.A_c) ** 2).clamp_min(0)
            i0, t0 = _cell(p, p.pop_n[0], p.pop_lo[0], p.pop_hi[0], x)
            i1, t1 = _cell(p, p.pop_n[1], p.pop_lo[1], p.pop_hi[1], y)
            d = (1 - t0) * ((1 - t1) * pop[i0, i1] + t1 * pop[i0, i1 + 1]) + t0 * (
                (1 - t1) * pop[i0 + 1, i1] + t1 * pop[i0 + 1, i1 + 1])
            inside = (x >= p.pop_lo[0]) & (x <= p.pop_hi[0]) & (y >= p.pop_lo[1]) & (y <= p.pop_hi[1])
            sN = sN + act * inside * h * d
        for j in range(1, N):
            # partners i + j (mod N)
            q = [torch.roll(t, -j, 1) for t in (x, y, z, act)]
            both = act & q[3]
            dh = torch.sqrt(((x - q[0]) ** 2 + (y - q[1]) ** 2).clamp_min(1e-12))
            dz = (z - q[2]).abs()
            viol = viol | (both & (dh < p.sep_h) & (dz < p.sep_v))
            if p.sep_mode:
                g = torch.minimum(1 - dh / p.sep_h, 1 - dz / p.sep_v)
                soft = soft + both * torch.nn.functional.softplus(p.sp_beta * g, threshold=700.0) / p.sp_beta
    Jf = 1 - fuel * (H / Ha) / (H * p.dt * ac["Tmax"] * ac["Cf1"] * (1 + p.v_max / ac["Cf2"]))
    d0, c = (ac["Z"] - z0).abs(), p.v_max * math.sin(p.gamma_max) * p.dt
    K = torch.minimum(torch.floor(d0 / c), Ha.to(F64))
    sup, inf = d0 + c * (Ha + 1) / 2, (K * d0 - c * K * (K + 1) / 2) / Ha
    J1 = 1 - sA / Ha / math.pi
    dep = p.alpha_dep[0] * J1 + p.alpha_dep[1] * Jf + p.alpha_dep[2] * (sup - sB / Ha) / (sup - inf) + p.alpha_dep[3] * (
        1 - sC / Ha / torch.maximum(p.v_max - ac["v_D"], ac["v_D"] - p.v_min))
    arr = p.alpha_arr[0] * J1 + p.alpha_arr[1] * (1 - sB / Ha * 2 / math.pi) + p.alpha_arr[2] * Jf
    JT = (1 - p.w_noise) * torch.where(arrival, arr, dep) + p.w_noise * (1 - sN / Ha)
    cost = torch.where(out, 0.0, -torch.log(JT.clamp_min(1e-30)))
    bad = torch.tensor(math.inf, dtype=F64, device=DEV)
    return torch.where(dead | viol, bad, cost), torch.where(dead, bad, cost + torch.where(out, 0.0, p.mu_sep * soft))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch"):
        return None       # a chain of discrete choices (resampling, selection)
    if kind == "weights":
        c = _costs(case, seed).to(F64)
        cmin = c.min(dim=1, keepdim=True).values
        return {"wt": torch.where(torch.isinf(c), 0.0, torch.exp(_kappa(case["J"]) * (cmin - c)))}
    p = _problem(case, seed)
    if kind == "wind":
        return {"W": _wind64(p)}
    if kind == "move":
        g = torch.Generator(device=DEV).manual_seed(seed)
        lo, hi = torch.tensor(p.ctrl_lo, device=DEV), torch.tensor(p.ctrl_hi, device=DEV)
        u = (lo + torch.rand((p.L, p.N, p.S, 3), generator=g, device=DEV) * (hi - lo)).float()
        anc = torch.randint(0, p.L, (p.N, p.L), generator=g, device=DEV, dtype=torch.int32)
        anc = (anc // 3 * 3).sort(dim=1).values.long()
        el, ei = torch.arange(p.L, device=DEV)[:, None, None], torch.arange(p.N, device=DEV)[None, :, None]
        w = _philox(_key(p), el, ei, torch.arange((3 * p.S + 3) // 4, device=DEV) | (1 << 24), case["J"] | (p.mpc_step << 16))
        z = torch.stack(_normals(w[0], w[1]) + _normals(w[2], w[3]), -1).reshape(p.L, p.N, -1)[..., :3 * p.S]
        par = u[anc.T, torch.arange(p.N, device=DEV)[None, :]].to(F64)
        new = par + torch.tensor(p.move_sigma, dtype=F64, device=DEV) * z.reshape(par.shape)
        lo64, hi64 = (torch.tensor(v, dtype=F64, device=DEV) for v in (p.ctrl_lo, p.ctrl_hi))
        return {"u": torch.minimum(torch.maximum(new, lo64), hi64)}
    u = _controls(p, case, seed).to(F64)
    J = case["J"]
    M = min(_kappa(J), p.M) if p.sample_mode else p.M
    W = None if p.wind_mode else _wind64(p)
    if kind == "rollout":
        step = max(1, int(2e9 / (60 * p.N * p.L)))
        hard, soft = torch.zeros((p.N, p.L), dtype=F64, device=DEV), torch.zeros((p.N, p.L), dtype=F64, device=DEV)
        with torch.no_grad():
            for m in range(0, M, step):
                a, b = _rollout64(p, u, J, torch.arange(m, min(M, m + step), device=DEV), W)
                hard += a.sum(0)
                soft += b.sum(0)
        return {"cbar": hard / M, "soft": soft / M if p.sep_mode else None}
    # the gradient, sample by sample: the graph of one sample's rollout has to fit the card
    if 8 * p.N * p.L * p.H * (400 + 14 * p.N) > 1e11:
        return None
    cbar, grad = torch.zeros((p.N, p.L), dtype=F64, device=DEV), torch.zeros_like(u)
    for m in range(M):
        v = u.detach().requires_grad_(True)
        _, soft = _rollout64(p, v, J, torch.arange(m, m + 1, device=DEV), W)
        torch.where(torch.isinf(soft), 0.0, soft).sum().backward()
        grad += v.grad
        cbar += soft.detach()[0]
    bad = torch.isinf(cbar).any(0)
    grad[bad] = 0.0
    return {"cost": torch.where(bad, math.inf, cbar.sum(0)) / M, "grad": grad / M, "cbar": cbar / M}
