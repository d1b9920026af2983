"""Timed cases of the library: what a program that generates SPARKLING
trajectories (arxiv 2108.02991) asks of it, through the Python binding.

A case names an operation, the pattern (Nc shots of Ns samples), the density
grid and the options that the program sets:

  grad       sparkling_grad, with A and R
  step       sparkling_step, in place (an iteration of an optimisation)
  energy     sparkling_energy_fn and its backward
  batched    sparkling_step_batched, trajectories of uneven size
  project    sparkling_project of a pattern that is not feasible yet
  multires   sparkling_multires, Algorithm 1 over several resolutions

"fast" cases set the interpolated attraction and the mesh repulsion.
"""
import math

import numpy as np
import torch

import paper_2108_02991_gb300 as sp

_DEFAULTS = dict(dtype="f32", acc="kahan", density="power", n_iter=100, pin=True, mixed=False,
                 eps=0.0, perturb=0.0, mesh=0)


def _case(name, op, Nc, Ns, n, **kw):
    nx, ny, nz = n if isinstance(n, tuple) else (n, n, n)
    c = dict(_DEFAULTS, op=op, Nc=Nc, Ns=Ns, nx=nx, ny=ny, nz=nz)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest workload: one gradient of 1024 samples, the call of
        # tests, tuning loops and toy problems; launches and latency count.
        _case("grad_tiny_f32", "grad", 16, 64, 32, perturb=0.3),
        # A step of a 2-D-sized problem with ragged sizes everywhere, FP64.
        _case("step_odd_f64", "step", 37, 129, (50, 33, 45), dtype="f64", acc="fp64", pin=False),
        # A step of the small workload (64 shots, one low-resolution volume).
        _case("step_small_f32", "step", 64, 1024, 64),
        # The regularised kernel (fixed-step convergence) and the opt-in
        # mixed-precision projection, at an in-between size.
        _case("step_regularised_mixed", "step", 128, 500, 80, mixed=True, eps=1e-3,
              density="gauss"),
        # Energy and its gradient through autograd, FP64 fold, odd shots.
        _case("energy_autograd_f32", "energy", 250, 331, 96, acc="fp64"),
        # An iteration of the medium workload: the ordinary exact step.
        _case("step_medium_f32", "step", 512, 512, 128, density="gauss"),
        # Sixteen trajectories of uneven size in one launch, graph-replayed.
        _case("batched_16_f32", "batched", 512, 512, 64, density="gauss", pin=False, B=16,
              min_shots=32),
        # Multi-shot projection at high resolution: the largest pattern.
        _case("project_hr_f32", "project", 4096, 2560, 1, perturb=0.05),
        # Multi-shot projection, FP64 samples, the paper's 127 shots and 200
        # iterations, shots of odd length.
        _case("project_f64", "project", 127, 2047, 1, dtype="f64", n_iter=200, perturb=0.05),
        # A step on the fast summations at 1e6 samples (field + mesh).
        _case("fast_step_1m_f32", "step", 2048, 512, 192, mesh=128),
        # The fast gradient of the high-resolution pattern, 1e7 samples.
        _case("fast_grad_hr_f32", "grad", 4096, 2560, 256, mesh=256, perturb=0.375),
        # Algorithm 1 from a quarter of the resolution, fixed steps and then
        # Barzilai-Borwein, on a small pattern.
        _case("multires_small_f32", "multires", 32, 256, 32, levels=2, n_git=22, n_fixed=20),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    """One more case: an operation, and sizes spread over its range.  FP64
    samples are drawn where the FP64 step and projection carry them; sums over
    pairs are FP32 for every sample type, so their own outputs are drawn in
    FP32, and a step's only where 1/N times a sum is small beside a sample."""
    op = rng.choice(["grad", "step", "step", "energy", "batched", "project", "fast", "multires"])
    dtype = rng.choice(["f32", "f32", "f64"])
    acc = rng.choice(["kahan", "fp64"])
    density = rng.choice(["power", "gauss"])
    pin = rng.random() < 0.6
    if op == "project":
        Nc, Ns = _log(rng, 1, 2047), _log(rng, 16, 3072)
        return _case(None, op, Nc, Ns, 1, dtype=dtype, pin=pin, perturb=0.05,
                     n_iter=rng.choice([50, 100, 200]), mixed=dtype == "f32" and rng.random() < 0.2)
    if op == "multires":
        Ns = 4 * _log(rng, 16, 64)
        return _case(None, op, _log(rng, 8, 40), Ns, _log(rng, 16, 40), acc=acc,
                     density=density, pin=pin, levels=rng.choice([1, 2]),
                     n_git=rng.choice([4, 8, 12]), n_fixed=20)
    if op == "batched":
        B = _log(rng, 2, 16)
        Ns = rng.choice([256, 384, 500, 512])
        return _case(None, op, _log(rng, 32, 400), Ns, _log(rng, 24, 64), dtype=dtype, acc=acc,
                     density="gauss", pin=pin, B=B, min_shots=8)
    if op == "fast":
        Nc, Ns = _log(rng, 64, 2048), _log(rng, 128, 1024)
        mesh = max(24, min(160, int(round(1.2 * (Nc * Ns) ** (1.0 / 3.0)))))
        return _case(None, rng.choice(["grad", "step"]), Nc, Ns, _log(rng, 32, 160), density=density,
                     pin=pin, mesh=mesh, perturb=rng.choice([0.0, 0.3]))
    nx = _log(rng, 16, 120)
    ny, nz = (max(8, int(nx * rng.uniform(0.6, 1.2))) for _ in range(2))
    Nc, Ns = _log(rng, 8, 384), _log(rng, 33, 1024)
    while Nc * Ns * (nx * ny * nz + Nc * Ns) > 3e11:      # at most about half the medium step
        Nc = max(8, Nc // 2)
        nx = max(16, nx - 8)
    if op != "step" or Nc * Ns < 4096:
        dtype = "f32"
    mixed = op == "step" and dtype == "f32" and rng.random() < 0.2
    return _case(None, op, Nc, Ns, (nx, ny, nz), dtype=dtype, acc=acc, density=density, pin=pin,
                 eps=rng.choice([0.0, 0.0, 1e-3]), mixed=mixed)


# --- inputs --------------------------------------------------------------------


def _dt(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _alpha_beta(Ns):
    return 1.0 / (2.0 * Ns), 1.0 / (8.0 * Ns * Ns)


def _spokes(Nc, Ns, gen, perturb, scale=1.0):
    """Golden-angle radial spokes with jitter, float64 [Nc * Ns, 3]."""
    i = torch.arange(Nc, dtype=torch.float64, device="cuda")
    z = (i + 0.5) / Nc
    phi = i * (math.pi * (3.0 - math.sqrt(5.0)))
    rxy = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    u = torch.stack([rxy * torch.cos(phi), rxy * torch.sin(phi), z], 1)
    radius = 0.95 * scale * _alpha_beta(Ns)[0] * (Ns - 1) / 2.0
    t = radius * (2.0 * torch.arange(Ns, dtype=torch.float64, device="cuda") / max(Ns - 1, 1) - 1.0)
    K = u[:, None, :] * t[None, :, None]
    K += 1e-3 * torch.randn(K.shape, generator=gen, dtype=torch.float64, device="cuda")
    if perturb:
        K += perturb * (2.0 * torch.rand(K.shape, generator=gen, dtype=torch.float64,
                                         device="cuda") - 1.0)
    return K.clamp_(-0.5, 0.5).reshape(Nc * Ns, 3)


def _density(case, n, sigma=0.15, floor=0.05):
    """[nz, ny, nx] float32, sum 1: inverse power with a plateau, or Gaussian."""
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m - 0.5 for m in n]
    r2 = ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2
    if case["density"] == "power":
        rho = 1.0 / torch.clamp(r2, min=1.0 / max(n) ** 2)
    else:
        rho = torch.exp(-r2 / (2.0 * sigma * sigma)) + floor
    return (rho / rho.sum()).float().contiguous()


def _inputs(case, seed):
    """Everything random or derived that both prepare() and exact() need."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    Nc, Ns, op = case["Nc"], case["Ns"], case["op"]
    n = (case["nx"], case["ny"], case["nz"])
    a, b = _alpha_beta(Ns)
    s = {}
    if op == "batched":
        rng = np.random.default_rng(seed)
        # sizes and options belong to the case; positions come from the seed
        shots = np.random.default_rng(Nc * 131 + case["B"]).integers(case["min_shots"], Nc + 1,
                                                                     size=case["B"])
        s["off"] = [0] + [int(v) * Ns for v in np.cumsum(shots)]
        s["K"] = torch.cat([_spokes(int(c), Ns, gen, case["perturb"]) for c in shots])
        s["rho"] = [_density(case, n, float(rng.uniform(0.1, 0.3)), 0.0) for _ in shots]
        s["eta"] = [1.0 / (int(c) * Ns) for c in shots]
        s["cons"] = [(a * float(rng.uniform(0.5, 1.5)), b * float(rng.uniform(0.5, 1.5)))
                     for _ in shots]
        s["K"] = s["K"].to(_dt(case)).contiguous()
        return s
    if op == "multires":
        Ns0 = Ns >> case["levels"]
        # the coarse samples of the same spokes
        s["K"] = _spokes(Nc, Ns0, gen, case["perturb"])
    else:
        s["K"] = _spokes(Nc, Ns, gen, case["perturb"])
    s["K"] = s["K"].to(_dt(case)).contiguous()
    if op != "project":
        s["rho"] = [_density(case, n)]
    s["eta"] = [1.0 / (Nc * Ns)]
    s["cons"] = [(a, b)]
    return s


def _acc(case):
    return sp.ACC_FP64 if case["acc"] == "fp64" else sp.ACC_KAHAN32


def _pin(case):
    return case["Ns"] // 2 if case["pin"] else -1


def prepare(case, seed):
    s = _inputs(case, seed)
    ctx = sp.sparkling_create(0)
    if case["mixed"]:
        sp.sparkling_set_projection(ctx, sp.PROJECTION_MIXED)
    if case["eps"]:
        sp.sparkling_set_regularisation(ctx, case["eps"])
    s.update(case=case, ctx=ctx, acc=_acc(case))
    s["grids"] = [sp.make_grid(r) for r in s.get("rho", [])]
    s["projs"] = [sp.make_proj(a, b, 0.5, case["n_iter"], _pin(case)) for a, b in s["cons"]]
    if case["mesh"]:
        sp.sparkling_set_attraction(ctx, sp.ATTRACTION_FIELD)
        sp.sparkling_set_repulsion(ctx, sp.REPULSION_MESH, sp.make_mesh(case["mesh"]))
        sp.sparkling_attraction_field(ctx, s["grids"][0])
    op = case["op"]
    if op == "grad":
        s["out"] = [torch.empty_like(s["K"]) for _ in range(3)]
    elif op == "project":
        s["work"] = torch.empty_like(s["K"])
    elif op == "multires":
        s["work"] = torch.empty(case["Nc"] * case["Ns"], 3, dtype=s["K"].dtype, device="cuda")
        s["sched"] = sp.make_schedule(s["eta"][0], case["n_git"], case["n_fixed"])
    elif op == "energy":
        s["K"].requires_grad_(True)
    return s


def run(s):
    case, ctx, K = s["case"], s["ctx"], s["K"]
    op, Nc, Ns = case["op"], case["Nc"], case["Ns"]
    if op == "grad":
        G, A, R = s["out"]
        sp.sparkling_grad(ctx, K, s["grids"][0], s["acc"], G, A, R)
        return {"G": G, "A": A, "R": R}
    if op == "step":
        sp.sparkling_step(ctx, K, Nc, Ns, s["grids"][0], s["eta"][0], s["projs"][0], s["acc"])
        return K
    if op == "energy":
        loss = sp.sparkling_energy_fn(K, s["rho"][0], ctx, acc=s["acc"]).to(K.dtype)
        (dK,) = torch.autograd.grad(loss, K)
        return {"F": loss.detach(), "dK": dK}
    if op == "batched":
        sp.sparkling_step_batched(ctx, K, s["off"], Ns, s["grids"], s["eta"], s["projs"], s["acc"])
        return K
    if op == "project":
        s["work"].copy_(K)
        sp.sparkling_project(ctx, s["work"], Nc, Ns, s["projs"][0])
        return s["work"]
    if op == "multires":
        s["work"][:K.shape[0]].copy_(K)
        sp.sparkling_multires(ctx, s["work"], Nc, Ns, s["grids"][0], s["projs"][0], s["sched"],
                              case["levels"], s["acc"])
        return s["work"]
    raise ValueError(op)


# --- what a pass cannot do without -----------------------------------------------

_ATTR_FLOPS = 9.0       # dx, r2 (fma), rsqrt, rho *, sum, fma; dy and dz are shared by a grid row
_REP_FLOPS = 22.0       # per unordered pair: 3 sub, 3 fma, rsqrt, 3 + 3 fma
_PROJ_FLOPS = 85.0      # per sample and FISTA iteration


def _shots(case):
    if case["op"] != "batched":
        return [case["Nc"]]
    return [int(v) for v in np.random.default_rng(case["Nc"] * 131 + case["B"]).integers(
        case["min_shots"], case["Nc"] + 1, size=case["B"])]


def _eval_flops(case, N):
    P = case["nx"] * case["ny"] * case["nz"]
    if case["mesh"]:
        M = case["mesh"]
        # interpolation, spreading and gathering, four transforms, near pairs
        near = 4.0 / 3.0 * math.pi * (10.0 / M) ** 3 * N
        return N * (60.0 + 64 * 8 + min(near, N) * 12) + 4 * 2.5 * 8 * M ** 3 * math.log2(8 * M ** 3)
    return _ATTR_FLOPS * N * P + _REP_FLOPS * N * (N - 1) / 2


def work(case):
    es = 4 if case["dtype"] == "f32" else 8
    P = case["nx"] * case["ny"] * case["nz"]
    op, Ns = case["op"], case["Ns"]
    b = f = 0.0
    for Nc in _shots(case):
        N = Nc * Ns
        k = 3.0 * es * N
        grid = 16.0 * P if case["mesh"] else 4.0 * P
        if case["mesh"]:
            grid += 3 * 4.0 * (2 * case["mesh"]) ** 3
        if op == "grad":
            b += 4 * k + grid
            f += _eval_flops(case, N)
        elif op in ("step", "batched"):
            b += 2 * k + grid
            f += _eval_flops(case, N) + _PROJ_FLOPS * N * case["n_iter"]
        elif op == "energy":
            b += 2 * k + grid
            f += _eval_flops(case, N) + 8.0 * N * P + 10.0 * N * (N - 1) / 2
        elif op == "project":
            b += 2 * k
            f += _PROJ_FLOPS * N * case["n_iter"]
        elif op == "multires":
            for l in range(case["levels"], -1, -1):
                n = Nc * (Ns >> l)
                b += case["n_git"] * (2 * 3.0 * es * n + grid)
                f += case["n_git"] * (_eval_flops(case, n) + _PROJ_FLOPS * n * case["n_iter"])
    return {"bytes": b, "flops": f}


# --- the same in 64 bits -----------------------------------------------------------

_CHUNK = 1 << 27        # pair terms held at a time
_MOST_PAIRS = 1.0e11    # beyond this exact() would take too long


def _forces64(K, rho, eps, energy=False):
    """(A, R, sum_q rho |d|, sum_j |d|) of every sample, direct sums."""
    N = K.shape[0]
    nz, ny, nx = rho.shape
    ax = [(torch.arange(m, dtype=torch.float64, device="cuda") + 0.5) / m - 0.5
          for m in (nx, ny, nz)]
    w0 = rho.double().reshape(1, nz * ny, nx)
    A, R = torch.empty_like(K), torch.empty_like(K)
    ea = torch.zeros(N, dtype=torch.float64, device="cuda")
    er = torch.zeros_like(ea)

    def inverse(r2):
        w = r2.rsqrt()
        return w if eps > 0 else w.nan_to_num_(posinf=0.0)

    step = max(1, _CHUNK // (nx * ny * nz))
    for i in range(0, N, step):
        k = K[i:i + step]
        dx, dy, dz = (k[:, c, None] - ax[c][None, :] for c in range(3))
        yz = (dz[:, :, None] ** 2 + dy[:, None, :] ** 2).reshape(-1, nz * ny) + eps * eps
        r2 = yz[:, :, None] + (dx ** 2)[:, None, :]
        if energy:
            ea[i:i + step] = (r2.sqrt() * w0).sum((1, 2))
        w = inverse(r2).mul_(w0)
        A[i:i + step, 0] = (w.sum(1) * dx).sum(1)
        wyz = w.sum(2).reshape(-1, nz, ny)
        A[i:i + step, 1] = (wyz.sum(1) * dy).sum(1)
        A[i:i + step, 2] = (wyz.sum(2) * dz).sum(1)
        del r2, w
    step = max(1, _CHUNK // N)
    for i in range(0, N, step):
        d = [K[i:i + step, c, None] - K[None, :, c] for c in range(3)]
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + eps * eps
        if energy:
            er[i:i + step] = r2.sqrt().sum(1) - eps
        w = inverse(r2)
        for c in range(3):
            R[i:i + step, c] = (w * d[c]).sum(1) / N
        del d, r2, w
    return A, R, ea, er


def _project64(K, Nc, Ns, alpha, beta, n_iter, pin):
    """Dual FISTA of the amplitude, slew, box and pin constraints."""
    k = K.reshape(Nc, Ns, 3)
    tau = 1.0 / 20.0
    y1 = torch.zeros(Nc, max(Ns - 1, 0), 3, dtype=torch.float64, device="cuda")
    y2 = torch.zeros(Nc, max(Ns - 2, 0), 3, dtype=torch.float64, device="cuda")
    q1, q2 = y1.clone(), y2.clone()

    def primal(d1, d2):
        s = k.clone()
        if Ns > 1:
            s[:, 1:] -= d1
            s[:, :-1] += d1
        if Ns > 2:
            s[:, 2:] -= d2
            s[:, 1:-1] += 2.0 * d2
            s[:, :-2] -= d2
        s.clamp_(-0.5, 0.5)
        if pin >= 0:
            s[:, pin] = 0.0
        return s

    def prox(z, r):
        n = torch.linalg.vector_norm(z, dim=2, keepdim=True)
        return z * torch.where(n > r, 1.0 - r / n, torch.zeros_like(n))

    t = 1.0
    for _ in range(n_iter):
        s = primal(y1, y2)
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        m = (t - 1.0) / tn
        t = tn
        if Ns > 1:
            n1 = prox(y1 + tau * (s[:, 1:] - s[:, :-1]), tau * alpha)
            y1, q1 = n1 + m * (n1 - q1), n1
        if Ns > 2:
            n2 = prox(y2 + tau * (s[:, 2:] - 2.0 * s[:, 1:-1] + s[:, :-2]), tau * beta)
            y2, q2 = n2 + m * (n2 - q2), n2
    return primal(q1, q2).reshape(Nc * Ns, 3)


def _upsample64(K, Nc, d):
    c = K.reshape(Nc, d, 3)
    f = torch.empty(Nc, 2 * d, 3, dtype=torch.float64, device="cuda")
    f[:, 0::2] = c
    f[:, 1:-1:2] = 0.5 * (c[:, 1:] + c[:, :-1])
    f[:, -1] = c[:, -1] + (0.5 * (c[:, -1] - c[:, -2]) if d > 1 else 0.0)
    return f.reshape(Nc * 2 * d, 3)


def exact(case, seed):
    s = _inputs(case, seed)
    op, Nc, Ns, eps = case["op"], case["Nc"], case["Ns"], case["eps"]
    P = case["nx"] * case["ny"] * case["nz"]
    if op != "project" and sum(c * Ns * (P + c * Ns) for c in _shots(case)) > _MOST_PAIRS:
        return None
    K = s["K"].double()
    if op == "project":
        if Nc * Ns * case["n_iter"] > 2e9:
            return None
        return _project64(K, Nc, Ns, *s["cons"][0], case["n_iter"], _pin(case))
    if op == "grad":
        A, R, _, _ = _forces64(K, s["rho"][0], eps)
        return {"G": A - R, "A": A, "R": R}
    if op == "energy":
        A, R, ea, er = _forces64(K, s["rho"][0], eps, energy=True)
        N = K.shape[0]
        return {"F": ea.sum() / N - er.sum() / (2.0 * N * N), "dK": (A - R) / N}
    if op in ("step", "batched"):
        off = s.get("off", [0, Nc * Ns])
        out = []
        for t in range(len(off) - 1):
            k = K[off[t]:off[t + 1]]
            A, R, _, _ = _forces64(k, s["rho"][t], eps)
            out.append(_project64(k - s["eta"][t] * (A - R), k.shape[0] // Ns, Ns, *s["cons"][t],
                                  case["n_iter"], _pin(case)))
        return torch.cat(out)
    if op == "multires":
        a, b = s["cons"][0]
        pin = _pin(case)
        for l in range(case["levels"], -1, -1):
            nl, eta = Ns >> l, s["eta"][0]
            Kp = Gp = None
            for t in range(case["n_git"]):
                A, R, _, _ = _forces64(K, s["rho"][0], eps)
                G = A - R
                if t >= case["n_fixed"] and t > 0:
                    ds, dy = K - Kp, G - Gp
                    ss, sy = float((ds * ds).sum()), float((ds * dy).sum())
                    if sy > 0:
                        eta = min(max(ss / sy, 1e-12), 1e3)
                Kp, Gp = K, G
                K = _project64(K - eta * G, Nc, nl, a * 2.0 ** l, b * 4.0 ** l, case["n_iter"],
                               pin >> l if pin >= 0 else -1)
                if case["dtype"] == "f32":      # the samples are kept in 32 bits between steps
                    K = K.float().double()
            if l > 0:
                K = _upsample64(K, Nc, nl)
                if case["dtype"] == "f32":
                    K = K.float().double()
        return K
    raise ValueError(op)
