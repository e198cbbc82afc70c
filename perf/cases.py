"""Performance cases of the coupled step: what a user of this framework has it do.

Each case goes through the public entry points of ``paper_2410_11129_gb300.fcd``
(``Channel``, ``Batch``, ``Tangent``, ``Adjoint`` and the C calls they wrap). A
case is a dict of plain values; the seed varies the droplet's place, the capillary
and magnetic Bond numbers and the field angle around the case's own.

``exact`` restates the paper's step (arXiv 2410.11129, Secs. 2.1-2.5) in plain
torch float64 on the device: the potential by conjugate gradients with a
constant-permeability Fourier preconditioner, gradients by torch.autograd.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2410_11129_gb300 import fcd

# ------------------------------------------------------------------ the cases
DEVICE = "cuda"
PRE_STEPS = 6  # steps that prepare() takes: the calls measured come in the middle of a run


def _channel(kind, nx, ny, precision, tol, steps, ferro="shell", chi=1.0, r1=0.15, r2=0.3,
             Ca=0.15, Bo_m=2.0, alpha_deg=0.0, ratio=1.0, xi=5.0, eps_n=1e-4, open_x=0, count=1,
             topology="partial", **more):
    return dict(kind=kind, nx=nx, ny=ny, precision=precision, tol=tol, steps=steps, ferro=ferro,
                chi=chi, r1=r1, r2=r2, Ca=Ca, Bo_m=Bo_m, alpha_deg=alpha_deg, ratio=ratio, xi=xi,
                eps_n=eps_n, open_x=open_x, count=count, topology=topology, **more)


def listed():
    core = dict(ferro="core", chi=2.0, Ca=0.2, Bo_m=3.0, alpha_deg=90.0, ratio=2.0)
    return [
        # the 200x40 FP64 parity channel: the smallest run of the repository, all latency
        dict(_channel("step", 200, 40, "fp64", 1e-10, 10, Ca=0.1, Bo_m=1.0, xi=4.0, eps_n=1e-12),
             name="step-200x40-fp64"),
        # the FP64 channel whose runs the gradients differentiate (and finite differences repeat)
        dict(_channel("step", 800, 100, "fp64", 1e-10, 10, eps_n=1e-6), name="step-800x100-fp64"),
        # the FP32 production channel, state sampled every 50 steps
        dict(_channel("step", 1600, 200, "fp32", 1e-4, 50, **core), name="step-1600x200-fp32"),
        # the precision-study channel in the mass-conserving storage form
        dict(_channel("step", 2400, 300, "fp32_offset", 1e-4, 40, **core), name="step-2400x300-offset"),
        # the paper's own grid as an open channel (inlet, convective outlet)
        dict(_channel("step", 900, 150, "fp32", 1e-4, 50, r1=0.3 / 1.75, open_x=1), name="step-900x150-open-fp32"),
        # the largest grid: 2.5 GB of state, far outside L2
        dict(_channel("step", 9600, 1200, "fp32", 1e-3, 16, **core), name="step-9600x1200-fp32"),
        # a ragged lattice with the compensated potential (tolerance below 1e-4) and total spreading
        dict(_channel("step", 402, 123, "fp32_offset", 1e-5, 20, Bo_m=1.0, alpha_deg=30.0,
                      topology="non-engulfing"), name="step-402x123-pair-offset"),
        # a breakup watcher: a few steps, then the observables on the host
        dict(_channel("observe", 1600, 200, "fp32", 1e-4, 5, **core), name="observe-1600x200-fp32"),
        # a potential solve from nothing for given phase fields (a field study without flow)
        dict(_channel("solve", 800, 100, "fp64", 1e-10, 1, eps_n=1e-6), name="solve-800x100-fp64"),
        # a slice of the regime map: uneven channels advanced together
        dict(_channel("batch", 1600, 200, "fp32", 1e-4, 10, count=24), name="batch-24-fp32"),
        # forward-mode gradients along the four parameters
        dict(_channel("tangent", 800, 100, "fp64", 1e-10, 4, alpha_deg=20.0, eps_n=1e-6),
             name="tangent-800x100"),
        # reverse mode from a fresh context: forward pass with checkpoints, one sweep, all gradients
        dict(_channel("adjoint", 800, 100, "fp64", 1e-10, 20, alpha_deg=20.0, eps_n=1e-6,
                      checkpoint=10), name="adjoint-800x100"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["observe", "solve", "batch", "tangent", "adjoint"])
    ferro = rng.choice(["core", "shell"])
    common = dict(ferro=ferro, chi=rng.choice([0.5, 1.0, 2.0]), Ca=round(rng.uniform(0.08, 0.5), 3),
                  Bo_m=round(rng.uniform(0.5, 4.0), 2), alpha_deg=round(rng.uniform(0.0, 90.0), 1),
                  ratio=rng.choice([1.0, 2.0]), r2=0.3, r1=round(rng.uniform(0.13, 0.2), 3))
    if kind in ("tangent", "adjoint", "solve") or (kind == "step" and rng.random() < 0.3):
        ny = _log_int(rng, 36, 120)
        nx = 2 * _log_int(rng, 2 * ny, 4 * ny)
        steps = {"tangent": 3, "adjoint": rng.choice([8, 12, 16]), "solve": 1, "step": 10}[kind]
        more = {"checkpoint": rng.choice([4, 7, 20])} if kind == "adjoint" else {}
        return _channel(kind, nx, ny, "fp64", 1e-10, steps, xi=4.0, eps_n=1e-6,
                        open_x=int(kind != "solve" and rng.random() < 0.25), **common, **more)
    if kind == "batch":
        return _channel(kind, 2 * rng.randrange(400, 1200), rng.choice([100, 150, 200]), "fp32",
                        1e-4, 10, count=rng.randrange(4, 24), **common)
    ny = _log_int(rng, 40, 1000 if kind == "step" else 400)
    nx = 2 * _log_int(rng, 2 * ny, 4 * ny)
    tol = 1e-3 if ny > 400 else rng.choice([1e-4, 1e-4, 1e-5])
    common["topology"] = rng.choice(["partial", "partial", "non-engulfing"])
    return _channel(kind, nx, ny, rng.choice(["fp32", "fp32_offset"]), tol,
                    5 if kind == "observe" else (40 if ny < 350 else 12),
                    xi=4.0 if ny < 60 else 5.0, open_x=int(rng.random() < 0.25), **common)


# ------------------------------------------------------------- from case to run
def _config(case, seed, index=0):
    """The parameter dictionary of fcd.make_params for this case and seed (instance
    `index` of a batch: its own length and Bo_m x Ca point)."""
    rng = np.random.default_rng([int(seed) & 0xffffffff, index])
    jitter = lambda spread: 1.0 + spread * rng.uniform(-1.0, 1.0)
    nx, ny = case["nx"], case["ny"]
    Ca, Bo = case["Ca"] * jitter(0.05), case["Bo_m"] * jitter(0.05)
    if case["kind"] == "batch":
        nx = int(nx * (0.5 + (0.618034 * index) % 1.0)) // 32 * 32  # uneven lengths, the same for every seed
        Ca, Bo = rng.uniform(0.05, 0.6), rng.choice([0.5, 1.0, 2.0, 4.0, 8.0])
    r1, r2 = case["r1"] * ny, case["r2"] * ny
    chi = [0.0, 0.0, 0.0]
    chi[0 if case["ferro"] == "core" else 1] = case["chi"]
    cfg = dict(nx=nx, ny=ny, rho=[1.0, 1.0 / case["ratio"], 1.0],
               nu=[1 / 6, 1 / 6 / case["ratio"], 1 / 6], chi=chi, mobility=0.3, xi=case["xi"],
               eta=0.0, Ca=Ca, Bo_m=Bo, alpha=math.radians(case["alpha_deg"] + 5.0 * rng.uniform(-1, 1)),
               r1=r1, r2=r2, xc=1.2 * r2 + 0.2 * r2 * rng.uniform(0, 1) + 8.0,
               yc=0.5 * (ny - 1) + 0.03 * ny * rng.uniform(-1, 1), s13_over_s12=1.0, s23_over_s12=1.0,
               sigma23=0.0, u_max=0.01, ferro_phase=1 if case["ferro"] == "core" else 2,
               precision=case["precision"], mag_tol=case["tol"], mag_max_iter=200,
               eps_n=case["eps_n"], open_x=case["open_x"])
    if case["topology"] == "non-engulfing":  # Table 2 ratios; total spreading needs eta > 0
        cfg.update(s13_over_s12=0.3, s23_over_s12=0.3)
        cfg["eta"] = cfg["rho"][2] * cfg["nu"][2] * (2 * cfg["u_max"] / 3) / Ca / 0.3
    return cfg


def _populations(ch):
    """The populations (f 9 planes, g 18) in the FP64 exchange layout, on the device."""
    out = torch.empty((27, ch.ny, ch.nx), dtype=torch.float64, device=DEVICE)
    at = lambda plane: ctypes.c_void_p(out[plane].data_ptr())
    ch.check(fcd.load().fcd_get_populations(ch.h, at(0), at(9), None))
    return out


def _kept(case, pops):
    """What a program keeps of them: the context's own precision."""
    return pops if case["precision"] == "fp64" else pops.float()


OBSERVED = ("T_o", "T_i", "lx_o", "ly_o", "lx_i", "ly_i", "xc_core", "yc_core", "xc_shell", "yc_shell")


def prepare(case, seed):
    kind = case["kind"]
    cfg = _config(case, seed)
    state = {"case": dict(case), "cfg": cfg}
    if kind == "batch":
        state["batch"] = fcd.Batch([_config(case, seed, i) for i in range(case["count"])])
        state["batch"].step(PRE_STEPS + 2)  # the steps in which a batch times its two modes, and two more
    elif kind == "tangent":
        state["ch"] = fcd.Tangent(cfg)
        state["ch"].step(PRE_STEPS)
    elif kind != "adjoint":
        state["ch"] = fcd.Channel(cfg)
        state["ch"].step(PRE_STEPS)
    if kind == "solve":
        pops = _populations(state["ch"])
        state["f"], state["g"], state["psi"] = pops[:9].contiguous(), pops[9:].contiguous(), torch.zeros_like(pops[0])
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    ch = state.get("ch")
    if kind == "step":
        ch.step(case["steps"])
        return _kept(case, _populations(ch))
    if kind == "observe":
        ch.step(case["steps"])
        o = ch.observe(allow=(fcd.FCD_ENOCONV,))
        # mag_iters and mag_resid describe the solver's path, not the state
        return {"mass": np.array(o["mass"], np.float32), "shape": np.array([o[k] for k in OBSERVED], np.float32),
                "breakup": o["breakup"], "b_step": o["b_step"]}
    if kind == "solve":
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())
        ch.check(fcd.load().fcd_set_populations(ch.h, ptr(state["f"]), ptr(state["g"]), ptr(state["psi"]), PRE_STEPS))
        ch.solve_magnetic()
        return ch.field("psi", out=torch.empty((ch.ny, ch.nx), dtype=torch.float64, device=DEVICE))
    if kind == "batch":
        state["batch"].step(case["steps"])
        # the instances write from their own streams: convert once all of them have
        pops = [_populations(inst) for inst in state["batch"].instances]
        return [_kept(case, p) for p in pops]
    if kind == "tangent":
        ch.step(case["steps"])
        o = ch.tangent_observe(allow=(fcd.FCD_ENOCONV,))
        return {"values": np.array([o["T_o"], o["overlap"], o["lx_o"], o["ly_o"]]),
                **{k: np.array(o[k]) for k in ("dT_o", "doverlap", "dlx_o", "dly_o")}}
    adj = fcd.Adjoint(state["cfg"], case["checkpoint"])
    try:
        adj.step(case["steps"])
        o = adj.gradient(1.0, 0.01, initial=True, allow=(fcd.FCD_ENOCONV,))
    finally:
        adj.close()
    # dg0 in single precision: in the bulk phi sits on an edge of its clamp up to round-off (0 or 1
    # +- 1e-17), where the derivative is that of either side (about 3e-7 of dg0's norm)
    return {"values": np.array([o["T_o"], o["overlap"]]), "grad": np.array(o["grad"]),
            "df0": o["df0"], "dg0": o["dg0"].astype(np.float32)}


def work(case):
    """Each step reads and writes the 27 populations and the potential once, and computes the
    collision of a node in about 770 operations (as many again, five times over, for the values
    with four derivatives; about twice as many for its reverse); then the outputs."""
    size = 8 if case["precision"] == "fp64" else 4
    nodes = case["nx"] * case["ny"] * case["count"]
    kind, steps = case["kind"], case["steps"]
    if kind == "solve":  # phases from the populations, psi' in and out; ten residuals and sweeps
        return {"bytes": 20.0 * 8 * nodes, "flops": 400.0 * nodes}
    per_step = 56.0 * size * nodes
    bytes_, flops = per_step * steps, 770.0 * nodes * steps
    if kind == "tangent":
        bytes_, flops = 5 * bytes_, 5 * flops
    elif kind == "adjoint":  # forward, the states kept and read, and the reverse steps
        bytes_, flops = 3 * bytes_, 3 * flops
    elif kind == "observe":
        bytes_ += 18.0 * size * nodes
    else:
        bytes_ += 27.0 * 2 * size * nodes
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------------ exact
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _shift(v, a, odd=False, clamp_x=False):
    """v at the node + e_a: mirrored rows beyond the walls (negated where odd), periodic or
    mirrored columns."""
    if EY[a]:
        edge = v[-1:] if EY[a] > 0 else v[:1]
        edge = -edge if odd else edge
        v = torch.cat([v[1:], edge]) if EY[a] > 0 else torch.cat([edge, v[:-1]])
    if EX[a] and clamp_x:
        return torch.cat([v[:, 1:], v[:, -1:]], 1) if EX[a] > 0 else torch.cat([v[:, :1], v[:, :-1]], 1)
    return torch.roll(v, -EX[a], 1) if EX[a] else v


def _grad(v, **kw):
    n = [_shift(v, a, **kw) for a in range(9)]
    return (3 * sum(WT[a] * EX[a] * n[a] for a in range(9) if EX[a]),
            3 * sum(WT[a] * EY[a] * n[a] for a in range(9) if EY[a]),
            6 * sum(WT[a] * (n[a] - v) for a in range(1, 9)))


def _operator(k, psi):
    return sum(3 * WT[a] * (k + _shift(k, a)) * (_shift(psi, a, odd=True) - psi) for a in range(1, 9))


def _source(k, hx, hy):
    """-L psi0 for psi0 = -(hx x + hy y)."""
    return sum(3 * WT[a] * (k + _shift(k, a)) * (EX[a] * hx + EY[a] * hy) for a in range(1, 9))


def _solve(k, b, x=None, tol=1e-14):
    """L(k) x = b by conjugate gradients on -L, preconditioned with the operator of uniform k
    (diagonal in a Fourier basis along x and the sines of the odd walls along y)."""
    ny, nx = k.shape
    tx = 2 * math.pi * torch.arange(nx // 2 + 1, device=k.device, dtype=k.dtype) / nx
    ty = math.pi * torch.arange(2 * ny, device=k.device, dtype=k.dtype) / ny
    cx, cy = torch.cos(tx)[None], torch.cos(ty)[:, None]
    lam = -6 * ((2 * cx + 2 * cy - 4) / 9 + (4 * cx * cy - 4) / 36)
    lam[0, 0] = 1.0

    def precondition(r):
        h = torch.fft.rfft2(torch.cat([r, -r.flip(0)]))
        h[0] = 0
        return torch.fft.irfft2(h / lam, s=(2 * ny, nx))[:ny]

    x = torch.zeros_like(b) if x is None else x
    r = _operator(k, x) - b
    stop = tol * float(b.abs().max())
    if stop == 0:
        return torch.zeros_like(b)
    z = precondition(r)
    p, rz, least, stale = z, (r * z).sum(), math.inf, 0
    for _ in range(200):
        q = -_operator(k, p)
        s = rz / (p * q).sum()
        x, r = x + s * p, r - s * q
        top = float(r.abs().max())
        stale = 0 if top < 0.5 * least else stale + 1
        least = min(least, top)
        if top <= stop or stale > 5 or not math.isfinite(top):
            break
        z = precondition(r)
        rz, old = (r * z).sum(), rz
        p = z + rz / old * p
    return x


class _Inverse(torch.autograd.Function):
    """L(k)^-1 r for fixed k (L is symmetric)."""

    @staticmethod
    def forward(ctx, r, k):
        ctx.save_for_backward(k)
        return _solve(k, r)

    @staticmethod
    def backward(ctx, g):
        return _solve(ctx.saved_tensors[0], g), None


def _potential(k, hx, hy, guess):
    with torch.no_grad():
        psi = _solve(k, _source(k, hx, hy), guess)
    if k.requires_grad or torch.is_tensor(hx) and hx.requires_grad:
        return psi + _Inverse.apply(_source(k, hx, hy) - _operator(k, psi), k.detach())
    return psi


def _constants(cfg, theta):
    """Lattice constants for theta = (Bo_m, Ca, alpha, nu_r) (Eqs. 14, 26-27, 40-41)."""
    bo, ca, alpha, nu_r = theta
    rho, chi, nu3 = cfg["rho"], cfg["chi"], cfg["nu"][2]
    s23 = rho[2] * nu3 * (2 * cfg["u_max"] / 3) / ca
    s12 = s23 / cfg["s23_over_s12"]
    s13 = cfg["s13_over_s12"] * s12
    if cfg["ferro_phase"] == 1:
        h2 = 2 * s12 * bo / (chi[0] * cfg["r1"])
    else:
        h2 = 2 * (s12 * cfg["r1"] + s23 * cfg["r2"]) * bo / (chi[1] * (cfg["r2"] ** 2 - cfg["r1"] ** 2))
    h = torch.sqrt(h2)
    return dict(s12=s12, s13=s13, s23=s23, gam=[s12 + s13 - s23, s12 + s23 - s13, s13 + s23 - s12],
                hx=h * torch.cos(alpha), hy=h * torch.sin(alpha), rho=rho, ik=[1 / (1 + c) for c in chi],
                tau=[3 * cfg["nu"][0], 3 * nu3 / nu_r, 3 * nu3], eta=cfg["eta"], xi=cfg["xi"],
                eps_n=cfg["eps_n"], om=1 / (0.5 + 3 * cfg["mobility"]), u_avg=2 * cfg["u_max"] / 3,
                G=0.0 if cfg["open_x"] else 8 * rho[2] * nu3 * cfg["u_max"] / cfg["ny"] ** 2)


def _gamma(ux, uy):
    uu = 1.5 * (ux * ux + uy * uy)
    eu = [3 * (EX[a] * ux + EY[a] * uy) for a in range(9)]
    return [WT[a] * (eu[a] + 0.5 * eu[a] ** 2 - uu) for a in range(9)]  # Gamma_a - w_a


def _start(cfg):
    """Concentric tanh profiles, Poiseuille flow, populations at equilibrium."""
    nx, ny = cfg["nx"], cfg["ny"]
    y = torch.arange(ny, dtype=torch.float64, device=DEVICE)[:, None]
    x = torch.arange(nx, dtype=torch.float64, device=DEVICE)[None]
    dx = x - cfg["xc"]
    dx = dx - nx * torch.floor(dx / nx + 0.5)
    r = torch.sqrt(dx * dx + (y - cfg["yc"]) ** 2)
    p1, po = (0.5 * (1 - torch.tanh(2 * (r - cfg[n]) / cfg["xi"])) for n in ("r1", "r2"))
    ux = (cfg["u_max"] * 4 * (y + 0.5) * (ny - 0.5 - y) / ny ** 2).expand(ny, nx)
    f = torch.stack(_gamma(ux, torch.zeros_like(ux)))
    wt = torch.tensor(WT, dtype=torch.float64, device=DEVICE)[:, None, None]
    return f, torch.stack([p1 * (f + wt), (po - p1) * (f + wt)])


def _clamp(p):
    return [q.clamp(0, 1) for q in p]


def _step(f, g, C, cfg, psi):
    """One coupled step; psi: the last potential (the solve's starting point)."""
    kw = dict(clamp_x=bool(cfg["open_x"]))
    p = [g[0].sum(0), g[1].sum(0)]
    p.append(1 - p[0] - p[1])
    h = _clamp(p)
    k = 1 / sum(C["ik"][i] * h[i] for i in range(3))
    psi = _potential(k, C["hx"], C["hy"], psi)
    d = [_grad(p[0], **kw), _grad(p[1], **kw)]
    d.append(tuple(-(u + v) for u, v in zip(*d)))
    gam, q3 = C["gam"], p[0] * p[1] * p[2]
    gp = sum(gam[i] * p[i] for i in range(3))
    sij = {(0, 1): C["s12"], (0, 2): C["s13"], (1, 2): C["s23"]}
    fx = fy = 0.0
    for i in range(3):  # Eqs. 25, 28, 36; the part common to all phases drops out of the sum
        j, m = [q for q in range(3) if q != i]
        dh = (2 * p[i] * (sij[min(i, j), max(i, j)] * p[j] ** 2 + sij[min(i, m), max(i, m)] * p[m] ** 2)
              + p[j] * p[m] * gp + gam[i] * q3 + 2 * C["eta"] * p[i] * p[j] ** 2 * p[m] ** 2)
        mu = 12 / C["xi"] * dh - 0.75 * C["xi"] * gam[i] * d[i][2]
        fx, fy = fx + mu * d[i][0], fy + mu * d[i][1]
    px, py, _ = _grad(psi, odd=True)
    hh = 0.5 * ((C["hx"] - px) ** 2 + (C["hy"] - py) ** 2)  # Eqs. 5, 7, 9
    fx = fx + hh * k * k * sum(C["ik"][i] * d[i][0] for i in range(3))
    fy = fy + hh * k * k * sum(C["ik"][i] * d[i][1] for i in range(3))
    rho = sum(C["rho"][i] * h[i] for i in range(3))
    rx, ry, _ = _grad(rho, **kw)
    ps = f.sum(0)
    jx = sum(EX[a] * f[a] for a in range(9) if EX[a])
    jy = sum(EY[a] * f[a] for a in range(9) if EY[a])
    fx, fy = fx - ps / 3 * rx + C["G"], fy - ps / 3 * ry
    tau = sum(C["tau"][i] * h[i] for i in range(3))
    s = 1 / (0.5 + tau)
    ux, uy = jx + fx / (2 * rho), jy + fy / (2 * rho)
    # stress of f - f^eq: rate s on its deviator, 1 on its trace (Eqs. 12-13)
    dev = _gamma(ux, uy)
    ne = [f[a] - (WT[a] * ps + dev[a]) for a in range(9)]
    xx, yy, xy = (sum(c[a] * ne[a] for a in range(9)) for c in (
        [v * v for v in EX], [v * v for v in EY], [u * v for u, v in zip(EX, EY)]))
    tr, dd = xx + yy, xx - yy
    fmx = -tau * ((0.5 * tr + 0.5 * s * dd) * rx + s * xy * ry)
    fmy = -tau * (s * xy * rx + (0.5 * tr - 0.5 * s * dd) * ry)
    fx, fy = fx + fmx, fy + fmy
    ux, uy = ux + fmx / (2 * rho), uy + fmy / (2 * rho)
    dev = _gamma(ux, uy)
    ne = [f[a] - (WT[a] * ps + dev[a]) for a in range(9)]
    dd = (ne[1] + ne[3]) - (ne[2] + ne[4])
    xy = (ne[5] + ne[7]) - (ne[6] + ne[8])
    post = []
    for a in range(9):
        v = WT[a] * ps + dev[a] + 0.5 * WT[a] * 3 * (EX[a] * fx + EY[a] * fy) / rho
        if a:
            v = v + 0.25 * (1 - s) * ((EX[a] ** 2 - EY[a] ** 2) * dd if a < 5 else EX[a] * EY[a] * xy)
        post.append(v)
    fn = _stream(post, cfg)
    # phase fields (Eqs. 29-31)
    n = []
    for i in range(3):
        m2 = d[i][0] ** 2 + d[i][1] ** 2
        size = torch.where(m2 > 0, torch.sqrt(torch.where(m2 > 0, m2, 1.0)), 0.0)
        t = 4 / C["xi"] * h[i] * (1 - h[i]) / (size + C["eps_n"])
        n.append((t * d[i][0], t * d[i][1]))
    om, gn = C["om"], []
    for i in range(2):
        qx = n[i][0] - sum(v[0] for v in n) / 3
        qy = n[i][1] - sum(v[1] for v in n) / 3
        gn.append(_stream([(1 - om) * g[i][a] + om * p[i] * (WT[a] + dev[a])
                           + (1 - 0.5 * om) * WT[a] * (EX[a] * qx + EY[a] * qy) for a in range(9)], cfg))
    gn = torch.stack(gn)
    if cfg["open_x"]:
        fn, gn = _open_ends(f, g, fn, gn, C, cfg)
    return fn, gn, psi


def _stream(post, cfg):
    """Push streaming with half-way bounce-back; populations leaving an open end are dropped."""
    out = []
    for a in range(9):
        v = post[a]
        if EX[a]:
            v = torch.roll(v, EX[a], 1)
            if cfg["open_x"]:
                keep = torch.ones(v.shape[1], dtype=v.dtype, device=v.device)
                keep[0 if EX[a] > 0 else -1] = 0
                v = v * keep
        if EY[a] > 0:  # the bottom row receives what was sent into the wall
            v = torch.cat([post[OPP[a]][:1], v[:-1]])
        elif EY[a] < 0:
            v = torch.cat([v[1:], post[OPP[a]][-1:]])
        out.append(v)
    return torch.stack(out)


def _open_ends(f, g, fn, gn, C, cfg):
    """Inlet of Eq. 37 (Zou-He, corners by both momenta) and the convective outlet."""
    ny = cfg["ny"]
    y = torch.arange(ny, dtype=torch.float64, device=f.device)
    u = cfg["u_max"] * 4 * (y + 0.5) * (ny - 0.5 - y) / ny ** 2
    l = [fn[a, :, 0] for a in range(9)]
    low, top = y == 0, y == ny - 1
    five = torch.where(top, l[4] - l[2] - l[6] + l[7] + l[8], l[7] + u / 6 - 0.5 * (l[2] - l[4]))
    eight = torch.where(low, l[2] - l[4] + l[5] + l[6] - l[7], l[6] + u / 6 + 0.5 * (l[2] - l[4]))
    five, eight = torch.where(low, l[5], five), torch.where(top, l[8], eight)
    one = torch.where(low | top, u + l[3] - five + l[6] + l[7] - eight, l[3] + 2 * u / 3)
    inlet = {1: one, 5: five, 8: eight}
    U, zero = C["u_avg"], torch.zeros_like(u)
    po, pb = f[:, :, -1].sum(0), fn[:, :, -2].sum(0)
    wall = {3: torch.zeros_like(low), 6: low, 7: top}  # from the wall, not through the outlet
    into = {5: low, 8: top, 1: torch.zeros_like(low)}

    def plane(v, first=None, last=None):
        cols = [v[:, :1] if first is None else first[:, None], v[:, 1:-1],
                v[:, -1:] if last is None else last[:, None]]
        return torch.cat(cols, 1)

    f2, g2 = [], [[], []]
    for a in range(9):
        last = None
        if a in wall:
            last = torch.where(wall[a], fn[a, :, -1], ((f[a, :, -1] - WT[a] * po)
                               + U * (fn[a, :, -2] - WT[a] * pb)) / (1 + U))
        f2.append(plane(fn[a], inlet.get(a), last))
        for i in range(2):
            first = torch.where(into[a], gn[i, a, :, 0], zero) if a in into else None
            last = torch.where(wall[a], gn[i, a, :, -1], (g[i, a, :, -1] + U * gn[i, a, :, -2])
                               / (1 + U)) if a in wall else None
            g2[i].append(plane(gn[i, a], first, last))
    return torch.stack(f2), torch.stack([torch.stack(v) for v in g2])


def _span(v):
    """Length between the first upward and the last downward crossing of 1/2 along dim 0 of a
    (n, columns) array, zero beyond its ends; 0 where it is not crossed."""
    z = torch.zeros_like(v[:1])
    a, b = torch.cat([z, v]), torch.cat([v, z])
    at = torch.arange(-1, v.shape[0], device=v.device, dtype=v.dtype)[:, None]
    up, down = (a < 0.5) & (b >= 0.5), (a >= 0.5) & (b < 0.5)
    big = float(v.shape[0] + 5)
    first = torch.where(up, at, big).argmin(0, keepdim=True)
    last = torch.where(down, at, -big).argmax(0, keepdim=True)
    some = up.any(0) & down.any(0)
    pick = lambda w, i: torch.gather(w, 0, i)[0]
    one = torch.ones_like(some, dtype=v.dtype)
    au, bu, ad, bd = pick(a, first), pick(b, first), pick(a, last), pick(b, last)
    lo = at[first[0], 0] + (0.5 - au) / torch.where(some, bu - au, one)
    hi = at[last[0], 0] + (ad - 0.5) / torch.where(some, ad - bd, one)
    return torch.where(some, hi - lo, torch.zeros_like(lo))


def _observe(g, cfg):
    """Masses, extents, deformations and centroids (Eq. 42), and the overlap sum phi_1 phi_3."""
    nx, ny = cfg["nx"], cfg["ny"]
    p1, p2 = g[0].sum(0), g[1].sum(0)
    p3 = 1 - p1 - p2
    core, shell = p1.clamp(0, 1), p1.clamp(0, 1) + p2.clamp(0, 1)
    cut = 0 if cfg["open_x"] else int(shell.detach().sum(0).argmin())
    x = torch.arange(nx, device=g.device, dtype=g.dtype)
    x = torch.where(x >= cut, x, x + nx)
    y = torch.arange(ny, device=g.device, dtype=g.dtype)
    out = {"mass": torch.stack([p1.sum(), p2.sum(), p3.sum()]), "overlap": (p1 * p3).sum()}
    for name, v in (("o", shell), ("i", core)):
        line = v[ny // 2] if ny % 2 else 0.5 * (v[ny // 2 - 1] + v[ny // 2])
        lx, ly = _span(torch.roll(line, -cut)[:, None])[0], _span(v).max()
        out["lx_" + name], out["ly_" + name], out["T_" + name] = lx, ly, (ly - lx) / (ly + lx)
        part = "shell" if name == "o" else "core"
        out["xc_" + part] = (v.sum(0) * x).sum() / v.sum() % nx
        out["yc_" + part] = (v.sum(1) * y).sum() / v.sum()
    return out


def _theta(cfg, grad=False):
    return torch.tensor([cfg["Bo_m"], cfg["Ca"], cfg["alpha"], cfg["nu"][2] / cfg["nu"][1]],
                        dtype=torch.float64, device=DEVICE, requires_grad=grad)


def _advance(cfg, steps, theta, f, g):
    C = _constants(cfg, theta)
    psi = None
    for _ in range(steps):
        f, g, psi = _step(f, g, C, cfg, None if psi is None else psi.detach())
    return f, g


def exact(case, seed):
    kind = case["kind"]
    cfg = _config(case, seed)
    total = PRE_STEPS + case["steps"]
    if case["nx"] * case["ny"] * total * case["count"] > 1.2e9:
        return None
    if kind in ("tangent", "adjoint"):
        theta = _theta(cfg, True)
        f0, g0 = _start(cfg)
        if kind == "tangent":
            o = _observe(_advance(cfg, total, theta, f0, g0)[1], cfg)
            names = ("T_o", "overlap", "lx_o", "ly_o")
            d = {"d" + n: torch.autograd.grad(o[n], theta, retain_graph=True)[0] for n in names}
            return {"values": torch.stack([o[n].detach() for n in names]), **d}
        f0.requires_grad_(True)
        g0.requires_grad_(True)
        o = _observe(_advance(cfg, case["steps"], theta, f0, g0)[1], cfg)
        dt, df, dg = torch.autograd.grad(o["T_o"] + 0.01 * o["overlap"], (theta, f0, g0))
        return {"values": torch.stack([o["T_o"].detach(), o["overlap"].detach()]), "grad": dt, "df0": df, "dg0": dg}
    with torch.no_grad():
        if kind == "batch":
            out = []
            for i in range(case["count"]):
                c = _config(case, seed, i)
                out.append(torch.cat([v.reshape(-1, c["ny"], c["nx"])
                                      for v in _advance(c, total + 2, _theta(c), *_start(c))]))
            return out
        f, g = _advance(cfg, PRE_STEPS if kind == "solve" else total, _theta(cfg), *_start(cfg))
        if kind == "solve":
            C = _constants(cfg, _theta(cfg))
            p = [g[0].sum(0), g[1].sum(0)]
            h = _clamp(p + [1 - p[0] - p[1]])
            k = 1 / sum(C["ik"][i] * h[i] for i in range(3))
            return _potential(k, C["hx"], C["hy"], None)
        if kind == "observe":
            o = _observe(g, cfg)
            return {"mass": o["mass"], "shape": torch.stack([o[n] for n in OBSERVED]), "breakup": None, "b_step": None}
        return torch.cat([f, g.reshape(18, *f.shape[1:])])
