"""Performance cases of the split-operator library, through its public Python entry points.

Three kinds of work are listed, each as a user's program does it:

* ``run``: one simulation on a handle that the program keeps.  A pass starts a run (the
  packet built by the library, or a stored spinor and its time), takes ``steps`` Strang
  steps with a read-out every ``obs_every`` steps (0: none) and fetches the final spinor;
  with ``densities`` it also fetches the momentum-space and y-integrated densities.
* ``batch``: independent simulations of mixed grids advanced together, as the surrogate's
  training data are generated: every member's packet, the steps, the read-outs, the
  members' spinors.
* ``train``: minibatch Adam steps of the surrogate network from given parameters, then the
  trained parameters, the losses and the predictions of a ragged held-out set.

``exact`` restates the method in 64-bit torch without the library.
"""
import math
import random

import numpy as np
import torch

from paper_2307_01571_gb300 import kd
from paper_2307_01571_gb300 import workloads as W

PREC = {"fp32": kd.KD_FP32, "fp64": kd.KD_FP64, "dw": kd.KD_DW}
REAL_BYTES = {"fp32": 4, "fp64": 8, "dw": 8}
UNITS = W.ATOMIC
WIDTHS = [5, 256, 256, 256, 4]   # the surrogate network
N_ROWS, N_HELD = 3686, 410       # 4096 solver runs split 90/10
BATCH_SHAPES = [(128, 128), (256, 128), (256, 256), (512, 256)]


def listed():
    return [
        # the smallest call: an interactive run of a few steps on a tiny grid
        dict(name="fp32_64x64", kind="run", prec="fp32", field="gauss", nx=64, ny=64, steps=20,
             obs_every=20, start="packet", densities=False),
        # a small production run (the plane-wave grid in the fast form)
        dict(name="fp32_128x128", kind="run", prec="fp32", field="gauss", nx=128, ny=128, steps=200,
             obs_every=100, start="packet", densities=False),
        # the paper's own grid (long rows, few of them), no read-outs on the way
        dict(name="fp32_2048x128", kind="run", prec="fp32", field="gauss", nx=2048, ny=128, steps=400,
             obs_every=0, start="packet", densities=False),
        # the benchmark workload's grid, field and read-out interval
        dict(name="fp32_1024x512", kind="run", prec="fp32", field="gauss", nx=1024, ny=512, steps=200,
             obs_every=100, start="spinor", densities=False),
        # a state larger than L2 (256 MiB): the largest grid the benchmark runs
        dict(name="fp32_4096x2048", kind="run", prec="fp32", field="gauss", nx=4096, ny=2048, steps=30,
             obs_every=0, start="spinor", densities=False),
        # the plain FP64 plane-wave run with all of its read-outs
        dict(name="fp64_128x128", kind="run", prec="fp64", field="plane", nx=128, ny=128, steps=200,
             obs_every=100, start="packet", densities=True),
        # the FP64 reference form of the benchmark workload
        dict(name="fp64_1024x512", kind="run", prec="fp64", field="gauss", nx=1024, ny=512, steps=20,
             obs_every=20, start="spinor", densities=False),
        # the FP64-accurate form on the grid of the on/off study of the longitudinal field
        dict(name="dw_2048x128", kind="run", prec="dw", field="gauss", nx=2048, ny=128, steps=50,
             obs_every=50, start="packet", densities=False),
        # the FP64-accurate form of the benchmark workload
        dict(name="dw_1024x512", kind="run", prec="dw", field="gauss", nx=1024, ny=512, steps=50,
             obs_every=50, start="spinor", densities=False),
        # many simulations at once: the solver behind the surrogate's training data
        dict(name="batch_16", kind="batch", members=16, steps=200, obs_every=100),
        # the surrogate's training at its default batch, on the CUDA cores
        dict(name="train_fp32_b256", kind="train", prec="fp32", batch=256, steps=16),
        # the surrogate's training at a large batch, on the tensor cores
        dict(name="train_bf16_b1024", kind="train", prec="bf16", batch=1024, steps=16),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.12:
        return dict(kind="batch", members=rng.randint(3, 16), steps=rng.randint(40, 160),
                    obs_every=rng.choice([0, 40]))
    if u < 0.28:
        return dict(kind="train", prec=rng.choice(["fp32", "bf16"]),
                    batch=int(round(math.exp(rng.uniform(math.log(32), math.log(1024))))),
                    steps=rng.randint(4, 16))
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "dw"])
    nx = 1 << rng.randint(6, 12 if prec == "fp32" else 11)
    ny = 1 << rng.randint(6, 11 if prec == "fp32" else 10)
    # point-steps of the listed cases of the same form: 250 M, 10 M and 26 M
    most = {"fp32": 240e6, "fp64": 10e6, "dw": 26e6}[prec] / (nx * ny)
    steps = int(max(4, math.exp(rng.uniform(math.log(4), math.log(max(5.0, min(400.0, most)))))))
    every = rng.choice([0, max(1, steps // 2), steps])
    return dict(kind="run", prec=prec, field=rng.choice(["gauss", "gauss", "gauss", "plane"]), nx=nx, ny=ny,
                steps=steps, obs_every=every, start=rng.choice(["packet", "spinor"]),
                densities=prec == "fp64" and rng.random() < 0.5)


# ------------------------------------------------------------------ the inputs -----
def _setup(rng, nx, ny, field):
    """Seeded field and packet on a box centred on the beam: nx/16 by ny/16 wavelengths up
    to the benchmark workload's 40 (80 for longer axes), waist a quarter of the box or so."""
    k, lam = W.laser(UNITS)
    lx = min(nx / 16.0, 40.0 if nx <= 1024 else 80.0)
    ly = min(ny / 16.0, 40.0) if ny != 128 or nx < 1024 else 40.0
    grid = W.Grid(nx, ny, -lx / 2 * lam, lx / 2 * lam, -ly / 2 * lam, ly / 2 * lam)
    w0 = max(2.0, rng.uniform(0.2, 0.35) * ly) * lam
    a0 = math.exp(rng.uniform(math.log(0.05), math.log(0.4)))
    gauss = field == "gauss"
    f = W.Field(kind=W.GAUSS if gauss else W.PLANE, longitudinal=1 if gauss else 0, a0=a0, k_L=k,
                epsilon=1.0 / (k * w0) if gauss else 0.0, env_T=0.0 if gauss else 200 * W.dt_of(UNITS),
                phase0=rng.uniform(0.0, 6.0), p_shift_x=0.0, p_shift_y=UNITS.mc,
                box_vy=UNITS.c / math.sqrt(2.0) if gauss else 0.0)
    hk = UNITS.hbar * k
    p = W.Packet(rng.uniform(-1.2, -0.8) * hk, UNITS.mc, rng.uniform(-0.1, 0.1) * lx * lam,
                 rng.uniform(-0.1, 0.1) * ly * lam, 2.0 * hk / min(lx, ly), rng.choice([1, -1]), 0)
    return grid, f, p


def _run_setup(case, seed):
    return _setup(random.Random(seed), case["nx"], case["ny"], case["field"])


def _batch_setup(case, seed):
    rng = random.Random(seed)
    # the same shapes in every batch of a size, so that a seed changes values and not work
    return [_setup(rng, *BATCH_SHAPES[i % 4], "gauss") for i in range(case["members"])]


def _train_arrays(case, seed):
    g = np.random.default_rng(seed)
    x = g.uniform(-1.7, 1.7, (N_ROWS + N_HELD, WIDTHS[0]))
    x[:, 4] = g.choice([-1.0, 1.0], N_ROWS + N_HELD)
    mix = g.standard_normal((WIDTHS[0], WIDTHS[-1])) / 2.0
    t = np.tanh(x @ mix) + 0.5 * np.sin(2.0 * x[:, :1]) * x[:, 1:2]
    parts = []
    for fi, fo in zip(WIDTHS[:-1], WIDTHS[1:]):
        lim = math.sqrt(6.0 / fi)
        parts += [g.uniform(-lim, lim, fo * fi), np.zeros(fo)]
    idx = g.integers(0, N_ROWS, (case["steps"], case["batch"])).astype(np.int32)
    return (x.astype(np.float32), t.astype(np.float32), np.concatenate(parts).astype(np.float32), idx)


def _lr(i):
    return 1e-5 * (1.0 - 0.01 * i)   # the tail of the cosine-decayed step size


# ---------------------------------------------------------------- the programs -----
def prepare(case, seed):
    if case["kind"] == "run":
        grid, f, p = _run_setup(case, seed)
        sim = kd.Sim(UNITS, grid, f, PREC[case["prec"]])
        dtype = torch.complex64 if case["prec"] == "fp32" else torch.complex128
        out = torch.empty(sim.shape, dtype=dtype, device="cuda")
        sim.init_packet(p)
        psi0 = sim.get_spinor(torch.empty_like(out)) if case["start"] == "spinor" else None
        return dict(case=case, sim=sim, packet=p, psi0=psi0, out=out, dt=W.dt_of(UNITS))
    if case["kind"] == "batch":
        setups = _batch_setup(case, seed)
        sims = [kd.Sim(UNITS, g, f, kd.KD_FP32) for g, f, _ in setups]
        for s in sims:
            s.autotune(W.dt_of(UNITS))
        outs = [torch.empty(s.shape, dtype=torch.complex64, device="cuda") for s in sims]
        return dict(case=case, sims=sims, packets=[p for _, _, p in setups], outs=outs,
                    batch=kd.Batch(sims), dts=[W.dt_of(UNITS)] * len(sims))
    x, t, p0, idx = _train_arrays(case, seed)
    net = kd.MLP(WIDTHS)
    net.set_precision(kd.KD_MLP_BF16 if case["prec"] == "bf16" else kd.KD_MLP_FP32)
    return dict(case=case, net=net, p0=p0, held=x[N_ROWS:], x=torch.from_numpy(x[:N_ROWS]).cuda(),
                t=torch.from_numpy(t[:N_ROWS]).cuda(), idx=torch.from_numpy(idx).cuda(),
                loss=torch.empty(case["steps"], dtype=torch.float32, device="cuda"))


def _records(obs, prec):
    """The read-outs of a run as a table, in the precision of the form that made them."""
    rows = [[o[k] for k in kd.OBS_FIELDS] for o in obs]
    return torch.tensor(rows, dtype=torch.float32 if prec == "fp32" else torch.float64)


def run(state):
    case = state["case"]
    if case["kind"] == "run":
        sim = state["sim"]
        if case["start"] == "packet":
            sim.init_packet(state["packet"])
        else:
            sim.set_spinor(state["psi0"])
            sim.set_time(0.0)
        obs = sim.step(state["dt"], case["steps"], obs_every=case["obs_every"])
        res = {"psi": sim.get_spinor(state["out"])}
        if obs:
            res["obs"] = _records(obs, case["prec"])
        if case["densities"]:
            res["momentum"] = sim.momentum_density()
            res["density_x"] = sim.density_x()
        return res
    if case["kind"] == "batch":
        for s, p in zip(state["sims"], state["packets"]):
            s.init_packet(p)
        obs = state["batch"].step(state["dts"], case["steps"], obs_every=case["obs_every"])
        res = {"psi": [s.get_spinor(o) for s, o in zip(state["sims"], state["outs"])]}
        if case["obs_every"]:
            res["obs"] = torch.stack([_records(o, "fp32") for o in obs])
        return res
    net, x, t, idx, loss = (state[k] for k in ("net", "x", "t", "idx", "loss"))
    net.set_params(state["p0"])
    for i in range(case["steps"]):
        net.train_step_gather(x.data_ptr(), t.data_ptr(), N_ROWS, idx[i].data_ptr(), case["batch"], _lr(i),
                              loss_dev=loss[i].data_ptr())
    return {"params": net.get_params(), "loss": loss, "held": net.forward(state["held"])}


# -------------------------------------------------------------------- the floor ----
def _run_work(nx, ny, steps, obs, real):
    """Two read-and-write sweeps of the four complex components per step (a 2D transform of
    a distributed state cannot do with fewer), the spinor in and out, one more read per
    read-out; 5 N log2 N per complex transform, forward and inverse, and the two factors."""
    pts = float(nx * ny)
    spinor = pts * 8 * real
    lg = math.log2(nx) + math.log2(ny)
    return {"bytes": spinor * (4.0 * steps + 2 + obs), "flops": pts * (steps * (40.0 * lg + 150.0) + obs * 20.0 * lg)}


def work(case):
    if case["kind"] == "run":
        n = case["steps"] // case["obs_every"] if case["obs_every"] else 0
        return _run_work(case["nx"], case["ny"], case["steps"], n, REAL_BYTES[case["prec"]])
    if case["kind"] == "batch":
        n = case["steps"] // case["obs_every"] if case["obs_every"] else 0
        parts = [_run_work(*BATCH_SHAPES[i % 4], case["steps"], n, 4) for i in range(case["members"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    mac = sum(a * b for a, b in zip(WIDTHS[:-1], WIDTHS[1:]))
    npar = mac + sum(WIDTHS[1:])
    row = 4.0 * (WIDTHS[0] + WIDTHS[-1]) + 4
    return {"bytes": case["steps"] * (24.0 * npar + case["batch"] * row) + N_HELD * row + 8.0 * npar,
            "flops": 2.0 * mac * (3.0 * case["steps"] * case["batch"] + N_HELD)}


# ------------------------------------------- the method in 64 bits, by torch alone ----
DEV = "cuda" if torch.cuda.is_available() else "cpu"
C128 = torch.complex128


def _momenta(n, length, shift):
    dp = UNITS.hbar * 2.0 * math.pi / length
    i = torch.arange(n, device=DEV, dtype=torch.float64)
    return dp * torch.where(i < n // 2, i, i - n), dp, shift


def _grids(grid, f):
    px, dpx, _ = _momenta(grid.nx, grid.x_max - grid.x_min, 0)
    py, dpy, _ = _momenta(grid.ny, grid.y_max - grid.y_min, 0)
    px, py = px[None, :].expand(grid.ny, grid.nx), py[:, None].expand(grid.ny, grid.nx)
    return px, py, px + f.p_shift_x, py + f.p_shift_y, dpx, dpy


def _bispinor(pix, piy, spin):
    """Normalised positive-energy bispinors for chi = (1, +-1)/sqrt 2, [ny][nx][4]."""
    c, mc2 = UNITS.c, UNITS.mc2
    e = torch.sqrt(mc2 * mc2 + c * c * (pix * pix + piy * piy))
    nrm = torch.sqrt((e + mc2) / (2.0 * e))
    chi = (math.sqrt(0.5), math.copysign(math.sqrt(0.5), spin))
    fac = c / (e + mc2) * nrm
    pm, pp = torch.complex(pix, -piy), torch.complex(pix, piy)
    return torch.stack([(nrm * chi[0]).to(C128), (nrm * chi[1]).to(C128), fac * chi[1] * pm, fac * chi[0] * pp], -1)


def _packet(grid, f, p):
    px, py, pix, piy, _, _ = _grids(grid, f)
    mag = torch.exp(-((pix - p.p0x) ** 2 + (piy - p.p0y) ** 2) / (4.0 * p.sigma_p ** 2))
    ph = -((p.r0x - grid.x_min) * px + (p.r0y - grid.y_min) * py) / UNITS.hbar
    phi = torch.polar(mag, ph)[..., None] * _bispinor(pix, piy, p.spin)
    psi = torch.fft.ifft2(phi, dim=(0, 1))
    cell = (grid.x_max - grid.x_min) / grid.nx * (grid.y_max - grid.y_min) / grid.ny
    return psi / torch.sqrt((psi.abs() ** 2).sum() * cell)


def _potential(grid, f, psi, t, tau):
    """exp(-i tau V/hbar) psi, V = -m c^2 alpha.a, a the sum of the two beams d = +-1."""
    x = (grid.x_min + (grid.x_max - grid.x_min) / grid.nx * torch.arange(grid.nx, device=DEV, dtype=torch.float64))[None, :]
    y = (grid.y_min + f.box_vy * t + (grid.y_max - grid.y_min) / grid.ny *
         torch.arange(grid.ny, device=DEV, dtype=torch.float64))[:, None]
    k, s = f.k_L, f.a0
    if f.env_T > 0.0:
        s *= math.sin(math.pi * t / f.env_T) ** 2 if 0.0 <= t <= f.env_T else 0.0
    wt = UNITS.c * k * t + f.phase0
    ax = torch.zeros((grid.ny, grid.nx), device=DEV, dtype=torch.float64)
    ay = torch.zeros_like(ax)
    for d in (-1.0, 1.0):
        if f.kind == W.PLANE:
            ay = ay - torch.sin(wt - d * k * x)
            continue
        w0 = 1.0 / (k * f.epsilon)
        xr = k * w0 * w0 / 2.0
        w = w0 * torch.sqrt(1.0 + (x / xr) ** 2)
        ph = wt - d * k * x + torch.atan(d * x / xr) - d * x * y * y / (xr * w * w)
        g = w0 / w * torch.exp(-y * y / (w * w))
        ay = ay - g * torch.sin(ph)
        if f.longitudinal:
            ax = ax - 2.0 * d * g * f.epsilon * (y / w) * torch.cos(ph + torch.atan(d * x / xr))
    ax, ay = s * ax, s * ay
    a = torch.sqrt(ax * ax + ay * ay)
    kap = tau * UNITS.mc2 / UNITS.hbar
    cos, sinc = torch.cos(kap * a), kap * torch.sinc(kap * a / math.pi)
    q1, q2 = torch.complex(sinc * ay, sinc * ax), torch.complex(-sinc * ay, sinc * ax)   # i s (a_x -+ i a_y)
    return torch.stack([cos * psi[..., 0] + q1 * psi[..., 3], cos * psi[..., 1] + q2 * psi[..., 2],
                        cos * psi[..., 2] + q1 * psi[..., 1], cos * psi[..., 3] + q2 * psi[..., 0]], -1)


def _observe(grid, f, p, psi, t):
    px, py, pix, piy, dpx, dpy = _grids(grid, f)
    cell = (grid.x_max - grid.x_min) / grid.nx * (grid.y_max - grid.y_min) / grid.ny
    phi = torch.fft.fft2(psi, dim=(0, 1))
    wgt = cell / (grid.nx * grid.ny)
    den = torch.stack([(phi.abs() ** 2).sum(-1)] +
                      [((_bispinor(pix, piy, s).conj() * phi).sum(-1).abs() ** 2) for s in (1, -1)], -1) * wgt
    hk = UNITS.hbar * f.k_L

    def window(pc, half):
        ix = torch.round(px / dpx) - math.floor((pc - f.p_shift_x) / dpx + 0.5)
        iy = torch.round(py / dpy) - math.floor((p.p0y - f.p_shift_y) / dpy + 0.5)
        m = (ix.abs() <= math.floor(half / dpx + 1e-9)) & (iy.abs() <= math.floor(half / dpy + 1e-9))
        return den[m]

    win, wdf, tgt = window(p.p0x, hk / 2), window(p.p0x + 2 * hk, hk / 2), window(p.p0x + 2 * hk, 0.0)
    norm = float((psi.abs() ** 2).sum() * cell)
    si, sd, mx = win.sum(0).tolist(), wdf.sum(0).tolist(), wdf.max(0).values.tolist()
    rec = [t, norm, si[0], sd[0], si[1], si[2], sd[1], sd[2], *mx, *tgt[0].tolist()]
    return rec, den


def _exact_run(grid, f, p, psi, steps, every):
    dt = W.dt_of(UNITS)
    px, py, pix, piy, _, _ = _grids(grid, f)
    c, mc2, hb = UNITS.c, UNITS.mc2, UNITS.hbar
    e = torch.sqrt(mc2 * mc2 + c * c * (pix * pix + piy * piy))
    phase = torch.polar(torch.ones_like(e), f.box_vy * py * dt / hb)
    cos, sin = torch.cos(e * dt / hb) * phase, -1j * torch.sin(e * dt / hb) / e * phase
    pm, pp = c * torch.complex(pix, -piy), c * torch.complex(pix, piy)
    rows = []
    for n in range(steps):
        phi = torch.fft.fft2(_potential(grid, f, psi, n * dt, dt / 2), dim=(0, 1))
        h = torch.stack([mc2 * phi[..., 0] + pm * phi[..., 3], mc2 * phi[..., 1] + pp * phi[..., 2],
                         pm * phi[..., 1] - mc2 * phi[..., 2], pp * phi[..., 0] - mc2 * phi[..., 3]], -1)
        psi = torch.fft.ifft2(cos[..., None] * phi + sin[..., None] * h, dim=(0, 1))
        psi = _potential(grid, f, psi, (n + 1) * dt, dt / 2)
        if every and (n + 1) % every == 0:
            rows.append(_observe(grid, f, p, psi, (n + 1) * dt)[0])
    return psi, rows


def _exact_train(case, seed):
    x, t, p0, idx = _train_arrays(case, seed)
    x, t = (torch.from_numpy(v).to(DEV, torch.float64) for v in (x, t))
    par = torch.from_numpy(p0).to(DEV, torch.float64)
    m1, m2, losses = torch.zeros_like(par), torch.zeros_like(par), []

    def forward(par, a):
        off = 0
        for i, (fi, fo) in enumerate(zip(WIDTHS[:-1], WIDTHS[1:])):
            w, b = par[off:off + fo * fi].view(fo, fi), par[off + fo * fi:off + fo * fi + fo]
            off += fo * fi + fo
            a = a @ w.T + b
            if i < len(WIDTHS) - 2:
                a = torch.nn.functional.gelu(a)
        return a

    for i in range(case["steps"]):
        rows = torch.from_numpy(idx[i].astype(np.int64)).to(DEV)
        q = par.clone().requires_grad_(True)
        loss = ((forward(q, x[rows]) - t[rows]) ** 2).mean()
        (g,) = torch.autograd.grad(loss, q)
        losses.append(loss.detach())
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        par = par - _lr(i) * (m1 / (1 - 0.9 ** (i + 1))) / (torch.sqrt(m2 / (1 - 0.999 ** (i + 1))) + 1e-8)
    return {"params": par, "loss": torch.stack(losses), "held": forward(par, x[N_ROWS:])}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "batch":
        got = [_exact_run(g, f, p, _packet(g, f, p), case["steps"], case["obs_every"])
               for g, f, p in _batch_setup(case, seed)]
        res = {"psi": [psi for psi, _ in got]}
        if case["obs_every"]:
            res["obs"] = torch.tensor([rows for _, rows in got], dtype=torch.float64)
        return res
    grid, f, p = _run_setup(case, seed)
    psi, rows = _exact_run(grid, f, p, _packet(grid, f, p), case["steps"], case["obs_every"])
    res = {"psi": psi}
    if rows:
        res["obs"] = torch.tensor(rows, dtype=torch.float64)
    if case["densities"]:
        res["momentum"] = _observe(grid, f, p, psi, 0.0)[1]
        res["density_x"] = (psi.abs() ** 2).sum((0, 2)) * ((grid.y_max - grid.y_min) / grid.ny)
    return res
