"""The work a user of the solver has it do, one case at a time, for timing it.

Every case is a plain dict. ``prepare`` makes what a user's program holds before the call, ``run``
is one pass through the public binding (``paper_2407_12263_gb300.lbm``), ``work`` the bytes and
operations of a pass and ``exact`` the same outputs in FP64 with plain torch.

Kinds of case
  step     a simulation advances `steps` time steps and its fields are sampled on the device
  fields   the same with the finite-difference scheme, its fields read back to the host
  job      a whole static-droplet job: initial fields from the host, steps, the metrics
  batch    many independent rising-bubble boxes advanced together, then sampled
  train    one training iteration of the surrogate network (gradients, then the Adam update)
  forward  the network's prediction for a batch of coarse fields
  jump     a trajectory restarted from coarse fields and fast-forwarded by the judged surrogate
  project  the divergence-free part of a periodic velocity field
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2407_12263_gb300 import lbm

STORAGE = {"fp32": lbm.LBM_STORAGE_FP32, "fp16": lbm.LBM_STORAGE_FP16, "bf16": lbm.LBM_STORAGE_BF16}
E9 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
CS2 = 1.0 / 3.0
P0 = CS2
XI, MOBILITY, COURANT = 4.0, 0.02, 0.997
CHANNELS = (5, 32, 32, 32, 5)
N_PARAMS = sum(o * i * 27 + o for i, o in zip(CHANNELS, CHANNELS[1:]))
# normalisation of (phi, u, v, w, p): what the mean and spread of Taylor-Green trajectories are
MEAN_STD = (0.99, 0.0, 0.0, 0.0, CS2, 0.1, 0.016, 0.016, 0.012, 2e-4)


def listed():
    return [
        # the 2D static droplet every accuracy study starts from: one small grid, many short steps
        _step("droplet2d_64", "droplet", (64, 64, 1), "fp32", steps=32),
        # the 3D static droplet at the published benchmark's size
        _step("droplet3d_128", "droplet", (128, 128, 128), "fp32", steps=50),
        # droplet breakup in a Taylor-Green vortex, sampled as the surrogate's training data is
        _step("taylor_green_256_fp16", "vortex", (256, 256, 256), "fp16", steps=16, factor=4),
        # Rayleigh-Taylor box: walls, gravity, density ratio 3
        _step("rayleigh_taylor_512", "layers", (128, 128, 512), "fp32", steps=16, factor=4, walls=4),
        # the same flow on an odd grid in BF16, as a resolution study takes it
        _step("rayleigh_taylor_odd_bf16", "layers", (94, 75, 301), "bf16", steps=32, walls=4),
        # the finite-difference comparison scheme in 2D with its fields plotted on the host
        dict(name="fd2d_fields", kind="fields", flow="droplet", nx=200, ny=168, nz=1, storage="fp32", steps=40,
             factor=1, walls=0),
        # a static-droplet job from initial fields to spurious currents, Laplace jump and mass
        dict(name="droplet_job_128", kind="job", flow="droplet", nx=128, ny=128, nz=128, storage="fp32", steps=20,
             factor=1, walls=0),
        # a parameter study of rising bubbles in walled boxes of 32 to 96 cells
        dict(name="bubbles_batch", kind="batch", count=24, smallest=32, storage="fp32", steps=24),
        # training of the surrogate at its own size, and on an odd grid with a ragged batch
        dict(name="train_64", kind="train", nx=64, ny=64, nz=64, batch=4),
        dict(name="train_odd", kind="train", nx=30, ny=26, nz=45, batch=3),
        # one prediction
        dict(name="forward_64", kind="forward", nx=64, ny=64, nz=64, batch=1),
        # one judged jump of a 128^3 trajectory
        dict(name="jump_128", kind="jump", nx=128, ny=128, nz=128, factor=2, storage="fp16"),
    ]


def _step(name, flow, grid, storage, steps, factor=1, walls=0):
    return dict(name=name, kind="step", flow=flow, nx=grid[0], ny=grid[1], nz=grid[2], storage=storage, steps=steps,
                factor=factor, walls=walls)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step2d", "step3d", "step3d", "walled", "walled", "fields", "job", "batch", "train", "forward",
                       "jump", "project"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind in ("step2d", "fields"):
        c = _step("", "droplet", (log_int(40, 600), log_int(40, 600), 1), storage, steps=rng.randint(8, 64))
        c["kind"] = "fields" if kind == "fields" else "step"
    elif kind in ("step3d", "walled", "job"):
        grid = tuple(log_int(24, 220) for _ in range(3))
        c = _step("", "layers" if kind == "walled" else rng.choice(["droplet", "vortex"]), grid, storage,
                  steps=rng.randint(8, 32), walls=4 if kind == "walled" else 0)
        if kind == "job":
            c.update(kind="job", flow="droplet", steps=rng.randint(10, 30))
        elif rng.random() < 0.4:  # a grid that the surrogate's sampling takes
            c["factor"] = rng.choice([2, 3, 4])
            for a in ("nx", "ny", "nz"):
                c[a] = max(c["factor"] * 8, c[a] // c["factor"] * c["factor"])
    elif kind == "batch":
        return dict(kind="batch", count=log_int(6, 40), smallest=rng.choice([20, 24, 32, 36]), storage=storage,
                    steps=rng.randint(8, 32))
    elif kind in ("train", "forward"):
        return dict(kind=kind, nx=log_int(12, 72), ny=log_int(12, 72), nz=log_int(12, 72), batch=rng.randint(1, 4))
    elif kind == "jump":
        f = rng.choice([2, 4])
        return dict(kind="jump", nx=f * log_int(16, 40), ny=f * log_int(16, 40), nz=f * log_int(16, 40), factor=f,
                    storage=rng.choice(["fp32", "fp16"]))
    else:
        return dict(kind="project", nx=log_int(16, 128), ny=log_int(16, 128), nz=log_int(16, 128))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
_streams = {}


def _stream():
    """The one stream a program runs its handles and its network on."""
    dev = torch.cuda.current_device()
    if dev not in _streams:
        _streams[dev] = torch.cuda.Stream()
    return _streams[dev]


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _gen(seed, salt):
    return torch.Generator(device="cpu").manual_seed(seed * 1009 + salt)


def _uniform(gen, lo, hi, n=1):
    v = (torch.rand(n, generator=gen, dtype=torch.float64) * (hi - lo) + lo).tolist()
    return v[0] if n == 1 else v


def _coords(grid):
    nx, ny, nz = grid
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    return x, y, z


def _params(case, seed):
    """The arguments of a handle: fluid properties of the flow, a little different for each seed."""
    gen = _gen(seed, 1)
    p = dict(tau_f=_uniform(gen, 0.6, 0.9), tau_g=0.8, M=MOBILITY, xi=XI, sigma=_uniform(gen, 0.8e-3, 1.2e-3),
             rho_ratio=1.0, mu_ratio=1.0, body_force=(0.0, 0.0, 0.0))
    if case["flow"] == "vortex":  # Re = 1000, We = 20 on the box
        n = case["nx"]
        p["tau_f"] = 3.0 * 0.04 * n / 1000.0
        p["sigma"] = 0.04 ** 2 * (n / 4.0) / 20.0
    if case["flow"] == "layers":  # density ratio 3, Re = 256, Ca = 1 on the box's width
        n, g = case["nx"], 0.04 ** 2 / case["nx"]
        p.update(rho_ratio=3.0, tau_f=3.0 * 3.0 * 0.04 * n / 256.0, body_force=(0.0, 0.0, -g))
        p["sigma"] = p["tau_f"] / 3.0 * 0.04
    return p


def _initial(case, seed):
    """phi0 and u0 on the device, FP64."""
    gen = _gen(seed, 2)
    grid = _grid(case)
    nx, ny, nz = grid
    x, y, z = _coords(grid)
    u = torch.zeros((3,) + x.shape, dtype=torch.float64, device="cuda")
    if case["flow"] == "layers":
        a = 0.05 * nx * _uniform(gen, 0.6, 1.4)
        px, py = _uniform(gen, 0.0, 2 * math.pi, 2)
        zi = (nz - 1) / 2.0 + a * torch.cos(2 * math.pi * x / nx + px) * torch.cos(2 * math.pi * y / ny + py)
        return 0.5 * (1.0 + torch.tanh(2.0 * (z - zi) / XI)), u
    least = min(n for n in grid if n > 1)
    radius = least * _uniform(gen, 0.17, 0.23)
    d2 = torch.zeros_like(x)
    for c, n in ((x, nx), (y, ny), (z, nz)):
        if n > 1:
            d = (c - ((n - 1) / 2.0 + _uniform(gen, -2.0, 2.0))).abs()
            d = torch.minimum(d, n - d)
            d2 += d * d
    phi = 0.5 * (1.0 + torch.tanh(2.0 * (d2.sqrt() - radius) / XI))
    u0 = 0.04 * _uniform(gen, 0.8, 1.0) if case["flow"] == "vortex" else 0.01 * _uniform(gen, 0.8, 1.0)
    X, Y, Z = 2 * math.pi * x / nx, 2 * math.pi * y / ny, 2 * math.pi * z / nz
    u[0] = u0 * torch.sin(X) * torch.cos(Y) * (torch.cos(Z) if nz > 1 else 1.0)
    u[1] = -u0 * torch.cos(X) * torch.sin(Y) * (torch.cos(Z) if nz > 1 else 1.0)
    return phi, u


def _host(t):
    return np.ascontiguousarray(t.cpu().numpy())


def _lattice(case, seed, scheme=lbm.LBM_SCHEME_DIFFERENCE_FREE):
    grid = _grid(case)
    return lbm.Lattice(grid, lbm.LBM_D2Q9 if grid[2] == 1 else lbm.LBM_D3Q19, **_params(case, seed), scheme=scheme,
                       storage=STORAGE[case["storage"]], walls=case["walls"], courant=COURANT,
                       stream=_stream().cuda_stream)


def _bubble_cases(case, seed):
    """Boxes of widths s, 3/2 s, 2 s and 3 s and heights of one or two widths, walls on every side."""
    gen = _gen(seed, 3)
    s0 = case["smallest"]
    out = []
    for i in range(case["count"]):
        s = (s0, 3 * s0 // 2, 2 * s0, 3 * s0)[i % 4]
        h = 1 + (i // 4) % 2
        rho, mu = _uniform(gen, 2.0, 10.0), _uniform(gen, 1.0, 10.0)
        R = s / 8.0
        u = 0.04
        g = u * u / (2 * R)
        sigma = (rho - 1.0) * g * 4 * R * R / math.exp(_uniform(gen, 0.0, math.log(50.0)))
        out.append(dict(nx=s, ny=s, nz=h * s, walls=7, R=R,
                        params=dict(tau_f=_uniform(gen, 0.05, 0.4), tau_g=0.8, M=MOBILITY, xi=XI, sigma=sigma,
                                    rho_ratio=rho, mu_ratio=mu, body_force=(0.0, 0.0, -g))))
    return out


def _bubble_phi(c):
    x, y, z = _coords(_grid(c))
    m = c["nx"] / 2.0 - 0.5
    r = ((x - m) ** 2 + (y - m) ** 2 + (z - 4.0 * c["R"]) ** 2).sqrt()
    return 0.5 * (1.0 + torch.tanh(2.0 * (r - c["R"]) / XI))


def _weights(seed, last):
    """He-normal weights of the network, the last layer scaled by `last`, small biases."""
    gen = _gen(seed, 4)
    out = []
    for l, (ci, co) in enumerate(zip(CHANNELS, CHANNELS[1:])):
        w = torch.randn(co * ci * 27, generator=gen) * math.sqrt(2.0 / (27 * ci)) * (last if l == 3 else 1.0)
        out += [w, 0.05 * torch.randn(co, generator=gen) * (last if l == 3 else 1.0)]
    return torch.cat(out)


def _smooth(gen, shape, modes=6):
    """Smooth periodic fields of order one, FP32 on the device: what normalised coarse fields look like."""
    lead, (nz, ny, nx) = shape[:-3], shape[-3:]
    out = torch.zeros((math.prod(lead), nz, ny, nx), dtype=torch.float64, device="cuda")
    x, y, z = _coords((nx, ny, nz))
    for a in range(out.shape[0]):
        for _ in range(modes):
            k = torch.randint(-4, 5, (3,), generator=gen).tolist()
            amp, ph = _uniform(gen, 0.2, 0.8), _uniform(gen, 0.0, 2 * math.pi)
            out[a] += amp * torch.sin(2 * math.pi * (k[0] * x / nx + k[1] * y / ny + k[2] * z / nz) + ph)
    noise = torch.randn(out.shape, generator=torch.Generator(device="cuda").manual_seed(gen.initial_seed() % (1 << 31)),
                        device="cuda")
    return (out + 0.05 * noise).float().reshape(shape).contiguous()


def _net_fields(case, seed):
    gen = _gen(seed, 5)
    shape = (case["batch"], 5, case["nz"], case["ny"], case["nx"])
    x = _smooth(gen, shape)
    return x, (x + 0.3 * _smooth(gen, shape)).contiguous()


def _jump_fields(case, seed):
    """Coarse fields of a Taylor-Green trajectory: a droplet in the vortex, pressure about 1/3."""
    f = case["factor"]
    c = dict(flow="vortex", nx=case["nx"] // f, ny=case["ny"] // f, nz=case["nz"] // f)
    phi, u = _initial(c, seed)
    p = P0 + 0.25 * (u * u).sum(0)
    return torch.cat([phi[None], u, p[None]]).float().contiguous()


def _jump_case(case):
    return dict(case, flow="vortex", walls=0)


def _velocity(case, seed):
    return (0.03 * _smooth(_gen(seed, 6), (3, case["nz"], case["ny"], case["nx"]))).contiguous()


# ---------------------------------------------------------------- one pass
def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind in ("step", "fields", "job"):
        fd = kind == "fields"
        g = s["g"] = _lattice(case, seed, lbm.LBM_SCHEME_FINITE_DIFFERENCE if fd else lbm.LBM_SCHEME_DIFFERENCE_FREE)
        phi, u = _initial(case, seed)
        s["phi0"], s["u0"] = _host(phi), _host(u)
        if kind != "job":
            g.init_phi(s.pop("phi0"), s.pop("u0"), P0)
        if kind == "step":
            s["out"] = _coarse_out(case)
    elif kind == "batch":
        boxes = _bubble_cases(case, seed)
        b = s["b"] = lbm.Batch([lbm.make_case(_grid(c), lbm.LBM_D3Q19, **c["params"], walls=c["walls"],
                                              storage=STORAGE[case["storage"]]) for c in boxes],
                               stream=_stream().cuda_stream)
        for i, c in enumerate(boxes):
            b.case(i).init_phi(_host(_bubble_phi(c)), None, P0)
        s["out"] = [torch.empty((5,) + tuple(n // 2 for n in _grid(c)[::-1]), device="cuda") for c in boxes]
    elif kind in ("train", "forward"):
        s["x"], s["t"] = _net_fields(case, seed)
        s["net"] = lbm.Net(fp16=True, stream=_stream().cuda_stream)
        s["net"].set_params(_weights(seed, 0.1).numpy())
        s["y"] = torch.empty_like(s["x"])
    elif kind == "jump":
        g = s["g"] = _lattice(_jump_case(case), seed)
        phi, u = _initial(_jump_case(case), seed)
        g.init_phi(_host(phi), _host(u), P0)
        s["net"] = lbm.Net(fp16=True, stream=_stream().cuda_stream)
        s["net"].set_params(_weights(seed, 0.005).numpy())  # small changes, as a trained network predicts
        s["start"] = _jump_fields(case, seed)
        s["out"] = torch.empty_like(s["start"])
        lbm.lbm_surrogate_reserve(g.h, case["factor"])
    else:
        s["u"] = _velocity(case, seed)
        s["v"] = torch.empty_like(s["u"])
        s["work"] = torch.empty(lbm.lbm_project_workspace_bytes(_grid(case)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    return s


def _coarse_out(case):
    return torch.empty((5,) + tuple(n // (case["factor"] if n > 1 else 1) for n in _grid(case)[::-1]), device="cuda")


def _parts(out):
    return {"phi": out[0], "u": out[1:4], "p": out[4]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        state["g"].step(case["steps"])
        lbm.lbm_coarse_fields(state["g"].h, case["factor"], state["out"].data_ptr())
        return _parts(state["out"])
    if kind == "fields":
        state["g"].step(case["steps"])
        phi, p, u = state["g"].moments()
        return {"phi": phi.astype(np.float32), "u": u.astype(np.float32), "p": p.astype(np.float32)}
    if kind == "job":
        g, (centre, r_in, r_out) = state["g"], _spheres(case)
        g.init_phi(state["phi0"], state["u0"], P0)
        g.step(case["steps"])
        d = g.diagnostics(centre, r_in, r_out)
        sum_phi, sum_rho_phi = g.mass()
        return {"max_speed": d["max_speed"], "kinetic": d["kinetic"], "p_in": d["p_in"], "p_out": d["p_out"],
                "n_in": d["n_in"], "n_out": d["n_out"], "sum_phi": sum_phi, "sum_rho_phi": sum_rho_phi}
    if kind == "batch":
        state["b"].step(case["steps"])
        for i, out in enumerate(state["out"]):
            lbm.lbm_coarse_fields(state["b"].case(i).h, 2, out.data_ptr())
        return state["out"]
    if kind == "train":
        net, grid = state["net"], _grid(case)
        loss = net.gradients(state["x"].data_ptr(), state["t"].data_ptr(), case["batch"], grid)
        net.adam(1e-5)
        return {"loss": loss, "grads": net.get_grads()}
    if kind == "forward":
        state["net"].forward(state["x"].data_ptr(), state["y"].data_ptr(), case["batch"], _grid(case))
        return state["y"]
    if kind == "jump":
        h, f = state["g"].h, case["factor"]
        lbm.lbm_restart_from_coarse(h, f, state["start"].data_ptr(), P0)
        rep = lbm.lbm_surrogate_jump(h, state["net"], f, MEAN_STD, 100, 8, 1e-2, 2.0, 1.0)
        lbm.lbm_coarse_fields(h, f, state["out"].data_ptr())
        return dict(_parts(state["out"]), accepted=int(rep["accepted"]), relax_ratio=rep["relax_ratio"],
                    interface_shift=rep["interface_shift"], interface_limit=rep["interface_limit"])
    with torch.cuda.stream(_stream()):
        state["v"].copy_(state["u"])
    lbm.lbm_project_solenoidal(state["v"].data_ptr(), _grid(case), state["work"].data_ptr(), state["work"].numel(),
                               _stream().cuda_stream)
    return state["v"]


def _spheres(case):
    """Centre and radii of the pressure averages inside and outside the droplet."""
    grid = _grid(case)
    least = min(n for n in grid if n > 1)
    return tuple((n - 1) / 2.0 for n in grid), 0.1 * least, 0.4 * least


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "batch":
        cells = [math.prod(_grid(c)) for c in _bubble_cases(case, 0)]
        b = sum(_state_bytes(19, n, case["storage"], case["steps"], sum(cells)) + 5 * 4 * n / 8 for n in cells)
        return {"bytes": b, "flops": 900.0 * sum(cells) * case["steps"]}
    n = math.prod(_grid(case))
    if kind in ("step", "fields", "job"):
        q = 9 if case["nz"] == 1 else 19
        b = _state_bytes(q, n, case["storage"], case["steps"], n)
        b += {"step": 5 * 4 * n / case["factor"] ** (3 if q == 19 else 2), "fields": 5 * 8 * n, "job": 4 * 8 * n}[kind]
        return {"bytes": b, "flops": 45.0 * q * n * case["steps"]}
    if kind in ("train", "forward"):
        n *= case["batch"]
        macs = sum(27 * i * o for i, o in zip(CHANNELS, CHANNELS[1:]))
        if kind == "forward":
            return {"bytes": 4.0 * (2 * 5 * n + N_PARAMS), "flops": 2.0 * macs * n}
        inner = sum(27 * i * o for i, o in zip(CHANNELS[1:], CHANNELS[2:]))
        # read: fields, targets, weights and the optimiser's state; written: gradients, weights, state
        return {"bytes": 4.0 * (2 * 5 * n + 7 * N_PARAMS), "flops": 2.0 * (2 * macs + inner) * n}
    if kind == "jump":
        # the restart writes the state; the jump saves it, reads it for the prediction, and restarts
        # and judges it twice over 8 steps; the fields are read at the end
        nc = n / case["factor"] ** 3
        per = 304.0 if case["storage"] == "fp32" else 160.0
        macs = sum(27 * i * o for i, o in zip(CHANNELS, CHANNELS[1:]))
        return {"bytes": n * per * (0.5 + 1 + 0.5 + 2 * (0.5 + 8) + 0.5) + 20 * nc * 4,
                "flops": 16 * 850.0 * n + 2.0 * macs * nc}
    # transforms of a real field along three axes and back
    return {"bytes": 2 * 3 * 4.0 * n, "flops": 3 * 2 * 2.5 * n * math.log2(max(n, 2))}


def _state_bytes(q, n, storage, steps, resident):
    """The state read and written in every step, or once where the whole set (two copies) stays on
    the chip: it then fits the SMs' shared memory."""
    per = (8 * q if storage == "fp32" else 8 + 4 * (q - 1)) * 2.0
    once = per * resident <= 32e6
    return per * n * (1 if once else steps)


# ---------------------------------------------------------------- the same in FP64
class _Flow:
    """The scheme on plain FP64 populations: Lax-Wendroff propagation, macroscopic fields, collision."""

    def __init__(self, grid, prm, walls, fd=False):
        self.E = E9 if grid[2] == 1 else E19
        self.D = 2 if grid[2] == 1 else 3
        t = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if self.D == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.T = [t[sum(c * c for c in e)] for e in self.E]
        self.opp = [self.E.index(tuple(-c for c in e)) for e in self.E]
        self.prm, self.walls, self.fd = prm, walls, fd
        self.tau = 3.0 * prm["M"]

    def shift(self, a, e, other=None):
        """a at x + e; beyond a wall, `other` of the cell itself (or its own mirror image)."""
        r = torch.roll(a, (-e[2], -e[1], -e[0]), (0, 1, 2))
        if other is None:
            for ax in range(3):
                if e[ax] and self.walls >> ax & 1:  # one clamped move per axis
                    break
            else:
                return r
            n = a.shape
            idx = []
            for d, ax in ((0, 2), (1, 1), (2, 0)):
                i = torch.arange(n[d], device=a.device) + e[ax]
                idx.append(i.clamp(0, n[d] - 1) if self.walls >> ax & 1 else i % n[d])
            return a[idx[0]][:, idx[1]][:, :, idx[2]]
        for ax, d in ((0, 2), (1, 1), (2, 0)):
            if e[ax] and self.walls >> ax & 1:
                at = [slice(None)] * 3
                at[d] = -1 if e[ax] > 0 else 0
                r[tuple(at)] = other[tuple(at)]
        return r

    def gradient(self, phi):
        g = [torch.zeros_like(phi) for _ in range(3)]
        for e, t in zip(self.E[1:], self.T[1:]):
            v = t * self.shift(phi, e)
            for a in range(3):
                if e[a]:
                    g[a] += 3.0 * e[a] * v
        return g

    @staticmethod
    def dot(e, v):
        r = 0.0
        for c, w in zip(e, v):
            if c:
                r = r + c * w
        return r

    def normal(self, v, sign):
        s = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
        r = torch.where(s > 1e-24, sign / s.clamp_min(1e-300).sqrt(), torch.zeros_like(s))
        return [c * r for c in v]

    def equilibria(self, i, m):
        e, t = self.E[i], self.T[i]
        eu, u2 = self.dot(e, m["u"]), sum(c * c for c in m["u"])
        gam = 3 * eu + 4.5 * eu * eu - 1.5 * u2
        en, n2 = self.dot(e, m["n"]), sum(c * c for c in m["n"])
        pis = self.prm["sigma"] * m["gnorm"] * (sum(c * c for c in e) - en * en - (self.D - n2) / 3.0)
        feq = t * (3 * m["p"] + m["rho"] * gam - 4.5 * pis)
        return feq, t * (m["phi"] * (1 + gam) + self.tau * self.dot(e, m["S"])), gam, eu

    def init(self, phi, u, p):
        """Post-collision populations of the initial fields."""
        gphi = self.gradient(phi)
        m = dict(phi=phi, u=u, p=p, rho=1 + (self.prm["rho_ratio"] - 1) * phi, n=self.normal(gphi, 1.0))
        m["gnorm"] = sum(c * c for c in gphi).sqrt()
        m["S"] = [4 / self.prm["xi"] * phi * (1 - phi) * c for c in m["n"]]
        self.f, self.g = [], []
        for i in range(len(self.E)):
            feq, geq, _, _ = self.equilibria(i, m)
            self.f.append(feq + torch.zeros_like(phi))
            self.g.append(geq - self.T[i] * (self.tau - 0.5) * self.dot(self.E[i], gphi))

    def propagated(self, s):
        c, out = COURANT, []
        for i, e in enumerate(self.E):
            if i == 0:
                out.append(s[0])
                continue
            back = tuple(-v for v in e)
            lo, hi = self.shift(s[i], back, s[self.opp[i]]), self.shift(s[i], e, s[self.opp[i]])
            out.append(s[i] - c * (s[i] - lo) - 0.5 * c * (1 - c) * (hi - 2 * s[i] + lo))
        return out

    def macro(self, f, g):
        m, prm = {}, self.prm
        m["phi"] = phi = sum(g)
        m["rho"] = rho = 1 + (prm["rho_ratio"] - 1) * phi
        j = [sum(e[a] * v for e, v in zip(self.E, f) if e[a]) if a < self.D else torch.zeros_like(phi) for a in range(3)]
        m["u"] = u = [(j[a] + 0.5 * rho * prm["body_force"][a]) / rho for a in range(3)]
        if self.fd:
            gphi = self.gradient(phi)
            m["n"] = self.normal(gphi, 1.0)
        else:
            k = [(sum(e[a] * v for e, v in zip(self.E, g) if e[a]) if a < self.D else torch.zeros_like(phi)) - phi * u[a]
                 for a in range(3)]
            m["n"] = self.normal(k, -1.0)
        smag = 4 / prm["xi"] * phi * (1 - phi)
        m["S"] = [smag * c for c in m["n"]]
        if not self.fd:
            gphi = [(self.tau * CS2 * s - c) / ((self.tau + 0.5) * CS2) for s, c in zip(m["S"], k)]
        m["grho"] = [(prm["rho_ratio"] - 1) * c for c in gphi]
        m["gnorm"] = sum(c * c for c in gphi).sqrt()
        m["p"] = CS2 * (sum(f) + 0.5 * sum(a * b for a, b in zip(u, m["grho"])))
        return m

    def fields(self):
        m = self.macro(self.propagated(self.f), self.propagated(self.g))
        return torch.stack([m["phi"], *m["u"], m["p"]]), m

    def step(self, steps):
        prm = self.prm
        for _ in range(steps):
            f, g = self.propagated(self.f), self.propagated(self.g)
            self.f = self.g = None
            m = self.macro(f, g)
            rho, u = m["rho"], m["u"]
            eta = prm["tau_f"] / 3.0 * (1 + (prm["mu_ratio"] - 1) * m["phi"])
            omega = 1.0 / (3.0 * eta / rho + 0.5)
            G = [rho * c for c in prm["body_force"]]
            u_gr, u_G = sum(a * b for a, b in zip(u, m["grho"])), sum(a * b for a, b in zip(u, G))
            for i, e in enumerate(self.E):
                feq, geq, gam, eu = self.equilibria(i, m)
                F = self.T[i] * (gam * (self.dot(e, m["grho"]) - u_gr)
                                 + 3 * (self.dot(e, G) - u_G) + 9 * eu * self.dot(e, G))
                f[i] = f[i] - omega * (f[i] - feq + 0.5 * F) + F
                g[i] = g[i] - (g[i] - geq) / (self.tau + 0.5)
            self.f, self.g = f, g


def _means(a, f):
    if f == 1:
        return a
    c, nz, ny, nx = a.shape
    fz = f if nz > 1 else 1
    return a.reshape(c, nz // fz, fz, ny // f, f, nx // f, f).mean((2, 4, 6))


def _upsample(a, f):
    """Trilinear between coarse cell centres, periodic."""
    for d in range(1, 4):
        n = a.shape[d]
        x = (torch.arange(n * f, dtype=torch.float64, device=a.device) + 0.5) / f - 0.5
        i = x.floor()
        t = (x - i).reshape([-1 if k == d else 1 for k in range(4)])
        i = i.long()
        a = a.index_select(d, i % n) * (1 - t) + a.index_select(d, (i + 1) % n) * t
    return a


def _predict(x, params):
    h, at = x, 0
    for l, (ci, co) in enumerate(zip(CHANNELS, CHANNELS[1:])):
        w = params[at:at + co * ci * 27].reshape(co, ci, 3, 3, 3)
        b = params[at + co * ci * 27:at + co * ci * 27 + co]
        at += co * ci * 27 + co
        h = torch.nn.functional.pad(h, (1,) * 6, mode="circular")
        # one matrix product per tap: FP64 convolutions are not what cuDNN is made for
        n = x.shape[-3:]
        out = b[:, None, None, None] + sum(
            torch.einsum("oc,bczyx->bozyx", w[:, :, dz, dy, dx], h[:, :, dz:dz + n[0], dy:dy + n[1], dx:dx + n[2]])
            for dz in range(3) for dy in range(3) for dx in range(3))
        h = torch.relu(out) if l < 3 else out
    return x + h


def _solenoidal(u):
    """The part of u whose central-difference divergence vanishes."""
    U = torch.fft.fftn(u, dim=(1, 2, 3))
    s = []
    for a, d in ((0, 3), (1, 2), (2, 1)):
        n = u.shape[d]
        k = torch.arange(n, dtype=torch.float64, device=u.device)
        v = torch.sin(2 * math.pi * k / n)
        v[(2 * k) % n == 0] = 0.0
        s.append(v.reshape([-1 if e == d - 1 else 1 for e in range(3)]))
    s2 = s[0] ** 2 + s[1] ** 2 + s[2] ** 2
    dot = (s[0] * U[0] + s[1] * U[1] + s[2] * U[2]) / torch.where(s2 > 0, s2, torch.ones_like(s2))
    return torch.fft.ifftn(torch.stack([U[a] - s[a] * dot for a in range(3)]), dim=(1, 2, 3)).real


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "fields", "job"):
        flow = _Flow(_grid(case), _params(case, seed), case["walls"], fd=kind == "fields")
        phi, u = _initial(case, seed)
        flow.init(phi, [u[0], u[1], u[2]], P0)
        flow.step(case["steps"])
        a, m = flow.fields()
        if kind != "job":
            return _parts(_means(a, case["factor"]))
        (cx, cy, cz), r_in, r_out = _spheres(case)
        d2 = 0.0
        for c, o, n in zip(_coords(_grid(case)), (cx, cy, cz), _grid(case)):
            d = (c - o).abs()
            d2 = d2 + torch.minimum(d, n - d) ** 2
        d = d2.sqrt()
        s2 = (a[1:4] ** 2).sum(0)
        inside, outside = d < r_in, d > r_out
        return {"max_speed": float(s2.max().sqrt()), "kinetic": float((0.5 * m["rho"] * s2).sum()),
                "p_in": float(a[4][inside].mean()), "p_out": float(a[4][outside].mean()), "n_in": int(inside.sum()),
                "n_out": int(outside.sum()), "sum_phi": float(a[0].sum()),
                "sum_rho_phi": float((m["rho"] * a[0]).sum())}
    if kind == "batch":
        out = []
        for c in _bubble_cases(case, seed):
            flow = _Flow(_grid(c), c["params"], c["walls"])
            phi = _bubble_phi(c)
            flow.init(phi, [torch.zeros_like(phi)] * 3, P0)
            flow.step(case["steps"])
            out.append(_means(flow.fields()[0], 2))
        return out
    if kind in ("train", "forward"):
        x, t = _net_fields(case, seed)
        params = _weights(seed, 0.1).double().cuda()
        if kind == "forward":
            return torch.cat([_predict(x[b:b + 1].double(), params) for b in range(case["batch"])])
        loss, grads = 0.0, torch.zeros_like(params)
        for b in range(case["batch"]):
            with torch.enable_grad():
                w = params.clone().requires_grad_()
                part = (_predict(x[b:b + 1].double(), w) - t[b:b + 1].double()).square().mean() / case["batch"]
                part.backward()
            loss += float(part)
            grads += w.grad
        return {"loss": loss, "grads": grads}
    if kind == "jump":
        f, c = case["factor"], _jump_case(case)
        flow = _Flow(_grid(case), _params(c, seed), 0)

        def restart(coarse, total):
            a = _upsample(coarse, f)
            flow.init(a[0], [a[1], a[2], a[3]], a[4])
            flow.g[0] += (total - a[0].sum()) / a[0].numel()

        total = _initial(c, seed)[0].sum()
        restart(_jump_fields(case, seed).double(), total)
        start = _means(flow.fields()[0], f)
        mean, std = (torch.tensor(v, dtype=torch.float64, device="cuda")[:, None, None, None]
                     for v in (MEAN_STD[:5], MEAN_STD[5:]))
        pred = _predict(((start - mean) / std)[None], _weights(seed, 0.005).double().cuda())[0] * std + mean
        pred[1:4] = _solenoidal(pred[1:4])
        restart(pred, total)
        flow.step(8)
        return dict(_parts(_means(flow.fields()[0], f)), accepted=None, relax_ratio=None, interface_shift=None,
                    interface_limit=None)
    return _solenoidal(_velocity(case, seed).double())
