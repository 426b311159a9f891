"""Workloads the performance of this package is measured on, each one pass
through its public entry points, with float64 values to compare against.

The cases stand for what a user runs: the forward and the differentiable MPM
of one scene, the batched MPM both ways, the lattice solvers and their
reverse mode, the learned surrogate's inference and training, and the
rendered-view loss. `listed()` has one size of each from the package's own
scenes; `draw()` takes sizes over the whole range of each kind, odd ones
among them. Inputs are smooth fields (wind, velocity, strain, flow) made on
the GPU from the seed.
"""
import math
import os
import random

import numpy as np
import torch

from paper_2603_09668_gb300 import autograd as AG
from paper_2603_09668_gb300 import binding as B
from paper_2603_09668_gb300 import inversion as INV
from paper_2603_09668_gb300 import rollout as RO
from paper_2603_09668_gb300 import surrogate as SU

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F32, F64 = torch.float32, torch.float64


def listed():
    return [
        # one substep of the fixed-corotated block: a caller that steps the
        # simulation itself; launches and their latency are all of it
        dict(name="substep_block8k", kind="substep", shape="block", n=8192, n_grid=32, material=1),
        # the flag sheet's rollout, re-sorted every 15 substeps: the headline
        dict(name="rollout_sheet400k", kind="rollout", shape="sheet", n=400040, n_grid=128,
             material=0, substeps=200, sort_every=15),
        # forward and reverse of one inversion iteration's scene: small, so
        # hundreds of dependent short kernels
        dict(name="frames_sheet5k", kind="frames", shape="sheet", n=5504, n_grid=64, material=0,
             substeps=200, every=25, nf=12, frames=1),
        # the checkpointed forward and reverse of the 100k sheet under a
        # spatio-temporal wind
        dict(name="frames_sheet100k", kind="frames", shape="sheet", n=100284, n_grid=64,
             material=0, substeps=40, every=20, nf=32, frames=16),
        # 64 uneven scenes advanced together: throughput of an ensemble
        dict(name="batch_rollout_64", kind="batch", scenes=64, n_lo=20000, n_hi=400000, mix=0,
             substeps=30, sort_every=15),
        # one checkpoint segment of 16 scenes differentiated
        dict(name="batch_adjoint_16", kind="batch_adjoint", scenes=16, n_lo=20000, n_hi=400000,
             mix=0, substeps=10),
        # the wind constraint: BGK steps around a leaf cluster with an inlet
        dict(name="lbm_128", kind="lbm", nx=128, ny=128, nz=128, bc_x=1, force=0.0, steps=20),
        # its reverse mode through autograd, checkpointed every 4 steps
        dict(name="lbm_adjoint_128", kind="lbm_adjoint", nx=128, ny=128, nz=128, bc_x=1, steps=8,
             every=4),
        # an inversion interval's guide: voxelized sheet, HOME-LBM steps,
        # velocity at the wind nodes; a small lattice, many short launches
        dict(name="guide_home_32", kind="guide", cells=32, nf=12, n=5504, model="home", steps=30),
        # two surrogate blocks between two checks of a 128^3 lattice, the
        # lattice read before and written after them
        dict(name="surrogate_64", kind="surrogate", n=64, blocks=2),
        # one training step of the surrogate
        dict(name="train_64", kind="train", n=64),
        # the image term of the inversion: two views of the 100k sheet, L1 and
        # D-SSIM, and their gradient down to the particles
        dict(name="views_sheet100k_512", kind="views", n=100284, width=512, height=512, views=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["substep", "rollout", "frames", "batch", "batch_adjoint", "lbm",
                       "lbm_adjoint", "guide", "surrogate", "train", "views"])
    c = dict(kind=kind)
    if kind in ("substep", "rollout", "frames"):
        n = _log(rng, 1000, {"substep": 400000, "rollout": 400000, "frames": 110000}[kind])
        c.update(shape=rng.choice(["sheet", "block"]), n=n, material=rng.randrange(2),
                 n_grid=rng.randint(24, max(32, min(128, int(0.65 * math.sqrt(n))))))
        if kind == "rollout":
            c.update(substeps=rng.randint(20, 200), sort_every=rng.choice([0, 10, 15, 20, 25]))
        if kind == "frames":
            every = rng.choice([5, 10, 20, 25])
            c.update(substeps=every * rng.randint(2, 4), every=every, nf=rng.randint(6, 32),
                     frames=rng.choice([1, 4, 16]))
    elif kind in ("batch", "batch_adjoint"):
        c.update(scenes=_log(rng, 2, 32 if kind == "batch" else 12), n_lo=3000,
                 n_hi=_log(rng, 10000, 300000), mix=rng.randrange(1 << 20),
                 substeps=rng.randint(5, 25) if kind == "batch" else rng.randint(2, 8))
        if kind == "batch":
            c.update(sort_every=rng.choice([0, 10, 15, 25]))
    elif kind in ("lbm", "lbm_adjoint"):
        c.update(nx=_log(rng, 20, 144), ny=_log(rng, 20, 128), nz=_log(rng, 20, 112),
                 bc_x=rng.randrange(2))
        if kind == "lbm":
            c.update(force=rng.choice([0.0, 1e-5]), steps=rng.randint(5, 25))
        else:
            c.update(steps=rng.randint(3, 8), every=rng.randint(1, 4))
    elif kind == "guide":
        c.update(cells=_log(rng, 24, 128), nf=rng.randint(8, 32), n=_log(rng, 2000, 200000),
                 model=rng.choice(["home", "home", "bgk"]), steps=rng.randint(5, 30))
    elif kind == "surrogate":
        c.update(n=16 * rng.randint(1, 5), blocks=rng.randint(1, 6))
    elif kind == "train":
        c.update(n=16 * rng.randint(1, 6))
    else:
        c.update(n=_log(rng, 1000, 110000), width=_log(rng, 64, 512), height=_log(rng, 64, 512),
                 views=rng.randint(1, 2))
    return c


# ------------------------------------------------------------------ inputs --

def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + salt)


def _modes(pos, comps, n_modes, kmax, g):
    """[comps][...] sums of cosines of unit amplitude over positions pos [3][...]."""
    out = torch.zeros((comps,) + tuple(pos.shape[1:]), dtype=F32, device=DEV)
    k = torch.randint(-kmax, kmax + 1, (comps, n_modes, 3), generator=g, device=DEV).float()
    phi = torch.rand((comps, n_modes), generator=g, device=DEV) * (2 * math.pi)
    k[..., 0] += (k == 0).all(-1).float()
    for c in range(comps):
        for m in range(n_modes):
            arg = k[c, m, 0] * pos[0] + k[c, m, 1] * pos[1] + k[c, m, 2] * pos[2]
            out[c] += torch.cos(2 * math.pi * arg + phi[c, m])
    return out


def _grid(nz, ny, nx, centred):
    """Positions [3][nz][ny][nx] in the unit cube: cell centres, or nodes from face to face."""
    ax = [(torch.arange(m, device=DEV).float() + 0.5) / m if centred
          else torch.linspace(0, 1, m, device=DEV) for m in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    return torch.stack([x, y, z])


def _wind(nf, frames, g):
    """[frames][nf][nf][nf][3]: 10 N/kg along x plus slowly turning modes."""
    pos = _grid(nf, nf, nf, False)
    a, b = _modes(pos, 3, 4, 3, g), _modes(pos, 3, 4, 3, g)
    s = torch.linspace(0, 1, frames, device=DEV).view(frames, 1, 1, 1, 1)
    v = 2.0 * (torch.cos(math.pi * s) * a + torch.sin(math.pi * s) * b)
    v[:, 0] += 10.0
    return v.permute(0, 2, 3, 4, 1).contiguous()


def _sheet_size(n):
    nu = max(2, int(round(math.sqrt(0.75 * n))))
    return nu, -(-n // (2 * nu))


def _particles(shape, n, g):
    """(x [3][n], pinned [n] or None): a two-layer flag pinned at its edge, or a block."""
    i = torch.arange(n, device=DEV)
    r = torch.rand((3, n), generator=g, device=DEV)
    if shape == "sheet":
        nu, nv = _sheet_size(n)
        h = 0.6 / (nu - 1)
        col = i // (2 * nv)
        x = torch.stack([0.2 + col * h, 0.4 + (i // 2) % nv * (0.4 / (nv - 1)),
                         0.5 + ((i % 2).float() - 0.5) * h]) + (r - 0.5) * (0.1 * h)
        return x.float().contiguous(), (col == 0).to(torch.uint8)
    sub = max(2, int(round((n / 2) ** (1 / 3))))
    cell = i * sub ** 3 // n
    idx = torch.stack([cell // (sub * sub), cell // sub % sub, cell % sub])
    lo = torch.tensor([0.375, 0.275, 0.375], device=DEV).view(3, 1)
    return ((idx + r) * (0.25 / sub) + lo).float().contiguous(), None


def _physics(shape, n, n_grid, material):
    vol = 0.6 * 0.4 * 2 * 0.6 / (_sheet_size(n)[0] - 1) if shape == "sheet" else 0.25 ** 3
    return dict(n_grid=n_grid, dt=1e-4 if n_grid <= 64 else 5e-5, gravity=(0.0, -9.8, 0.0),
                bc_band=3, material=material, E=5e4 if shape == "sheet" else 1e4, nu=0.3,
                p_mass=1000.0 * vol / n, p_vol=vol / n)


def _scene(shape, n, n_grid, material, nf, frames, steps, seed, salt=0):
    """Physics, particles in motion (smooth velocity with its gradient as C, a
    few per cent of strain), and the wind over the simulated time."""
    g = _gen(seed, salt)
    pr = _physics(shape, n, n_grid, material)
    x, pinned = _particles(shape, n, g)
    v = 0.15 * _modes(x, 3, 3, 2, g)
    C = 1.5 * _modes(x, 9, 2, 2, g)
    F = 0.01 * _modes(x, 9, 2, 3, g)
    F[[0, 4, 8]] += 1.0
    if pinned is not None:
        v *= 1 - pinned
        C *= 1 - pinned
    return pr, (x, v, C, F), pinned, _wind(nf, frames, g), steps * pr["dt"]


def _batch_plan(c):
    """(shape, n, n_grid, material) of each scene: log-uniform counts, half the
    scenes on 64^3 and half on 128^3, sheets and blocks."""
    r, out = random.Random(c["mix"]), []
    for _ in range(c["scenes"]):
        n = int(math.exp(r.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]))))
        shape = "sheet" if r.random() < 0.5 else "block"
        out.append((shape, n, 64 if r.random() < 0.5 else 128, 0 if shape == "sheet" else 1))
    return out


def _batch_scenes(c, seed):
    return [_scene(*s, 16, 8, c["substeps"], seed, 17 + i) for i, s in enumerate(_batch_plan(c))]


def _leaves(nz, ny, nx, g):
    """Solid mask of 50 ellipsoids in the middle of the lattice."""
    pos = _grid(nz, ny, nx, True)
    solid = torch.zeros((nz, ny, nx), dtype=torch.bool, device=DEV)
    axes = 0.02 + 0.04 * torch.rand((50, 3), generator=g, device=DEV)
    ctr = 0.3 + 0.4 * torch.rand((50, 3), generator=g, device=DEV)
    q = torch.randn((50, 3, 3), generator=g, device=DEV)
    a = torch.nn.functional.normalize(q[:, 0], dim=1)  # random orientations
    b = torch.nn.functional.normalize(q[:, 1] - (q[:, 1] * a).sum(1, True) * a, dim=1)
    q = torch.stack([a, b, torch.linalg.cross(a, b, dim=1)], 1)
    for e in range(50):
        d = torch.einsum("ab,azyx->bzyx", q[e], pos - ctr[e].view(3, 1, 1, 1))
        solid |= ((d / axes[e].view(3, 1, 1, 1)) ** 2).sum(0) <= 1.0
    return solid.to(torch.uint8)


CX = [0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 0, 0, 1, -1, 1, -1, 0, 0]
CY = [0, 0, 0, 1, -1, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 1, -1]
CZ = [0, 0, 0, 0, 0, 1, -1, 0, 0, 1, -1, 1, -1, 0, 0, -1, 1, -1, 1]
WQ = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _feq(rho, u):
    """Shifted equilibrium populations [19][...] (minus their weights)."""
    uu = 1.5 * (u * u).sum(0)
    out = []
    for i in range(19):
        cu = CX[i] * u[0] + CY[i] * u[1] + CZ[i] * u[2]
        out.append(WQ[i] * ((rho - 1) + rho * (3 * cu + 4.5 * cu * cu - uu)))
    return torch.stack(out)


def _flow(nz, ny, nx, seed, masked=True):
    """(shifted populations, mask, inlet velocity) of a flow past the leaves:
    the inlet's velocity with smooth departures, and a small non-equilibrium part."""
    g = _gen(seed, 5)
    solid = _leaves(nz, ny, nx, g) if masked else None
    a = (torch.rand(2, generator=g, device=DEV) - 0.5).tolist()
    u_in = (0.05 * math.cos(a[0]) * math.cos(a[1]), 0.05 * math.sin(a[0]),
            0.05 * math.cos(a[0]) * math.sin(a[1]))
    pos = _grid(nz, ny, nx, True)
    u = 0.006 * _modes(pos, 3, 3, 2, g) + torch.tensor(u_in, device=DEV).view(3, 1, 1, 1)
    rho = 1.0 + 0.002 * _modes(pos, 1, 3, 2, g)[0]
    if solid is not None:
        u *= 1 - solid
        rho = torch.where(solid.bool(), 1.0, rho)
    f = _feq(rho, u)
    f += 1e-4 * (torch.rand(f.shape, generator=g, device=DEV) - 0.5)
    return f.contiguous(), solid, u_in


def _coarse_inputs(n, seed):
    """Training pair of the surrogate: features [n^3][16] (density, velocity in
    inlet units, solid fraction, zeros) and the target change of velocity."""
    g = _gen(seed, 9)
    pos = _grid(n, n, n, True)
    x = torch.zeros((n ** 3, 16), dtype=F32, device=DEV)
    frac = _leaves(2 * n, 2 * n, 2 * n, g).float().view(n, 2, n, 2, n, 2).mean((1, 3, 5))
    flow = 0.15 * _modes(pos, 4, 3, 3, g)
    flow[1] += 1.0
    flow[0] *= 0.2
    x[:, :4] = (flow * (frac < 1)).view(4, -1).t()
    x[:, 4] = frac.view(-1)
    y = torch.zeros((n ** 3, 16), dtype=F32, device=DEV)
    y[:, :3] = _modes(pos, 3, 4, 4, g).view(3, -1).t() * 0.5
    return x, y


def _rotation(yaw, tilt):
    cy, sy, ct, st = math.cos(yaw), math.sin(yaw), math.cos(tilt), math.sin(tilt)
    return np.array([[1, 0, 0], [0, ct, -st], [0, st, ct]]) @ np.array([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]])


def _view_inputs(c, seed):
    """Waving sheet with its Gaussians, oblique cameras, and target images."""
    g = _gen(seed, 11)
    n, W, H = c["n"], c["width"], c["height"]
    x, _ = _particles("sheet", n, g)
    h = 0.6 / (_sheet_size(n)[0] - 1)
    x[2] += 0.02 * _modes(x, 1, 2, 2, g)[0]
    F = 0.03 * _modes(x, 9, 2, 3, g)
    F[[0, 4, 8]] += 1.0
    sigma0 = torch.zeros((6, n), dtype=F32, device=DEV)
    sigma0[:3] = h * h
    color = 0.5 + 0.15 * _modes(x, 3, 3, 4, g)
    opacity = 0.4 + 0.5 * torch.rand(n, generator=g, device=DEV)
    cams = []
    for k in range(c["views"]):
        R = _rotation(0.35 + 0.6 * k, 0.25).astype(np.float32).astype(np.float64)
        T = (np.array([0.0, 0.0, 1.2]) - R @ np.array([0.5, 0.6, 0.5])).astype(np.float32).astype(np.float64)
        f = 1.17 * min(W, H)
        cams.append(dict(R=R, T=T, fx=f, fy=f, cx=W / 2, cy=H / 2, width=W, height=H))
    target = 0.4 + 0.1 * _modes(_grid(1, H, W, True)[:, 0], 3 * c["views"], 4, 5, g)
    return x, F.contiguous(), sigma0, color.contiguous(), opacity, cams, target.view(c["views"], 3, H, W).contiguous()


# ----------------------------------------------------------------- prepare --

def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _mpm(pr, n):
    return B.MPM.from_params(pr, max_particles=n)


def _prepare_substep(c, seed):
    pr, st, pin, wind, total = _scene(c["shape"], c["n"], c["n_grid"], c["material"], 8, 1, 1, seed)
    s = B.MpmState(*st)
    return dict(kind="substep", mpm=_mpm(pr, c["n"]), state=s, out=B.MpmState.empty_like(s), pin=pin,
                wind=B.WindField(wind, total))


def _prepare_rollout(c, seed):
    pr, st, pin, wind, total = _scene(c["shape"], c["n"], c["n_grid"], c["material"], 32, 16,
                                      c["substeps"], seed)
    ro = RO.Rollout(_mpm(pr, c["n"]), c["n"], B.WindField(wind, total), c["substeps"],
                    sort_every=c["sort_every"], with_pins=pin is not None)
    return dict(kind="rollout", ro=ro, state=B.MpmState(*st), pin=pin)


def _frames_target(x):
    return x + 0.004 * torch.sin(9.0 * x.flip(0))


def _prepare_frames(c, seed):
    pr, st, pin, wind, total = _scene(c["shape"], c["n"], c["n_grid"], c["material"], c["nf"],
                                      c["frames"], c["substeps"], seed)
    leaf = [a.requires_grad_(True) for a in st]
    return dict(kind="frames", mpm=_mpm(pr, c["n"]), state=B.MpmState(*leaf), pin=pin,
                wind=wind.requires_grad_(True), total=total, every=c["every"],
                substeps=c["substeps"], E=torch.tensor(pr["E"], device=DEV, requires_grad=True),
                target=_frames_target(st[0].detach()))


def _prepare_batch(c, seed):
    sc = _batch_scenes(c, seed)
    state = B.MpmState(*(torch.cat([s[1][k] for s in sc], 1).contiguous() for k in range(4)))
    pin = torch.cat([s[2] if s[2] is not None else
                     torch.zeros(s[1][0].shape[1], dtype=torch.uint8, device=DEV) for s in sc])
    batch = B.MPMBatch([(s[0], s[1][0].shape[1], B.WindField(s[3], s[4])) for s in sc])
    ids0 = torch.arange(batch.n, dtype=torch.int32, device=DEV)
    return dict(kind="batch", batch=batch, state=state, pin=pin, ids0=ids0, ids=ids0.clone(),
                work=state.clone(), wpin=pin.clone(), substeps=c["substeps"], sort=c["sort_every"])


def _batch_seed_grad(n, seed):
    g = _gen(seed, 3)
    return [torch.randn((r, n), generator=g, device=DEV) / n for r in (3, 3, 9, 9)]


def _prepare_batch_adjoint(c, seed):
    s = _prepare_batch(dict(c, sort_every=0), seed)
    n = int(s["batch"].n)
    nw, _ = s["batch"].wind_layout()
    s.update(kind="batch_adjoint", g0=B.MpmState(*_batch_seed_grad(n, seed)),
             tape=torch.empty(max(1, (c["substeps"] - 1) * 24 * n), dtype=F32, device=DEV),
             g_wind=torch.zeros(nw, dtype=F32, device=DEV),
             g_E=torch.zeros(c["scenes"], dtype=F32, device=DEV))
    return s


TAU = 0.55


def _lbm(c, u_in, **kw):
    return B.LBM((c["nx"], c["ny"], c["nz"]), TAU, u_inlet=u_in, bc_x=c["bc_x"],
                 force=(c.get("force", 0.0), 0.0, 0.0), **kw)


def _prepare_lbm(c, seed):
    f, solid, u_in = _flow(c["nz"], c["ny"], c["nx"], seed)
    return dict(kind="lbm", lbm=_lbm(c, u_in), f=f, solid=solid, steps=c["steps"])


def _lattice_grad(f, seed):
    return torch.randn(f.shape, generator=_gen(seed, 6), device=DEV)


def _prepare_lbm_adjoint(c, seed):
    f, solid, u_in = _flow(c["nz"], c["ny"], c["nx"], seed)
    return dict(kind="lbm_adjoint", lbm=_lbm(c, u_in, max_tape=c["every"]), g=_lattice_grad(f, seed),
                f=f.requires_grad_(True), solid=solid, steps=c["steps"], every=c["every"])


def _guide_inputs(c, seed):
    g = _gen(seed, 8)
    x, _ = _particles("sheet", c["n"], g)
    x[2] += 0.05 * _modes(x, 1, 2, 2, g)[0]
    a = (torch.rand(1, generator=g, device=DEV) - 0.5).item()
    return x.contiguous(), (0.05 * math.cos(a), 0.0, 0.05 * math.sin(a))


def _prepare_guide(c, seed):
    x, u_in = _guide_inputs(c, seed)
    return dict(kind="guide", guide=INV.LbmGuide(c["cells"], 0.6, u_in, c["nf"], model=c["model"]),
                x=x, steps=c["steps"])


def _prepare_surrogate(c, seed):
    f, solid, u_in = _flow(2 * c["n"], 2 * c["n"], 2 * c["n"], seed)
    params = torch.from_numpy(_weights()).to(DEV)
    s = SU.SurrogateLBM(2 * c["n"], u_inlet=u_in, params=params)
    return dict(kind="surrogate", surr=s, f=f, solid=solid, out=f.clone(), blocks=c["blocks"])


def _weights():
    return np.load(os.path.join(os.path.dirname(SU.__file__), "weights", "surrogate_lbm128.npy")).astype(np.float32)


LR = 1e-5


def _prepare_train(c, seed):
    x, y = _coarse_inputs(c["n"], seed)
    s = B.Surrogate(c["n"])
    s.set_params(torch.from_numpy(_weights()).to(DEV))
    return dict(kind="train", surr=s, x=x, y=y, step=0,
                out=torch.empty((c["n"] ** 3, 16), dtype=F32, device=DEV),
                loss=torch.zeros(1, dtype=F32, device=DEV))


def _prepare_views(c, seed):
    x, F, s0, col, opa, cams, target = _view_inputs(c, seed)
    r = B.GaussianRenderer(c["n"], c["width"], c["height"])
    obs = INV.RenderObservation(r, [B.camera(**k) for k in cams], s0, col, opa)
    zero = [torch.zeros((k, c["n"]), dtype=F32, device=DEV) for k in (3, 3, 9, 9)]
    hw = (c["height"], c["width"])
    return dict(kind="views", obs=obs, state=B.MpmState(x, zero[1], zero[2], F), target=target,
                g=B.MpmState(*zero), loss=torch.zeros(1, dtype=F32, device=DEV),
                scratch=torch.empty((2, 3) + hw, dtype=F32, device=DEV),
                ws=torch.empty(30 * hw[0] * hw[1], dtype=F32, device=DEV),
                weight=1.0 / (3 * hw[0] * hw[1]))


# --------------------------------------------------------------------- run --

def run(state):
    return globals()["_run_" + state["kind"]](state)


def _run_substep(s):
    s["mpm"].substep(s["state"], s["out"], s["pin"], s["wind"], 0.0)
    return list(s["out"])


def _in_order(a, ids):
    out = torch.empty_like(a)
    out[:, ids] = a
    return out


def _run_rollout(s):
    s["ro"].load(s["state"], s["pin"])
    st, ids = s["ro"].run()
    ids = ids.long()
    return [_in_order(a, ids) for a in st]


def _run_frames(s):
    X = AG.mpm_frames(s["mpm"], s["state"], s["wind"], s["total"], s["E"], s["substeps"], s["every"],
                      pinned=s["pin"])
    loss = ((X - s["target"]) ** 2).sum() / s["target"].shape[1]
    g = torch.autograd.grad(loss, [s["wind"], s["E"], *s["state"]])
    return [X.detach(), loss.detach(), *g]


def _run_batch(s):
    for a, b in zip(s["work"], s["state"]):
        a.copy_(b)
    s["ids"].copy_(s["ids0"])
    s["wpin"].copy_(s["pin"])
    s["batch"].rollout(s["work"], s["wpin"], s["ids"], 0.0, s["substeps"], s["sort"])
    ids = s["ids"].long()
    return [_in_order(a, ids) for a in s["work"]]


def _run_batch_adjoint(s):
    for a, b in zip(s["work"], s["g0"]):
        a.copy_(b)
    s["g_wind"].zero_()
    s["g_E"].zero_()
    s["batch"].segment_adjoint(s["state"], s["tape"], s["work"], s["pin"], 0.0, s["substeps"],
                               s["g_wind"], s["g_E"])
    return [*s["work"], s["g_wind"], s["g_E"]]


def _run_lbm(s):
    return s["lbm"].step(s["f"], s["solid"], s["steps"])


def _run_lbm_adjoint(s):
    f = AG.lbm_steps(s["lbm"], s["f"], s["solid"], s["steps"], s["every"])
    (g,) = torch.autograd.grad(f, s["f"], s["g"])
    return [f.detach(), g]


def _run_guide(s):
    u = s["guide"].advance(s["x"], s["steps"])
    return [u, s["guide"].f, s["guide"].solid]


def _run_surrogate(s):
    m = s["surr"]
    m.surr.features(s["f"], s["solid"], SU.IN_SCALE)
    for _ in range(s["blocks"]):
        m.chained_block(s["solid"])
    return m.surr.write_lattice(s["solid"], s["out"])


def _run_train(s):
    m = s["surr"]
    s["step"] += 1
    s["loss"].zero_()
    m.set_features(s["x"])
    m.forward(s["out"])
    m.loss(s["y"], s["loss"])
    m.backward()
    grads = m.grads()
    m.adam(LR, s["step"])
    return [s["out"], s["loss"], grads, m.params()]


def _run_views(s):
    s["loss"].zero_()
    s["g"].x.zero_()
    s["g"].F.zero_()
    s["obs"].loss(s["state"], s["target"], s["weight"], s["loss"], s["g"], s["scratch"], s["ws"])
    return [s["scratch"][0], s["loss"], s["g"].x, s["g"].F]


# -------------------------------------------------------------------- work --

def work(case):
    c, k = case, case["kind"]
    if k in ("substep", "rollout", "frames"):
        nf, fr = {"substep": (8, 1), "rollout": (32, 16)}.get(k) or (c["nf"], c["frames"])
        wind, st = 12 * nf ** 3 * fr, 96 * c["n"]
        steps = 1 if k == "substep" else c["substeps"]
        if k == "frames":  # the frames and, for each input, its gradient
            return dict(bytes=2 * (wind + st) + 24 * c["n"] * (steps // c["every"]),
                        flops=3 * 1991.0 * c["n"] * steps)
        return dict(bytes=wind + 2 * st, flops=1991.0 * c["n"] * steps)
    if k in ("batch", "batch_adjoint"):
        n, wind = sum(p[1] for p in _batch_plan(c)), 12 * 16 ** 3 * 8 * c["scenes"]
        if k == "batch":
            return dict(bytes=192 * n + wind, flops=1991.0 * n * c["substeps"])
        return dict(bytes=3 * 96 * n + 2 * wind, flops=3 * 1991.0 * n * c["substeps"])
    if k in ("lbm", "lbm_adjoint"):
        cells = c["nx"] * c["ny"] * c["nz"]
        if k == "lbm":
            return dict(bytes=(2 * 76 + 1) * cells, flops=300.0 * cells * c["steps"])
        return dict(bytes=(4 * 76 + 1) * cells, flops=3 * 300.0 * cells * c["steps"])
    if k == "guide":
        cells, per = c["cells"] ** 3, 40 if c["model"] == "home" else 76
        return dict(bytes=(2 * per + 1) * cells + 12 * c["n"] + 24 * c["nf"] ** 3,
                    flops=400.0 * cells * c["steps"])
    conv = 2.0 * 27 * (5 * 32 + 2 * 32 * 32 + 32 * 3)
    if k == "surrogate":
        return dict(bytes=(2 * 76 + 1) * 8 * c["n"] ** 3, flops=c["blocks"] * conv * c["n"] ** 3)
    if k == "train":
        return dict(bytes=(64 + 64 + 12) * c["n"] ** 3 + 4 * 4 * 83056,
                    flops=3 * conv * c["n"] ** 3)
    px = c["width"] * c["height"]
    return dict(bytes=(12 + 36 + 24 + 16 + 48) * c["n"] + 24 * px * c["views"],
                flops=c["views"] * (400.0 * c["n"] + 1000.0 * px))


# ------------------------------------------------------- values in 64 bits --

def exact(case, seed):
    return globals()["_exact_" + case["kind"]](case, seed)


def _mat(a):
    return a.view(3, 3, -1)


def _mm(a, b):
    return (a.unsqueeze(2) * b.unsqueeze(0)).sum(1)


def _cof(a):
    r = [torch.linalg.cross(a[(i + 1) % 3], a[(i + 2) % 3], dim=0) for i in range(3)]
    return torch.stack(r)


def _kirchhoff(material, F, mu, lam):
    """P F^T of the two constitutive models."""
    eye = torch.eye(3, dtype=F64, device=F.device).unsqueeze(-1)
    J = (F[0] * torch.linalg.cross(F[1], F[2], dim=0)).sum(0)
    if material == 0:
        return mu * (_mm(F, F.transpose(0, 1)) - eye) + lam * torch.log(J) * eye
    R = F
    for _ in range(6):  # Newton's iteration to the rotation of F
        K = _cof(R)
        R = 0.5 * (R + K / (R[0] * K[0]).sum(0))
    return 2 * mu * _mm(F - R, F.transpose(0, 1)) + lam * (J - 1) * J * eye


def _wind_at_nodes(wind, total, t, N):
    """a_w [3][N^3] at the grid nodes (i, j, k) / N."""
    fr, nf = wind.shape[0], wind.shape[1]
    if fr > 1:
        s = min(max(t / total, 0.0), 1.0) * (fr - 1)
        k = min(int(s), fr - 2)
        w = (1 - (s - k)) * wind[k] + (s - k) * wind[k + 1]
    else:
        w = wind[0]
    p = torch.arange(N, dtype=F64, device=wind.device) / N * (nf - 1)
    i = p.floor().clamp(max=nf - 2).long()
    M = torch.zeros((N, nf), dtype=F64, device=wind.device)
    r = torch.arange(N, device=wind.device)
    M[r, i] = 1 - (p - i)
    M[r, i + 1] = p - i
    w = torch.einsum("xa,zyac->zyxc", M, w)
    w = torch.einsum("yb,zbxc->zyxc", M, w)
    return torch.einsum("zd,dyxc->czyx", M, w).reshape(3, -1)


def _substep64(pr, E, s, pinned, wind, total, t):
    x, v, C, F = s
    N, dt = pr["n_grid"], float(np.float32(pr["dt"]))
    m, vol = float(np.float32(pr["p_mass"])), float(np.float32(pr["p_vol"]))
    nu = float(np.float32(pr["nu"]))
    mu, lam = E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))
    X = x * N
    base = (X.detach() - 0.5).floor()
    f = X - base
    w = torch.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2])
    o = torch.arange(3, device=x.device)
    ok, oj, oi = (a.reshape(-1) for a in torch.meshgrid(o, o, o, indexing="ij"))
    W = w[oi, 0] * w[oj, 1] * w[ok, 2]  # [27][n]
    d = (torch.stack([oi, oj, ok], 1).to(F64).unsqueeze(-1) - f.unsqueeze(0)) / N  # [27][3][n]
    b = base.long()
    idx = ((b[2] + ok.unsqueeze(1)) * N + b[1] + oj.unsqueeze(1)) * N + b[0] + oi.unsqueeze(1)
    Fm = _mat(F)
    A = m * _mat(C) - dt * vol * 4 * N * N * _kirchhoff(pr["material"], Fm, mu, lam)
    mom = [W * (m * v[a] + (A[a].unsqueeze(0) * d).sum(1)) for a in range(3)]
    flat = idx.reshape(-1)
    zero = torch.zeros(N ** 3, dtype=F64, device=x.device)
    gm = zero.index_add(0, flat, (m * W).reshape(-1))
    q = torch.arange(N, device=x.device)
    inside = (q >= pr["bc_band"]) & (q <= N - 1 - pr["bc_band"])
    free = (inside.view(-1, 1, 1) & inside.view(1, -1, 1) & inside.view(1, 1, -1)).reshape(-1) & (gm.detach() > 0)
    den = torch.where(free, gm, torch.ones_like(gm))
    aw = _wind_at_nodes(wind, total, t, N)
    vp, Cp = [], []
    for a in range(3):
        va = zero.index_add(0, flat, mom[a].reshape(-1)) / den + dt * (float(np.float32(pr["gravity"][a])) + aw[a])
        gv = W * torch.where(free, va, zero)[idx]
        vp.append(gv.sum(0))
        Cp.append(4 * N * N * (gv.unsqueeze(1) * d).sum(0))
    vp, Cp = torch.stack(vp), torch.stack(Cp)
    Fn = (Fm + dt * _mm(Cp, Fm)).reshape(9, -1)
    xn, Cp = x + dt * vp, Cp.reshape(9, -1)
    if pinned is not None:
        p = pinned.bool()
        vp, Cp = torch.where(p, 0.0, vp), torch.where(p, 0.0, Cp)
        xn, Fn = torch.where(p, x, xn), torch.where(p, F, Fn)
    return xn, vp, Cp, Fn


def _steps64(sc, steps, every=0, E=None):
    """(state after the steps, positions after each `every`)."""
    pr, st, pin, wind, total = sc
    E = float(np.float32(pr["E"])) if E is None else E
    frames = []
    for k in range(steps):
        st = _substep64(pr, E, st, pin, wind, total, k * float(np.float32(pr["dt"])))
        if every and (k + 1) % every == 0:
            frames.append(st[0])
    return st, frames


def _wide(sc, grad=False):
    pr, st, pin, wind, total = sc
    up = [a.to(F64).requires_grad_(grad) for a in (*st, wind)]
    return pr, tuple(up[:4]), pin, up[4], total


def _exact_substep(c, seed):
    sc = _scene(c["shape"], c["n"], c["n_grid"], c["material"], 8, 1, 1, seed)
    return list(_steps64(_wide(sc), 1)[0])


def _exact_rollout(c, seed):
    sc = _scene(c["shape"], c["n"], c["n_grid"], c["material"], 32, 16, c["substeps"], seed)
    return list(_steps64(_wide(sc), c["substeps"])[0])


def _exact_frames(c, seed):
    sc = _scene(c["shape"], c["n"], c["n_grid"], c["material"], c["nf"], c["frames"], c["substeps"], seed)
    target = _frames_target(sc[1][0]).to(F64)
    sc = _wide(sc, True)
    E = torch.tensor(sc[0]["E"], dtype=F64, device=DEV, requires_grad=True)
    _, frames = _steps64(sc, c["substeps"], c["every"], E)
    X = torch.stack(frames)
    loss = ((X - target) ** 2).sum() / target.shape[1]
    g = torch.autograd.grad(loss, [sc[3], E, *sc[1]])
    return [X.detach(), loss.detach(), *g]


def _exact_batch(c, seed):
    if c["substeps"] * sum(p[1] for p in _batch_plan(c)) > 4e8:
        return None
    outs = [_steps64(_wide(s), c["substeps"])[0] for s in _batch_scenes(c, seed)]
    return [torch.cat([o[k] for o in outs], 1) for k in range(4)]


def _exact_batch_adjoint(c, seed):
    n = sum(p[1] for p in _batch_plan(c))
    g0 = [a.to(F64) for a in _batch_seed_grad(n, seed)]
    got, at = [], 0
    for s in _batch_scenes(c, seed):
        s = _wide(s, True)
        E = torch.tensor(s[0]["E"], dtype=F64, device=DEV, requires_grad=True)
        out, _ = _steps64(s, c["substeps"], 0, E)
        m = out[0].shape[1]
        got.append(torch.autograd.grad(out, [*s[1], s[3], E], [a[:, at:at + m] for a in g0]))
        at += m
    return [*(torch.cat([g[k] for g in got], 1) for k in range(4)),
            torch.cat([g[4].reshape(-1) for g in got]), torch.stack([g[5] for g in got])]


def _collide64(f, tau, force):
    """Post-collision populations (unshifted) of [19][nz][ny][nx]."""
    rho = f.sum(0)
    u = torch.stack([sum(c[i] * f[i] for i in range(19)) + 0.5 * force[a]
                     for a, c in enumerate((CX, CY, CZ))]) / rho
    uu = 1.5 * (u * u).sum(0)
    out = []
    for i in range(19):
        c = (CX[i], CY[i], CZ[i])
        cu = sum(c[a] * u[a] for a in range(3))
        feq = WQ[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - uu)
        src = sum((3 * (c[a] - u[a]) + 9 * cu * c[a]) * force[a] for a in range(3))
        out.append(f[i] - (f[i] - feq) / tau + (1 - 0.5 / tau) * WQ[i] * src)
    return out


def _stream64(post, solid, bc_x, inlet):
    """Pulled populations [19]: bounce-back at solid sources, inlet and outlet faces."""
    nx = post[0].shape[2]
    xs = torch.arange(nx, device=post[0].device).view(1, 1, -1)
    out = []
    for i in range(19):
        sh = (CZ[i], CY[i], CX[i])
        p = torch.roll(post[i], sh, (0, 1, 2))
        if solid is not None:
            p = torch.where(torch.roll(solid, sh, (0, 1, 2)), post[OPP[i]], p)
        if bc_x and CX[i]:
            p = torch.where(xs == 0, inlet[i], p) if CX[i] > 0 else torch.where(xs == nx - 1, post[i], p)
        out.append(p)
    return out


def _lbm64(c, f, solid, u_in, steps):
    wq = torch.tensor(WQ, dtype=F64, device=DEV).view(19, 1, 1, 1)
    tau = float(np.float32(TAU))
    u = torch.tensor([float(np.float32(a)) for a in u_in], dtype=F64, device=DEV)
    inlet = _feq(torch.ones((), dtype=F64, device=DEV), u) + wq.view(19)
    force = (float(np.float32(c.get("force", 0.0))), 0.0, 0.0)
    f, sb = f + wq, solid.bool()
    for _ in range(steps):
        fn = torch.stack(_stream64(_collide64(f, tau, force), sb, c["bc_x"], inlet))
        f = torch.where(sb, f, fn)
    return f - wq


def _exact_lbm(c, seed):
    f, solid, u_in = _flow(c["nz"], c["ny"], c["nx"], seed)
    return _lbm64(c, f.to(F64), solid, u_in, c["steps"])


def _exact_lbm_adjoint(c, seed):
    f, solid, u_in = _flow(c["nz"], c["ny"], c["nx"], seed)
    with torch.no_grad():  # the state before each step, then one step at a time backwards
        states = [f.to(F64)]
        for _ in range(c["steps"]):
            states.append(_lbm64(c, states[-1], solid, u_in, 1))
    g = _lattice_grad(f, seed).to(F64)
    for a in reversed(states[:-1]):
        a = a.requires_grad_(True)
        (g,) = torch.autograd.grad(_lbm64(c, a, solid, u_in, 1), a, g)
    return [states[-1], g]


def _rebuild64(m):
    """Populations (a list of 19) of the HOME moments rho, u, S."""
    rho, u = m[0], m[1:4]
    S = {(0, 0): m[4], (1, 1): m[5], (2, 2): m[6], (0, 1): m[7], (0, 2): m[8], (1, 2): m[9]}
    out = []
    for i in range(19):
        c = (CX[i], CY[i], CZ[i])
        e = 1 + 3 * sum(c[a] * u[a] for a in range(3))
        for (a, b), s in S.items():
            e = e + (4.5 * (c[a] * c[a] - 1 / 3) * s if a == b else 9.0 * c[a] * c[b] * s)
        for a in range(3):
            for b in range(3):
                h = c[b] * (c[a] * c[a] - 1 / 3)
                if a != b and h:
                    A = u[b] * S[a, a] + 2 * u[a] * S[min(a, b), max(a, b)] - 2 * u[a] * u[a] * u[b]
                    e = e + 13.5 * h * A
        out.append(WQ[i] * rho * e)
    return out


def _home64(m, solid, u_in, tau, steps):
    one = torch.ones((), dtype=F64, device=DEV)
    u = [one * float(np.float32(a)) for a in u_in]
    inlet = _rebuild64(torch.stack([one, *u, *(u[a] * u[b] for a, b in
                                               ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)))]))
    sb = solid.bool()
    for _ in range(steps):
        f = _stream64(_rebuild64(m), sb, 1, inlet)
        rho = sum(f)
        j = [sum(c[i] * f[i] for i in range(19)) for c in (CX, CY, CZ)]
        v = [a / rho for a in j]
        cc = (CX, CY, CZ)
        pi = {(a, b): sum(cc[a][i] * cc[b][i] * f[i] for i in range(19)) for a in range(3) for b in range(a, 3)}
        nq = {k: p - rho * ((k[0] == k[1]) / 3 + v[k[0]] * v[k[1]]) for k, p in pi.items()}
        tr = (nq[0, 0] + nq[1, 1] + nq[2, 2]) / 3
        S = {k: v[k[0]] * v[k[1]] + (1 - 1 / tau) * (q - (tr if k[0] == k[1] else 0)) / rho for k, q in nq.items()}
        mn = torch.stack([rho, *v, S[0, 0], S[1, 1], S[2, 2], S[0, 1], S[0, 2], S[1, 2]])
        m = torch.where(sb, m, mn)
    return m


def _exact_guide(c, seed):
    x, u_in = _guide_inputs(c, seed)
    n = c["cells"]
    w = (x / float(np.float32(1.0 / n))).floor().long()
    solid = torch.zeros((n, n, n), dtype=torch.uint8, device=DEV)
    solid[w[2], w[1], w[0]] = 1
    tau, one = float(np.float32(0.6)), torch.ones((n, n, n), dtype=F64, device=DEV)
    u = [one * float(np.float32(a)) for a in u_in]
    if c["model"] == "home":
        m = torch.stack([one, *u, u[0] * u[0], u[1] * u[1], u[2] * u[2], u[0] * u[1], u[0] * u[2], u[1] * u[2]])
        m = _home64(m, solid, u_in, tau, c["steps"])
        vel, out = m[1:4], torch.cat([m[:1] - 1, m[1:]])
    else:
        wq = torch.tensor(WQ, dtype=F64, device=DEV).view(19, 1, 1, 1)
        f = _feq(one, torch.stack(u)) + wq
        inlet = f[:, 0, 0, 0].clone()
        for _ in range(c["steps"]):
            f = torch.where(solid.bool(), f, torch.stack(
                _stream64(_collide64(f, tau, (0.0, 0.0, 0.0)), solid.bool(), 1, inlet)))
        vel = torch.stack([sum(k[i] * f[i] for i in range(19)) for k in (CX, CY, CZ)]) / f.sum(0)
        out = f - wq
    vel = torch.where(solid.bool(), 0.0, vel)
    # trilinear between cell centres at the wind nodes
    p = (torch.linspace(0, 1, c["nf"], dtype=F64, device=DEV) * n - 0.5).clamp(0, n - 1)
    i = p.floor().clamp(max=n - 2).long()
    M = torch.zeros((c["nf"], n), dtype=F64, device=DEV)
    r = torch.arange(c["nf"], device=DEV)
    M[r, i] = 1 - (p - i)
    M[r, i + 1] = p - i
    for e in ("xa,czya->czyx", "yb,czbx->czyx", "zd,cdyx->czyx"):
        vel = torch.einsum(e, M, vel)
    return [vel.reshape(3, -1), out, solid]


def _net64(x, params, n):
    """The network on channels-last features [n^3][16]; GELU in its tanh form."""
    ch, at = (16, 32, 32, 32, 16), 0
    a = x.view(n, n, n, 16)
    for k in range(4):
        w = params[at:at + 27 * ch[k] * ch[k + 1]].view(27, ch[k + 1], ch[k])
        at += w.numel()
        b = params[at:at + ch[k + 1]]
        at += ch[k + 1]
        pad = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        z = b.expand(n, n, n, ch[k + 1])
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            z = z + pad[dz:dz + n, dy:dy + n, dx:dx + n] @ w[t].t()
        a = torch.nn.functional.gelu(z, approximate="tanh") if k < 3 else z
    return a.reshape(-1, 16)


def _exact_surrogate(c, seed):
    n = c["n"]
    f32, solid, _ = _flow(2 * n, 2 * n, 2 * n, seed)
    f, sb = f32.to(F64), solid.bool()
    rho = torch.where(sb, 1.0, 1.0 + f.sum(0))
    u = torch.stack([sum(k[i] * f[i] for i in range(19)) for k in (CX, CY, CZ)]) / rho
    u = torch.where(sb, 0.0, u)
    params = torch.from_numpy(_weights()).to(DEV).to(F64)
    fluid = (~sb).to(F64)
    pool = lambda a: a.view(a.shape[:-3] + (n, 2, n, 2, n, 2)).sum((-5, -3, -1))
    cnt = pool(fluid)
    p = (torch.arange(2 * n, dtype=F64, device=DEV) * 0.5 - 0.25).clamp(0, n - 1)
    i = p.floor().clamp(max=n - 2).long()
    M = torch.zeros((2 * n, n), dtype=F64, device=DEV)
    r = torch.arange(2 * n, device=DEV)
    M[r, i] = 1 - (p - i)
    M[r, i + 1] = p - i
    for _ in range(c["blocks"]):
        x = torch.zeros((n, n, n, 16), dtype=F64, device=DEV)
        mean = pool(torch.cat([(rho - 1).unsqueeze(0), u]) * fluid) / cnt.clamp(min=1) / 0.05
        x[..., :4] = mean.permute(1, 2, 3, 0)
        x[..., 4] = 1 - cnt / 8
        du = _net64(x.view(-1, 16), params, n)[:, :3].t().reshape(3, n, n, n)
        for e in ("xa,czya->czyx", "yb,czbx->czyx", "zd,cdyx->czyx"):
            du = torch.einsum(e, M, du)
        u = torch.where(sb, 0.0, u + 1e-3 * du)
    return torch.where(sb, f, _feq(rho, u))


def _exact_train(c, seed):
    x, y = (a.to(F64) for a in _coarse_inputs(c["n"], seed))
    params = torch.from_numpy(_weights()).to(DEV).to(F64).requires_grad_(True)
    out = _net64(x, params, c["n"])
    fluid = (x[:, 4:5] < 1).to(F64)
    loss = (((out - y)[:, :3] ** 2) * fluid).sum() / (3 * fluid.sum())
    (g,) = torch.autograd.grad(loss, params)
    return [out.detach(), loss.detach().reshape(1), g, (params - LR * g / (g.abs() + 1e-8)).detach()]


def _image64(x, F, s0, col, opa, cam):
    """Alpha-blended image [3][H][W] from the list of (Gaussian, pixel) pairs
    inside three standard deviations, ordered by pixel and depth."""
    H, W = cam["height"], cam["width"]
    R, T = (torch.tensor(cam[k], dtype=F64, device=DEV) for k in ("R", "T"))
    fx, fy = float(np.float32(cam["fx"])), float(np.float32(cam["fy"]))
    t = R @ x + T.view(3, 1)
    Fm = _mat(F)
    S = torch.stack([torch.stack([s0[0], s0[3], s0[4]]), torch.stack([s0[3], s0[1], s0[5]]),
                     torch.stack([s0[4], s0[5], s0[2]])])
    Sig = _mm(_mm(Fm, S), Fm.transpose(0, 1))
    zero = torch.zeros_like(t[0])
    Jm = torch.stack([torch.stack([fx / t[2], zero, -fx * t[0] / t[2] ** 2]),
                      torch.stack([zero, fy / t[2], -fy * t[1] / t[2] ** 2])])
    A = (Jm.unsqueeze(2) * R.unsqueeze(-1).unsqueeze(0)).sum(1)
    cov = _mm(_mm(A, Sig), A.transpose(0, 1))
    a, b, d = cov[0, 0], cov[0, 1], cov[1, 1]
    mx, my = fx * t[0] / t[2] + cam["cx"], fy * t[1] / t[2] + cam["cy"]
    with torch.no_grad():
        rx, ry = 3 * a.sqrt(), 3 * d.sqrt()
        x0, x1 = (mx - rx - 0.5).ceil().clamp(0, W), (mx + rx - 0.5).floor().clamp(-1, W - 1)
        y0, y1 = (my - ry - 0.5).ceil().clamp(0, H), (my + ry - 0.5).floor().clamp(-1, H - 1)
        nx, ny = (x1 - x0 + 1).clamp(min=0).long(), (y1 - y0 + 1).clamp(min=0).long()
        ok = (t[2] > 0.01) & (a * d - b * b > 0)
        cnt = nx * ny * ok
        gid = torch.repeat_interleave(torch.arange(cnt.numel(), device=DEV), cnt)
        k = torch.arange(gid.numel(), device=DEV) - (cnt.cumsum(0) - cnt)[gid]
        px, py = x0[gid].long() + k % nx[gid], y0[gid].long() + k // nx[gid]

    def q_of(gid, px, py):
        dx, dy = px + 0.5 - mx[gid], py + 0.5 - my[gid]
        return (d[gid] * dx * dx - 2 * b[gid] * dx * dy + a[gid] * dy * dy) / (a * d - b * b)[gid]

    with torch.no_grad():
        keep = q_of(gid, px, py) <= 9
        gid, px, py = gid[keep], px[keep], py[keep]
        rank = torch.empty_like(t[2], dtype=torch.long)
        rank[torch.sort(t[2], stable=True)[1]] = torch.arange(t.shape[1], device=DEV)
        order = torch.argsort((py * W + px) * t.shape[1] + rank[gid])
        gid, px, py = gid[order], px[order], py[order]
        pix = py * W + px
        new = torch.ones_like(pix, dtype=torch.bool)
        new[1:] = pix[1:] != pix[:-1]
        first = new.nonzero().view(-1)[new.long().cumsum(0) - 1]
    alpha = opa[gid] * torch.exp(-0.5 * q_of(gid, px, py))
    lt = torch.log1p(-alpha)
    before = lt.cumsum(0) - lt
    Tr = torch.exp(before - before[first])
    img = torch.zeros((3, H * W), dtype=F64, device=DEV)
    return img.index_add(1, pix, Tr * alpha * col[:, gid]).view(3, H, W)


def _dssim64(img, tgt):
    k = torch.exp(-0.5 * ((torch.arange(11, dtype=F64, device=DEV) - 5) / 1.5) ** 2)
    k = (k / k.sum()).view(1, 1, 11, 1)

    def blur(a):
        a = torch.nn.functional.conv2d(a.unsqueeze(1), k, padding=(5, 0))
        return torch.nn.functional.conv2d(a, k.transpose(2, 3), padding=(0, 5)).squeeze(1)
    mx, my = blur(img), blur(tgt)
    sx, sy, sxy = blur(img * img) - mx * mx, blur(tgt * tgt) - my * my, blur(img * tgt) - mx * my
    s = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
    return 1 - s.mean()


def _exact_views(c, seed):
    x, F, s0, col, opa, cams, target = _view_inputs(c, seed)
    x, F = x.to(F64).requires_grad_(True), F.to(F64).requires_grad_(True)
    s0, col, opa, target = (a.to(F64) for a in (s0, col, opa, target))
    loss = 0.0
    for cam, tgt in zip(cams, target):
        img = _image64(x, F, s0, col, opa, cam)
        loss = loss + 0.9 * (img - tgt).abs().mean() + 0.1 * _dssim64(img, tgt)
    gx, gF = torch.autograd.grad(loss, [x, F])
    return [img.detach(), loss.detach().reshape(1), gx, gF]
