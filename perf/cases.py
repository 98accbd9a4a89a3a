"""The work that a user of this library has it do, as cases that can be timed and checked.

Kinds of case (key "kind"):
  lbm      start fields -> re-initialisation -> `steps` time steps -> statistics -> (rho, u): plain LBM
           trajectories, from one small channel (launch latency counts) to batches of porous media and
           one large domain (bandwidth counts)
  couple   the hybrid's hand-over: re-initialisation from fields, moments, vorticity, no time step between
  fno      one FNO inference pass (bfloat16 operands)
  train    FNO training pass: forward with saved activations, and its reverse mode (FP32)
  rollout  differentiable LBM: re-initialisation, `steps` steps, moments, and the adjoint of all of it
  steady   the steady hybrid driver: FNO start, then LBM with a residual check every 100 steps
  unsteady the super-time-stepping driver: cycles of LBM steps, FNO steps and re-initialisation

exact() restates each of them in 64-bit torch, without this library.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F
from torch.utils.checkpoint import checkpoint

from paper_2604_27158_gb300.adjoint import lbm_rollout
from paper_2604_27158_gb300.fno import Fno, FnoShape, Hybrid, HybridConfig
from paper_2604_27158_gb300.lbm import BC_PERIODIC, BC_PRESSURE, BC_VELOCITY, GridSpec, Lattice
from paper_2604_27158_gb300.train import fno_apply

# grid sizes (nx, ny) of the batches of uneven trajectories
UNEVEN = ((128, 128), (256, 128), (256, 256), (512, 256))
SHEAR_TAU, SHEAR_U = 0.5220, 0.0574  # double shear layer at 128 cells, 223 steps per FNO step


def listed():
    net = dict(c_in=4, c_out=3, width=32, layers=4, modes=12, dec_layers=1, dec_size=32, act="gelu", pad=0)
    return [
        # the plain-LBM workload: one body-force channel, where a step is latency and launches
        dict(name="lbm_channel_128x64", kind="lbm", scene="channel", nx=128, ny=64, grids=1, steps=100),
        # trajectories of uneven size past disks (velocity inlet, pressure outlet), advanced as one batch
        dict(name="lbm_uneven_100", kind="lbm", scene="disks", nx=0, ny=0, grids=100, steps=50),
        # the porous-media batch between two residual checks of the steady solve
        dict(name="lbm_porous_64x512x256", kind="lbm", scene="porous", nx=512, ny=256, grids=64, steps=100),
        # one large domain, far beyond L2
        dict(name="lbm_domain_4096", kind="lbm", scene="porous", nx=4096, ny=4096, grids=1, steps=20),
        # what an FNO prediction costs on its way back into the lattice, and the accuracy metric
        dict(name="couple_64x512x256", kind="couple", scene="porous", nx=512, ny=256, grids=64, steps=0),
        # FNO throughput: batch of LBM snapshots through the 32-channel network
        dict(name="fno_b32_256", kind="fno", B=32, H=256, W=256, **net),
        # one trajectory's prediction with the padded porous density network: latency
        dict(name="fno_b1_porous_density", kind="fno", B=1, H=256, W=512, c_in=1, c_out=1, width=16, layers=3,
             modes=6, dec_layers=3, dec_size=32, act="gelu", pad=9),
        # the larger network's training pass of the differentiable hybrid step
        dict(name="train_c64_b8_512", kind="train", B=8, H=512, W=512, c_in=4, c_out=3, width=64, layers=4,
             modes=13, dec_layers=1, dec_size=64, act="gelu", dx=False),
        # a minibatch of the offline training on steady states
        dict(name="train_c32_b8_256x512", kind="train", B=8, H=256, W=512, c_in=4, c_out=3, width=32, layers=4,
             modes=12, dec_layers=1, dec_size=32, act="gelu", dx=False),
        # the LBM half of the differentiable hybrid step: 32 steps, checkpoints every 8
        dict(name="rollout_b8_512", kind="rollout", scene="porous", nx=512, ny=512, grids=8, steps=32, every=8),
        # whole call: the first 400 steps of the steady solve of 20 porous media from the FNO start
        dict(name="steady_porous_20", kind="steady", nx=512, ny=256, grids=20, steps=400, **net),
        # whole call: one 1:1 cycle of the double-shear pair of networks (223 steps per FNO step)
        dict(name="unsteady_shear_100", kind="unsteady", nx=128, ny=128, grids=100, k=223, m=1, cycles=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice_draw(rng, most):
    """A batch of equal grids of any size and shape, at most `most` cells in all."""
    cells = _log(rng, 2000, most)
    grids = _log(rng, 1, max(1, min(100, cells // 1500)))
    per = cells / grids
    ratio = math.exp(rng.uniform(-0.9, 1.1))
    ny = min(4096, max(24, int(math.sqrt(per / ratio))))
    return dict(nx=min(8192, max(24, int(per / ny))), ny=ny, grids=grids)


def draw(rng):
    kind = rng.choice(["lbm", "lbm", "lbm", "couple", "fno", "fno", "train", "train", "rollout", "steady", "unsteady"])
    if kind in ("lbm", "couple", "rollout"):
        scene = rng.choice(["channel", "disks", "porous", "shear"])
        d = _lattice_draw(rng, 2_000_000 if kind == "rollout" else 16_000_000)
        cells = d["nx"] * d["ny"] * d["grids"]
        steps = 0 if kind == "couple" else rng.randint(1, 32) if kind == "rollout" else _log(rng, 1, 200)
        steps = min(steps, max(1, int(8e8 / cells))) if steps else 0
        more = dict(every=rng.randint(1, 9)) if kind == "rollout" else {}
        return dict(kind=kind, scene=scene, steps=steps, **d, **more)
    if kind == "steady":
        return dict(kind=kind, nx=_log(rng, 96, 512), ny=_log(rng, 48, 300), grids=rng.randint(1, 12),
                    steps=rng.choice([100, 150, 200, 350]), c_in=4, c_out=3, width=32, layers=4, modes=12,
                    dec_layers=1, dec_size=32, act="gelu", pad=0)
    if kind == "unsteady":
        n = rng.choice([96, 128, 128, 150])
        return dict(kind=kind, nx=n, ny=n, grids=_log(rng, 1, 80), k=rng.choice([50, 101, 223]), m=1,
                    cycles=rng.randint(1, 2))
    width = rng.choice([8, 14, 16, 16, 32, 32, 32, 48, 64, 64])
    modes = rng.choice([4, 6, 8, 12, 12, 13, 16, 20, 32])
    H, W = (max(2 * modes + 2, _log(rng, 40, 600)) for _ in range(2))
    per = 8 * 512 * 512 * 64 if kind == "train" else 100 * 128 * 128 * 32
    B = max(1, min(_log(rng, 1, 64), int(per / (H * W * max(16, width)) * 24 / max(24, 2 * modes))))
    c = dict(kind=kind, B=B, H=H, W=W, c_in=rng.choice([1, 2, 4]), c_out=rng.choice([1, 2, 3]), width=width,
             layers=rng.randint(1, 4), modes=modes, dec_layers=rng.choice([1, 1, 1, 3]),
             dec_size=rng.choice([16, 32, 32, 64]), act=rng.choice(["gelu", "gelu", "gelu", "relu"]))
    return dict(c, pad=rng.choice([0, 0, 9])) if kind == "fno" else dict(c, dx=rng.random() < 0.4)


# ------------------------------------------------------------------ inputs
def _sizes(case):
    if case.get("scene") == "disks" and not case["nx"]:
        return sorted(UNEVEN[i] for i in np.random.RandomState(case["grids"]).randint(0, 4, case["grids"]))
    return [(case["nx"], case["ny"])] * case["grids"]


def _disks(nx, ny, disks, wrap_x):
    """Solid cells of integer disks (cx, cy, r) [ny, nx]; y wraps, x wraps if asked."""
    s = np.zeros((ny, nx), bool)
    for cx, cy, r in disks:
        xs, ys = np.arange(cx - r, cx + r + 1), np.arange(cy - r, cy + r + 1)
        xs = xs if wrap_x else xs[(xs >= 0) & (xs < nx)]
        inside = (xs[None, :] - cx) ** 2 + (ys[:, None] - cy) ** 2 <= r * r
        s[np.ix_(ys % ny, xs % nx)] |= inside
    return s


def _geometry(scene, nx, ny, rs):
    """(GridSpec, solid) of one grid: obstacles are a jittered array of disks that do not overlap."""
    if scene == "shear":
        return GridSpec(nx, ny, SHEAR_TAU), np.zeros((ny, nx), bool)
    small = min(nx, ny) < 64
    rmin, rmax = (2, 4) if small else (4, 8) if scene == "channel" else (4, 12)
    cell = 2 * rmax + 4
    spots = [(i, j) for j in range(max(1, (ny - 2) // cell)) for i in range(max(1, (nx - 4) // cell))]
    if scene == "channel":
        spots = [spots[i] for i in rs.permutation(len(spots))[:6]]
    elif scene == "disks":
        mid = [s for s in spots if 0.2 * nx < 2 + s[0] * cell < 0.8 * nx - cell] or spots
        spots = [mid[i] for i in rs.permutation(len(mid))[:rs.randint(1, 5)]]
    disks = []
    for i, j in spots:
        r = int(rs.randint(rmin, rmax + 1))
        ox, oy = (int(rs.randint(r + 1, cell - r)) for _ in range(2))
        disks.append((2 + i * cell + ox, 1 + j * cell + oy, r))
    solid = _disks(nx, ny, disks, scene == "channel")
    if scene == "channel":
        solid[0] = solid[-1] = True
        return GridSpec(nx, ny, 0.8, fx=1e-6), solid
    solid[:, 0] = solid[:, -1] = False
    if scene == "disks":
        tau = float(rs.uniform(0.55, 0.8))
        u = min(float(rs.uniform(50, 200)) * (tau - 0.5) / 3.0 / ny, 0.08)
        return GridSpec(nx, ny, tau, bc_west=BC_VELOCITY, bc_east=BC_PRESSURE, west_value=u, east_value=1.0), solid
    return GridSpec(nx, ny, 0.7, bc_west=BC_PRESSURE, bc_east=BC_PRESSURE, west_value=1.001, east_value=1.0), solid


def _batch(case, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    grids, solid = zip(*(_geometry(case.get("scene", "porous"), nx, ny, rs) for nx, ny in _sizes(case)))
    return list(grids), list(solid)


def _fields(grids, scene, gen, drho=1e-3, umax=0.02):
    """Smooth (rho, u_x, u_y) of every grid, dense and concatenated, on the GPU."""
    out = [[], [], []]
    for g in grids:
        r = torch.rand(16, generator=gen, device="cuda", dtype=torch.float64).tolist()
        x = (torch.arange(g.nx, device="cuda", dtype=torch.float64) + 0.5)[None, :] / g.nx
        y = (torch.arange(g.ny, device="cuda", dtype=torch.float64) + 0.5)[:, None] / g.ny
        if scene == "shear":
            a1, a2, up, lo = 20 + 105 * r[0], 20 + 105 * r[1], 0.65 + 0.2 * r[2], 0.15 + 0.2 * r[3]
            ux = SHEAR_U * torch.where(y >= 0.5, torch.tanh(a1 * (up - y)), torch.tanh(a2 * (y - lo))).expand(g.ny, g.nx)
            uy = (SHEAR_U * 0.1 * torch.sin(2 * math.pi * (x + 0.25))).expand(g.ny, g.nx)
            f = (torch.ones_like(ux), ux, uy)
        else:
            waves = [sum(torch.cos(2 * math.pi * (int(4 * r[6 * w + 2 * k]) * x + int(4 * r[(6 * w + 2 * k + 1) % 16]) * y
                                                  + r[(3 * w + 5 * k) % 16])) for k in range(3)) / 3 for w in range(2)]
            f = (1 + drho * waves[0], umax * waves[1], umax * waves[0].flip(0) * 0.5)
        for o, v in zip(out, f):
            o.append(v.float().reshape(-1))
    return [torch.cat(o).contiguous() for o in out]


def _shapes(c):
    """Ordered shapes and initial ranges (lo, hi) of the parameter pack."""
    C, h, m, S = c["width"], c["width"] // 2, c["modes"], c["dec_size"]
    one = lambda o, i: [((o, i), -1 / math.sqrt(i), 1 / math.sqrt(i)), ((o,), -1 / math.sqrt(i), 1 / math.sqrt(i))]
    out = one(h, c["c_in"] + 2) + one(C, h)
    for _ in range(c["layers"]):
        out += [((C, C, m, m), 0.0, 1.0 / (C * C))] * 4 + one(C, C)
    fan = C
    for _ in range(c["dec_layers"]):
        out += one(S, fan)
        fan = S
    return out + one(c["c_out"], fan)


def _params(c, gen, out_scale=1.0):
    parts = [lo + (hi - lo) * torch.rand(int(np.prod(s)), generator=gen, device="cuda") for s, lo, hi in _shapes(c)]
    for k in (-1, -2):
        parts[k] = parts[k] * out_scale
    return torch.cat(parts)


def _shape(c):
    return FnoShape(c_in=c["c_in"], c_out=c["c_out"], width=c["width"], layers=c["layers"], modes=c["modes"],
                    dec_layers=c["dec_layers"], dec_size=c["dec_size"], activation=0 if c["act"] == "gelu" else 1,
                    padding=c.get("pad", 0))


def _net_input(c, gen):
    """Planes of (rho - 1, u_x, u_y, mask) as they come from the lattice; one plane: the mask."""
    B, H, W, n = c["B"], c["H"], c["W"], c["c_in"]
    low = torch.randn((B, n, max(2, H // 32), max(2, W // 32)), generator=gen, device="cuda")
    x = 0.02 * F.interpolate(low, size=(H, W), mode="bilinear", align_corners=True)
    if n in (1, 4):
        blobs = torch.randn((B, 1, max(2, H // 14), max(2, W // 14)), generator=gen, device="cuda")
        solid = F.interpolate(blobs, size=(H, W), mode="bilinear", align_corners=True) > 0.3
        x = x * ~solid
        x[:, n - 1:] = solid.float()
    return x.contiguous()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _pair(c):
    """Density and velocity networks of the double-shear layer."""
    base = dict(width=14, layers=3, dec_layers=1, dec_size=32, act="gelu", pad=9)
    return dict(base, c_in=1, c_out=1, modes=8), dict(base, c_in=2, c_out=2, modes=32)


def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    s = dict(case=case)
    if kind == "fno":
        s["net"] = Fno(_shape(case), _params(case, gen).cpu().numpy())
        s["x"] = _net_input(case, gen)
        return s
    if kind == "train":
        s["shape"] = _shape(case)
        s["params"] = torch.nn.Parameter(_params(case, gen))
        s["x"] = _net_input(case, gen).requires_grad_(case["dx"])
        s["dout"] = torch.randn((case["B"], case["c_out"], case["H"], case["W"]), generator=gen, device="cuda")
        return s
    if kind == "unsteady":
        case = dict(case, scene="shear")
    grids, solid = _batch(case, seed)
    s["lat"] = Lattice(grids, solid, u_max=0.3 if kind == "unsteady" else 0.2)
    if kind in ("lbm", "steady"):
        s["lat"].autotune(reps=3)
    if kind == "steady":
        s["net"] = Fno(_shape(case), _params(case, gen, 1e-2).cpu().numpy())
        s["hyb"] = Hybrid(s["lat"], s["net"], HybridConfig(mode=0, use_fno=1, neq_mode=1, check_every=100, tol=1e-12,
                                                           max_steps=case["steps"]))
        return s
    s["fields"] = _fields(grids, case.get("scene"), gen)
    if kind == "unsteady":
        s["net"], s["net_u"] = (Fno(_shape(c), _params(c, gen, 1e-2).cpu().numpy()) for c in _pair(case))
        s["hyb"] = Hybrid(s["lat"], s["net"], HybridConfig(mode=1, k_lbm=case["k"], m_fno=case["m"], neq_mode=1,
                                                           in_channels=1, in_channels_u=6), fno_u=s["net_u"])
    if kind == "rollout":
        s["fields"] = [f.requires_grad_(True) for f in s["fields"]]
        s["douts"] = [torch.randn(f.numel(), generator=gen, device="cuda") for f in s["fields"]]
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fno":
        return s["net"](s["x"])
    if kind == "train":
        out = fno_apply(s["shape"], s["params"], s["x"])
        grads = torch.autograd.grad(out, [s["params"]] + ([s["x"]] if case["dx"] else []), s["dout"])
        return dict(out=out.detach(), dparams=grads[0], **(dict(dx=grads[1]) if case["dx"] else {}))
    lat = s["lat"]
    if kind == "rollout":
        out = lbm_rollout(lat, *s["fields"], case["steps"], every=case["every"])
        grads = torch.autograd.grad(out, s["fields"], s["douts"])
        return dict(fields=[o.detach() for o in out], grads=list(grads))
    if kind == "steady":
        st, first, res = s["hyb"].advance()
        # the residual is formed from 32-bit velocities
        return dict(fields=list(lat.macro()), residual=res.astype(np.float32), first=first, steps=int(st.steps))
    lat.reinit(*s["fields"])
    if kind == "couple":
        rho, ux, uy = lat.macro()
        return dict(fields=[rho, ux, uy], vorticity=lat.vorticity(ux, uy))
    if kind == "unsteady":
        s["hyb"].advance(cycles=case["cycles"])
        return dict(fields=list(lat.macro()))
    lat.step(case["steps"])
    stats = lat.residual()
    return dict(fields=list(lat.macro()), stats=stats)


# ------------------------------------------------------------------ work
def _net_work(c, B, H, W):
    Hp, Wp = H + c.get("pad", 0), W + c.get("pad", 0)
    C, h, m, S = c["width"], c["width"] // 2, c["modes"], c["dec_size"]
    layer = 2 * Hp * Wp * C * (2 * m) * 2 + 2 * Hp * m * C * (2 * m) * 4 * 2 + 8 * 2 * m * m * C * C + 2 * Hp * Wp * C * C
    lift = 2 * H * W * (h * (c["c_in"] + 2) + C * h)
    dec = 2 * H * W * (C * S + (c["dec_layers"] - 1) * S * S + S * c["c_out"])
    return B * (c["layers"] * layer + lift + dec), sum(int(np.prod(s)) for s, _, _ in _shapes(c))


def work(case):
    kind = case["kind"]
    if kind in ("fno", "train"):
        B, H, W = case["B"], case["H"], case["W"]
        flops, n = _net_work(case, B, H, W)
        io = 4 * B * H * W * (case["c_in"] + case["c_out"])
        if kind == "fno":
            return {"bytes": io + 2 * n, "flops": flops}
        return {"bytes": io + 4 * B * H * W * (case["c_out"] + case["c_in"] * case["dx"]) + 8 * n, "flops": 3 * flops}
    sizes = _sizes(case)
    cells = sum(nx * ny for nx, ny in sizes)
    step = 100 * cells
    if kind == "couple":
        return {"bytes": cells * (12 + 36 + 12 + 4), "flops": 250 * cells}
    if kind == "lbm":
        return {"bytes": cells * (12 + 36 + 12), "flops": (case["steps"] + 3) * step}
    if kind == "rollout":  # each step forward, and its reverse at about twice the work
        return {"bytes": cells * (12 + 12 + 12 + 12), "flops": (3 * case["steps"] + 6) * step}
    if kind == "steady":
        flops, n = _net_work(case, case["grids"], case["ny"], case["nx"])
        return {"bytes": cells * (36 + 12) + 2 * n, "flops": flops + case["steps"] * step}
    nets = [_net_work(c, case["grids"], case["ny"], case["nx"]) for c in _pair(case)]
    return {"bytes": cells * (12 + 36 + 12) + 2 * sum(n for _, n in nets),
            "flops": case["cycles"] * (case["k"] * step + case["m"] * sum(f for f, _ in nets))}


# ------------------------------------------------------------------ in 64 bits
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Lbm64:
    """D2Q9 BGK of equal grids [B, ny, nx] in 64 bits (populations are f - w, lists of nine fields)."""

    def __init__(self, grids, solid):
        col = lambda f: torch.tensor([float(f(g)) for g in grids], dtype=torch.float64, device="cuda")[:, None, None]
        self.g, self.nx, self.ny = grids[0], grids[0].nx, grids[0].ny
        self.solid = torch.from_numpy(np.stack(solid)).cuda()
        self.tau, self.fx, self.fy = col(lambda g: g.tau), col(lambda g: g.fx), col(lambda g: g.fy)
        self.west, self.east = col(lambda g: g.west_value)[..., 0], col(lambda g: g.east_value)[..., 0]
        self.open = grids[0].bc_west != BC_PERIODIC
        self.blocked = [torch.roll(self.solid, (CY[i], CX[i]), (1, 2)) for i in range(9)]
        if self.open:
            for i in range(9):
                if CX[i]:
                    self.blocked[i][:, :, 0 if CX[i] > 0 else -1] = False

    def ends(self, f):
        """Zou-He completion of the open end columns."""
        if not self.open:
            return f
        f = list(f)
        for at, bc, v, sg in ((0, self.g.bc_west, self.west, 1.0), (self.nx - 1, self.g.bc_east, self.east, -1.0)):
            c = [p[:, :, at] for p in f]
            known, unknown = ((3, 6, 7), (1, 8, 5)) if sg > 0 else ((1, 8, 5), (3, 6, 7))
            g0 = c[0] + c[2] + c[4] + 2 * sum(c[i] for i in known)
            ru = sg * ((v - 1) - g0) if bc == BC_PRESSURE else (1 + g0) / (1 - sg * v) * v
            t = 0.5 * (c[2] - c[4])
            for i in unknown:
                new = c[OPP[i]] + (2 / 3 if CY[i] == 0 else 1 / 6) * sg * ru - CY[i] * t
                hot = torch.zeros(self.nx, dtype=torch.bool, device="cuda")
                hot[at] = True
                f[i] = torch.where(hot, new[:, :, None], f[i])
        return f

    def pull(self, fs):
        return self.ends([torch.where(self.blocked[i], fs[OPP[i]], torch.roll(fs[i], (CY[i], CX[i]), (1, 2)))
                          for i in range(9)])

    def moments(self, f):
        d = sum(f)
        rho = 1 + d
        jx = sum(CX[i] * f[i] for i in range(9) if CX[i]) + 0.5 * self.fx
        jy = sum(CY[i] * f[i] for i in range(9) if CY[i]) + 0.5 * self.fy
        return d, rho, jx / rho, jy / rho

    def eq(self, i, d, rho, ux, uy):
        cu = CX[i] * ux + CY[i] * uy
        return WT[i] * (d + rho * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy)))

    def step(self, *f):
        d, rho, ux, uy = self.moments(f)
        om, guo = 1 / self.tau, 1 - 0.5 / self.tau
        out = []
        for i in range(9):
            cu, cf = CX[i] * ux + CY[i] * uy, CX[i] * self.fx + CY[i] * self.fy
            src = guo * WT[i] * (3 * (cf - ux * self.fx - uy * self.fy) + 9 * cu * cf)
            out.append(torch.where(self.solid, 0.0, f[i] + om * (self.eq(i, d, rho, ux, uy) - f[i]) + src))
        return tuple(self.pull(out))

    def deriv(self, v, ax):
        vp, vm = torch.roll(v, -1, ax), torch.roll(v, 1, ax)
        okp, okm = ~torch.roll(self.solid, -1, ax), ~torch.roll(self.solid, 1, ax)
        if ax == 2 and self.open:
            okp[:, :, -1] = False
            okm[:, :, 0] = False
        zero = torch.zeros_like(v)
        d = torch.where(okp & okm, 0.5 * (vp - vm), torch.where(okp, vp - v, torch.where(okm, v - vm, zero)))
        return torch.where(self.solid, zero, d)

    def reinit(self, rho, ux, uy):
        rho, ux, uy = (torch.where(self.solid, c, v) for c, v in ((1.0, rho), (0.0, ux), (0.0, uy)))
        gxx, gxy, gyx, gyy = (self.deriv(u, a) for a in (2, 1) for u in (ux, uy))
        out = []
        for i in range(9):
            q = (CX[i] ** 2 - 1 / 3) * gxx + CX[i] * CY[i] * (gxy + gyx) + (CY[i] ** 2 - 1 / 3) * gyy
            out.append(torch.where(self.solid, 0.0, self.eq(i, rho - 1, rho, ux, uy) - 3 * self.tau * WT[i] * rho * q))
        return tuple(self.ends(out))

    def macro(self, f):
        _, rho, ux, uy = self.moments(f)
        return [torch.where(self.solid, c, v) for c, v in ((1.0, rho), (0.0, ux), (0.0, uy))]

    def stats(self, f, ux0, uy0):
        d, rho, ux, uy = self.moments(f)
        fl = ~self.solid
        tot = lambda v: torch.where(fl, v, 0.0).sum((1, 2))
        u2 = tot(ux * ux + uy * uy)
        zero = torch.zeros_like(u2)
        dp = zero
        if self.open:
            mean = lambda at: torch.where(fl[:, :, at], d[:, :, at], 0.0).sum(1) / fl[:, :, at].sum(1)
            dp = (mean(0) - mean(-1)) / 3
        return torch.stack([torch.sqrt(tot((ux - ux0) ** 2 + (uy - uy0) ** 2) / u2), torch.sqrt(u2), dp, tot(rho),
                            tot(rho * ux), tot(rho * uy), zero, fl.sum((1, 2)).double()], 1)


def _groups(grids, solid):
    """(grid indices, offset of the first, _Lbm64) of each run of equal grids."""
    at, off = 0, 0
    while at < len(grids):
        n = at
        while n < len(grids) and (grids[n].nx, grids[n].ny) == (grids[at].nx, grids[at].ny):
            n += 1
        yield slice(off, off + (n - at) * grids[at].nx * grids[at].ny), _Lbm64(grids[at:n], solid[at:n])
        off += (n - at) * grids[at].nx * grids[at].ny
        at = n


def _fno64(c, params, x, bf16):
    """The FNO in 64 bits; bf16: parameters and inputs are rounded to bfloat16 first, as inference takes them."""
    act = F.gelu if c["act"] == "gelu" else F.relu
    B, _, H, W = x.shape
    if bf16:
        params, x = params.bfloat16(), x.float().bfloat16()
    params, x = params.double(), x.double()
    p, at = [], 0
    for shape, _, _ in _shapes(c):
        n = int(np.prod(shape))
        p.append(params[at:at + n].view(shape))
        at += n
    p = iter(p)
    one = lambda v: torch.einsum("oi,bihw->bohw", next(p), v) + next(p)[:, None, None]
    ar = lambda n: (torch.arange(n, device="cuda", dtype=torch.float32) / max(n - 1, 1)).bfloat16().double()
    co = torch.stack([ar(W)[None, :].expand(H, W), ar(H)[:, None].expand(H, W)]).expand(B, 2, H, W)
    v = one(act(one(torch.cat([x, co], 1))))
    pad, m = c.get("pad", 0), c["modes"]
    v = F.pad(v, (0, pad, 0, pad))
    Hp, Wp = H + pad, W + pad

    def dft(n, k):
        ph = torch.remainder(torch.outer(k, torch.arange(n, device="cuda")), n).double() * (2 * math.pi / n)
        return torch.complex(torch.cos(ph), -torch.sin(ph))

    ky = torch.cat([torch.arange(m, device="cuda"), torch.arange(Hp - m, Hp, device="cuda")])
    fy, fx = dft(Hp, ky), dft(Wp, torch.arange(m, device="cuda"))
    scale = torch.full((m, 1), 2.0 / (Hp * Wp), device="cuda", dtype=torch.float64)
    scale[0] = 1.0 / (Hp * Wp)
    gx = fx.conj() * scale
    for _ in range(c["layers"]):
        r1, r2 = torch.complex(next(p), next(p)), torch.complex(next(p), next(p))
        X = fy @ torch.complex(v @ fx.real.T, v @ fx.imag.T)  # kept ky x kept kx
        Y = torch.einsum("bikl,iokl->bokl", X, torch.cat([r1, r2], 2))
        Z = fy.conj().T @ Y
        v = act(one(v) + Z.real @ gx.real - Z.imag @ gx.imag)
    v = v[:, :, :H, :W]
    for _ in range(c["dec_layers"]):
        v = act(one(v))
    return one(v)


def _clamp(rho, ux, uy):
    sp = torch.sqrt(ux * ux + uy * uy).clamp_min(1e-30)
    sc = torch.clamp(0.2 / sp, max=1.0)
    return rho.clamp(0.9, 1.1), ux * sc, uy * sc


def exact(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "fno":
        params = _params(case, gen)
        return _fno64(case, params, _net_input(case, gen), True)
    if kind == "train":
        params = _params(case, gen).double().requires_grad_(True)
        x = _net_input(case, gen).double().requires_grad_(case["dx"])
        dout = torch.randn((case["B"], case["c_out"], case["H"], case["W"]), generator=gen, device="cuda")
        total, gx, outs = torch.zeros_like(params), [], []
        for b in range(case["B"]):  # an item at a time: the 64-bit graph of a batch is large
            xb = x[b:b + 1].detach().requires_grad_(case["dx"])
            y = _fno64(case, params, xb, False)
            g = torch.autograd.grad(y, [params] + ([xb] if case["dx"] else []), dout[b:b + 1].double())
            total += g[0]
            outs.append(y.detach())
            gx += list(g[1:])
        return dict(out=torch.cat(outs), dparams=total, **(dict(dx=torch.cat(gx)) if case["dx"] else {}))
    if kind == "unsteady":
        case = dict(case, scene="shear")
    grids, solid = _batch(case, seed)
    if kind == "steady":
        params, B = _params(case, gen, 1e-2), case["grids"]
        L = _Lbm64(grids, solid)
        x = torch.zeros((B, 4, L.ny, L.nx), device="cuda")
        x[:, 3] = L.solid.float()
        y = _fno64(case, params, x, True)
        rho, ux, uy = _clamp(1 + y[:, 0], y[:, 1], y[:, 2])
        f = L.reinit(rho, ux, uy)
        for k in range(case["steps"]):
            if k and k % 100 == 0:
                _, ux, uy = L.macro(f)
            f = L.step(*f)
        return dict(fields=[v.reshape(-1) for v in L.macro(f)], residual=L.stats(f, ux, uy)[:, 0], first=None, steps=None)
    fields = [f.double() for f in _fields(grids, case.get("scene"), gen)]
    if kind == "unsteady":
        a, b = _pair(case)
        pa, pb = _params(a, gen, 1e-2), _params(b, gen, 1e-2)
        L = _Lbm64(grids, solid)
        f = L.reinit(*(v.view(-1, L.ny, L.nx) for v in fields))
        for _ in range(case["cycles"]):
            for _ in range(case["k"]):
                f = L.step(*f)
            rho, ux, uy = L.macro(f)
            for _ in range(case["m"]):
                r, u = _fno64(a, pa, (rho - 1)[:, None], True), _fno64(b, pb, torch.stack([ux, uy], 1), True)
                rho, ux, uy = _clamp(1 + r[:, 0], u[:, 0], u[:, 1])
            f = L.reinit(rho, ux, uy)
        return dict(fields=[v.reshape(-1) for v in L.macro(f)])
    if kind == "rollout":
        douts = [torch.randn(f.numel(), generator=gen, device="cuda") for f in fields]
        L = _Lbm64(grids, solid)
        fields = [f.view(-1, L.ny, L.nx).requires_grad_(True) for f in fields]
        f = L.reinit(*fields)
        for _ in range(case["steps"]):
            f = checkpoint(L.step, *f, use_reentrant=False)
        out = L.macro(f)
        grads = torch.autograd.grad(out, fields, [g.view(-1, L.ny, L.nx).double() for g in douts])
        return dict(fields=[o.detach().reshape(-1) for o in out], grads=[g.reshape(-1) for g in grads])
    parts = []
    for at, L in _groups(grids, solid):
        rho, ux, uy = (v[at].view(-1, L.ny, L.nx) for v in fields)
        f = L.reinit(rho, ux, uy)
        for _ in range(case["steps"]):
            f = L.step(*f)
        m = L.macro(f)
        last = L.deriv(m[2], 2) - L.deriv(m[1], 1) if kind == "couple" else L.stats(
            f, torch.where(L.solid, 0.0, ux), torch.where(L.solid, 0.0, uy))
        parts.append([v.reshape(-1) for v in m] + [last.reshape(-1) if kind == "couple" else last])
    cols = [torch.cat(v) for v in zip(*parts)]
    return dict(fields=cols[:3], **{"vorticity" if kind == "couple" else "stats": cols[3]})
