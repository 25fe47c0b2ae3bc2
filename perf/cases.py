"""Performance cases: the work that a user of this library has it do, through its public entry
points, from the smallest calls to the largest.

Five kinds of case:
  lattice  time steps of one lattice, then the density (FP64 lattices: the velocity too)
  batch    a sweep of independent lattices of uneven size advanced together
  measure  both contact angles, then mass and liquid centroid, of a density field
  forward  the warm-start network's prediction
  train    one training step of the warm-start network (loss and every gradient)

FP32 lattices hold their fields in FP32; the library hands fields out widened to FP64, and the
cases hand them on as FP32. `exact` computes the same results in 64 bits with plain torch / numpy.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2202_06516_gb300 import lbm

# Model of the workloads (Peng-Robinson) and its Carnahan-Starling variant, both at Tr = 0.7, with
# the coexistence densities handed to the library as a user with tabulated values does.
PR = dict(eos=0, Tr=0.7, k2=0.05, kappa=0.0063, tau=1.0, s_e=1.64, s_eps=1.54, s_q=1.9,
          rho_g=0.05563509, rho_l=8.08032155)
CS = dict(eos=1, Tr=0.7, k2=0.05, kappa=0.05, tau=1.0, s_e=1.64, s_eps=1.54, s_q=1.9,
          rho_g=0.00929172, rho_l=0.35814440)
MU_PER_DEGREE = 1.5e-3  # wall potential per degree of target angle


def _lattice(name, nx, ny, R, r, steps, **kw):
    c = dict(kind="lattice", nx=nx, ny=ny, R=R, r=r, steps=steps, cy=0.0, fp64=False, cs=False,
             bgk=False, interp=False, concave=False, stripes=False, gx=0.0, gy=0.0, buoyant=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain method's small workload: one drop on a cylinder, 100 steps between readings
        _lattice("step_200x120", 200, 120, 40.0, 25.0, 100),
        # a drop in a cavity of the curvature sweep, with interpolated bounce-back on its wall
        _lattice("step_cavity_520x190", 520, 190, 250.0, 50.0, 100, concave=True, interp=True),
        # the plain method at scale: sessile drop under a constant body force
        _lattice("step_2048x1024", 2048, 1024, 300.0, 150.0, 50, gy=-1e-6),
        # dynamic hysteresis: striped cylinder, tilted buoyant body force, 100 steps per reading
        _lattice("step_striped_4096x1024", 4096, 1024, 800.0, 120.0, 100, cy=-100.0, stripes=True,
                 gx=5e-7, gy=-1.3737387e-6, buoyant=True),
        # the small workload in FP64 with the other equation of state (accuracy studies)
        _lattice("step_fp64_200x120", 200, 120, 40.0, 25.0, 50, fp64=True, cs=True),
        # a parameter sweep of uneven lattices, residual checked every 40 steps
        dict(name="batch_64", kind="batch", n=64, nx_min=128, nx_max=768, ny_min=128, ny_max=512,
             steps=80, check=40),
        # one on-the-spot measurement on the smallest and on the largest workload
        dict(name="measure_200x120", kind="measure", nx=200, ny=120, R=40.0, r=25.0, cy=0.0,
             flat=False, concave=False),
        dict(name="measure_4096x1024", kind="measure", nx=4096, ny=1024, R=800.0, r=120.0,
             cy=-100.0, flat=False, concave=False),
        # the prediction for a single case (latency) and for a batch of held-out cases
        dict(name="forward_256_b1", kind="forward", H=256, W=256, base=32, B=1),
        dict(name="forward_256_b8", kind="forward", H=256, W=256, base=32, B=8),
        # training steps: the small network, and the full one at its training batch
        dict(name="train_128_base16_b8", kind="train", H=128, W=128, base=16, B=8),
        dict(name="train_256_b8", kind="train", H=256, W=256, base=32, B=8),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "batch", "measure", "forward", "train"])
    if kind in ("lattice", "measure"):
        fp64 = kind == "lattice" and rng.random() < 0.2
        nx = _logint(rng, 128, 400 if fp64 else 4096)
        ny = _logint(rng, 96, 240 if fp64 else 1024)
        concave = rng.random() < 0.25
        if concave:
            # the cavity spans the width; the drop sits at its bottom
            R = max(48, min(nx // 2 - 10, 3 * ny))
            r = rng.uniform(0.12, 0.25) * min(R, ny)
        else:
            R = max(20, int(rng.uniform(0.3, 0.6) * min(nx / 2.0, ny)))
            r = rng.uniform(0.5, 0.9) * min((ny - R) / 2.0, R, 150.0)
        R, r = float(R), float(max(12.0, round(r, 1)))
        if kind == "measure":
            return dict(kind="measure", nx=nx, ny=ny, R=R, r=r, cy=0.0,
                        flat=not concave and rng.random() < 0.2, concave=concave)
        steps = max(20, min(200, int(4.0e8 / (nx * ny * (8 if fp64 else 1)))))
        steps = rng.randint(max(10, steps // 2), steps)
        return _lattice(None, nx, ny, R, r, steps, fp64=fp64, cs=rng.random() < 0.25,
                        bgk=rng.random() < 0.25, concave=concave,
                        interp=not fp64 and rng.random() < 0.2,
                        stripes=not concave and rng.random() < 0.25,
                        gy=rng.choice([0.0, 1e-6, -1e-6]), buoyant=rng.random() < 0.3)
    if kind == "batch":
        lo = rng.choice([96, 128])
        return dict(kind="batch", n=rng.randint(3, 60), nx_min=lo, nx_max=_logint(rng, 160, 768),
                    ny_min=lo, ny_max=_logint(rng, 140, 512), steps=2 * rng.randint(10, 50),
                    check=2 * rng.randint(5, 20))
    H, W = 8 * _logint(rng, 8, 32), 8 * _logint(rng, 8, 32)
    if rng.random() < 0.5:  # powers of two: the sizes the network is trained at
        H, W = 2 ** int(math.log2(H)), 2 ** int(math.log2(W))
    return dict(kind=kind, H=H, W=W, base=rng.choice([8, 16, 32]), B=rng.randint(1, 8))


# --------------------------------------------------------------------------------- preparation
def _rng(seed, salt):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, salt])


def _drop(c, cx, r, theta0, W):
    """Drop centre: on top of the cylinder (cy, R) or at the bottom of the cavity, meeting the wall
    surface R + 1/2 at theta0 (law of cosines); small drops start tangent to a cylinder."""
    Rs, t = c["R"] + 0.5, math.radians(theta0)
    if c["concave"]:
        return (cx, c["R"] + 6.0 - math.sqrt(Rs * Rs + r * r + 2 * Rs * r * math.cos(t)), r, W)
    if r < 60 and theta0 == 90.0:
        return (cx, c["cy"] + Rs + r, r, W)
    return (cx, c["cy"] + math.sqrt(Rs * Rs + r * r - 2 * Rs * r * math.cos(t)), r, W)


def _setup(c, seed):
    """Model, circle, wall potentials and drop of a lattice case: the wetting and the drop's size
    come from the seed."""
    g = _rng(seed, 1)
    m = dict(CS if c["cs"] else PR)
    neutral = m["k2"] * float(_psi_prime(m, torch.tensor(m["rho_l"], dtype=torch.float64)))
    theta = g.uniform(70.0, 115.0)
    r = c["r"] * g.uniform(0.92, 1.0)
    cx = c["nx"] // 2
    cyc = c["R"] + 6.0 if c["concave"] else c["cy"]
    drop = _drop(c, float(cx), r, theta if c["concave"] else 90.0, 4.0 if c["cs"] else 5.6)
    scale = 0.3 if c["cs"] else 1.0  # the CS potentials are smaller
    walls = dict(circle=(float(cx), cyc, c["R"]), mu_circle=neutral + scale * MU_PER_DEGREE * (theta - 90.0),
                 mu_bottom=neutral, mu_top=neutral, concave=c["concave"])
    if c["stripes"]:
        walls["stripes"] = (40.0, neutral - scale * 0.03)
    return m, walls, drop


def _batch_sizes(c, seed):
    """Instances of a sweep: domains and cylinders drawn once in the case's ranges, wetting and drop
    sizes from the seed."""
    g, gs = _rng(c["n"], 2), _rng(seed, 5)
    out = []
    for _ in range(c["n"]):
        nx = int(g.integers(c["nx_min"], c["nx_max"] + 1))
        ny = int(g.integers(c["ny_min"], c["ny_max"] + 1))
        R = float(g.integers(20, max(21, min(200, (nx - 16) // 2, ny // 2)) + 1))
        r = float(g.uniform(12.0, max(12.5, min(90.0, (ny - R - 8) / 2.0))))
        one = dict(nx=nx, ny=ny, R=R, r=r, cy=0.0, cs=False, concave=False, stripes=False)
        out.append((one, _setup(one, int(gs.integers(1 << 30)))))
    return out


def _field(c, seed):
    """Density of an equilibrated-looking drop (Eq. 16 profile, thermal-like ripple of 1e-3) on the
    case's substrate, FP32-representable, as host doubles."""
    g = _rng(seed, 3)
    theta = g.uniform(60.0, 120.0)
    r = c["r"] * g.uniform(0.92, 1.0)
    cx = float(c["nx"] // 2) + g.uniform(-2.0, 2.0)
    if c["flat"]:
        x0, y0 = cx, -0.5 - r * math.cos(math.radians(theta))
    else:
        x0, y0 = _drop(c, cx, r, theta, 5.6)[:2]
    jj, ii = np.mgrid[0:c["ny"], 0:c["nx"]].astype(np.float64)
    d = np.hypot(ii - x0, jj - y0)
    rho = 0.5 * (PR["rho_g"] + PR["rho_l"]) + 0.5 * (PR["rho_g"] - PR["rho_l"]) * np.tanh(2.0 * (d - r) / 5.6)
    rho *= 1.0 + 1e-3 * np.sin(0.37 * ii + g.uniform(0, 6)) * np.cos(0.23 * jj)
    return rho.astype(np.float32).astype(np.float64)


def _circle(c):
    return None if c["flat"] else (float(c["nx"] // 2), c["R"] + 6.0 if c["concave"] else c["cy"], c["R"])


_LAYERS = lambda b: [(8, b), (b, b), (b, 2 * b), (2 * b, 2 * b), (2 * b, 4 * b), (4 * b, 4 * b),
                     (4 * b, 8 * b), (8 * b, 8 * b), (8 * b, 4 * b), (8 * b, 4 * b), (4 * b, 4 * b),
                     (4 * b, 2 * b), (4 * b, 2 * b), (2 * b, 2 * b), (2 * b, b), (2 * b, b), (b, b)]


def _net(c, seed):
    """Network weights (He-normal convolutions, small biases, a head that spreads phi over (0, 1))
    and a batch: the geometry planes of drops on cylinders, targets and the fluid mask."""
    g = _rng(seed, 4)
    w = []
    for ci, co in _LAYERS(c["base"]):
        w.append(g.normal(0.0, math.sqrt(2.0 / (9 * ci)), size=co * 9 * ci))
        w.append(g.normal(0.0, 0.02, size=co))
    w.append(g.normal(0.0, 0.3 / math.sqrt(c["base"]), size=c["base"]))
    w.append(g.normal(0.0, 0.1, size=1))
    w = np.concatenate(w).astype(np.float32)
    H, W, B = c["H"], c["W"], c["B"]
    y = torch.arange(H, dtype=torch.float32, device="cuda").view(H, 1).expand(H, W)
    x = torch.arange(W, dtype=torch.float32, device="cuda").view(1, W).expand(H, W)
    X = torch.zeros(B, H, W, 8, device="cuda")
    T = torch.zeros(B, H, W, device="cuda")
    for b in range(B):
        R = g.uniform(0.15, 0.4) * min(H, W)
        r = g.uniform(0.15, 0.25) * min(H, W)
        mu = MU_PER_DEGREE * g.uniform(-60.0, 60.0)
        dist = torch.minimum(torch.hypot(x - W / 2, y) - (R + 0.5), y + 0.5)
        fluid = (dist > 0).float()
        phi = 0.5 - 0.5 * torch.tanh(2.0 * (torch.hypot(x - W / 2, y - (R + 0.7 * r)) - r) / 8.5)
        X[b, :, :, 0] = 1.0 - fluid
        X[b, :, :, 1] = (1.0 - fluid) * (dist > -2.0) * (mu / 0.1)
        X[b, :, :, 2] = (phi * fluid).sum() / (H * W)
        X[b, :, :, 3] = y / H
        X[b, :, :, 4] = (x - W / 2) / W
        X[b, :, :, 5] = (dist / 64.0).clamp(-1.0, 1.0)
        X[b, :, :, 6] = mu / 0.1
        T[b] = phi * fluid
    return w, X.to(torch.bfloat16), T, (X[..., 0] == 0).to(torch.uint8)


def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "lattice":
        m, walls, drop = _setup(c, seed)
        stream = torch.cuda.Stream()
        lat = lbm.Lattice(c["nx"], c["ny"], **m, gx=c["gx"], gy=c["gy"],
                          g_rho_ref=m["rho_g"] if c["buoyant"] else 0.0,
                          precision=lbm.LBM_FP64 if c["fp64"] else lbm.LBM_FP32,
                          collision=lbm.LBM_BGK if c["bgk"] else lbm.LBM_MRT, stream=stream)
        lat.set_geometry(**walls, drop=drop,
                         boundary=lbm.LBM_BB_INTERP if c["interp"] else lbm.LBM_BB_HALFWAY)
        return dict(c, lat=lat, stream=stream)
    if kind == "batch":
        inst = _batch_sizes(c, seed)
        b = lbm.Batch([(o["nx"], o["ny"]) for o, _ in inst], **PR)
        for i, (_, (_, walls, drop)) in enumerate(inst):
            b.set_geometry(i, **walls, drop=drop)
        n = sum(o["nx"] * o["ny"] for o, _ in inst)
        return dict(c, b=b, sizes=[(o["nx"], o["ny"]) for o, _ in inst],
                    out=torch.empty(n, dtype=torch.float64, device="cuda"))
    if kind == "measure":
        lat = lbm.Lattice(c["nx"], c["ny"], **PR)
        lat.set_geometry(circle=_circle(c), concave=c["concave"], rho0=_field(c, seed))
        return dict(c, lat=lat)
    w, x, t, mask = _net(c, seed)
    sur = lbm.Surrogate(c["H"], c["W"], base=c["base"], max_batch=c["B"])
    sur.set_weights(w)
    return dict(c, sur=sur, x=x, t=t, mask=mask)


# ---------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "lattice":
        lat, nx, ny = s["lat"], s["nx"], s["ny"]
        lat.step(s["steps"])
        with torch.cuda.stream(s["stream"]):
            n = 3 if s["fp64"] else 1
            out = torch.empty(n, ny, nx, dtype=torch.float64, device="cuda")
            which = lbm.LBM_FIELD_RHO | (lbm.LBM_FIELD_VEL if s["fp64"] else 0)
            ptr = [out[k].data_ptr() if k < n else None for k in range(3)]
            lbm.lbm_read_fields(lat.ctx, which, nx, ny, device_out=ptr)
            return (out[0], out[1], out[2]) if s["fp64"] else out[0].float()
    if kind == "batch":
        b = s["b"]
        steps, conv, _ = b.run(s["steps"], check_every=s["check"], tol=1e-6)
        torch.cuda.current_stream().synchronize()  # the last pass may still read `out`
        o = 0
        for i, (nx, ny) in enumerate(s["sizes"]):
            lbm.lbm_read_fields(lbm.lbm_batch_instance(b.b, i), lbm.LBM_FIELD_RHO, nx, ny,
                                device_out=(s["out"][o:].data_ptr(), None, None))
            o += nx * ny
        return s["out"].float(), steps, conv
    if kind == "measure":
        angles = s["lat"].measure()
        return [_angle_out(a) for a in angles], _mass_out(s["lat"].mass())
    if kind == "forward":
        phi = torch.empty(s["B"], s["H"], s["W"], dtype=torch.float32, device="cuda")
        s["sur"].forward(s["x"].data_ptr(), s["B"], phi.data_ptr())
        return phi
    # the learning rate of the first warm-up step
    loss = s["sur"].train_step(s["x"].data_ptr(), s["t"].data_ptr(), s["mask"].data_ptr(), s["B"], 1.5e-6)
    return np.float32(loss), s["sur"].weights(grads=True)


def _angle_out(a):
    return (np.array([a.theta, a.alpha, a.beta, *a.contact, *a.p1, *a.p2, a.d1, a.d2]),
            np.array([a.status, a.link1, a.link2], dtype=np.int64))


def _mass_out(m):
    return m["mass"], int(m["n_liquid"]), m["cx"], m["cy"]


# ----------------------------------------------------------------------------- necessary work
def _fluid_share(c):
    if c.get("flat"):
        return 1.0
    i, j = np.meshgrid(np.arange(c["nx"]) - c["nx"] // 2, np.arange(c["ny"]))
    d = np.hypot(i, j - (c["R"] + 6.0 if c["concave"] else c["cy"]))
    return float(np.mean((d <= c["R"]) == c["concave"]))


def work(case):
    c, kind = case, case["kind"]
    if kind in ("lattice", "batch"):
        # per step and fluid node: nine populations and the density read and written once (80 bytes
        # in FP32), and about 300 operations (pressure, stencils, moments, streaming)
        if kind == "lattice":
            n = c["nx"] * c["ny"]
            f, e = n * _fluid_share(c), 8 if c["fp64"] else 4
            return {"bytes": c["steps"] * f * 20 * e + n * e, "flops": c["steps"] * f * 300}
        n = c["n"] * 0.25 * (c["nx_min"] + c["nx_max"]) * (c["ny_min"] + c["ny_max"])
        return {"bytes": c["steps"] * 0.9 * n * 80 + n * 4, "flops": c["steps"] * 0.9 * n * 300}
    if kind == "measure":
        # density and node class of every node once
        return {"bytes": c["nx"] * c["ny"] * 5, "flops": c["nx"] * c["ny"] * 4}
    px, b = c["B"] * c["H"] * c["W"], c["base"]
    area = [1, 1, 1 / 4, 1 / 4, 1 / 16, 1 / 16, 1 / 64, 1 / 64, 1 / 16, 1 / 16, 1 / 16, 1 / 4, 1 / 4,
            1 / 4, 1, 1, 1]
    flops = sum(2 * 9 * ci * co * px * a for (ci, co), a in zip(_LAYERS(b), area))
    nw = sum(9 * ci * co + co for ci, co in _LAYERS(b)) + b + 1
    if kind == "forward":
        return {"bytes": px * 20 + nw * 2, "flops": flops}
    # inputs, target, mask and every stored activation written and read once; the weights with
    # their gradient and both moments read and written
    act = sum(co * px * a for (_, co), a in zip(_LAYERS(b), area)) * 2
    return {"bytes": px * 21 + 2 * act + nw * 28, "flops": 3 * flops}


# ----------------------------------------------------------------- the same results in 64 bits
QX, QY = [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
WQ = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _psi_prime(m, rho):
    """Bulk chemical potential at k = 1 (Peng-Robinson or Carnahan-Starling)."""
    if m["eos"] == 0:
        a, b, om = 2 / 49, 2 / 21, 0.344
        T = m["Tr"] * 0.0778 * a / (0.45724 * b)
        al = (1 + (0.37464 + 1.54226 * om - 0.26992 * om * om) * (1 - math.sqrt(m["Tr"]))) ** 2
        s2, br = math.sqrt(2.0), b * rho
        return (T * torch.log(rho / (1 - br)) - a * al / (2 * s2 * b) * torch.log((s2 - 1 + br) / (s2 + 1 - br))
                + T / (1 - br) - a * al * rho / (1 + 2 * br - br * br))
    a, b = 1.0, 4.0
    T, n = m["Tr"] * 0.3773 * a / b, b * rho / 4
    return T * (torch.log(rho) + (8 * n - 9 * n ** 2 + 3 * n ** 3) / (1 - n) ** 3) - 2 * a * rho


def _shift(t, dx, dy):
    """t at (x + dx, y + dy): periodic in x; rows that leave the array wrap (callers mask them)."""
    return torch.roll(t, shifts=(-dy, -dx), dims=(-2, -1))


def _solid(nx, ny, circle, concave):
    """Solid nodes of the rows -4 .. ny + 3 (wall rows, the disc or the outside of the cavity)."""
    j, i = torch.meshgrid(torch.arange(-4, ny + 4, device="cuda", dtype=torch.float64),
                          torch.arange(nx, device="cuda", dtype=torch.float64), indexing="ij")
    wall = (j < 0) | (j >= ny)
    disc = torch.zeros_like(wall)
    if circle is not None:
        d2 = (i - circle[0]) ** 2 + (j - circle[1]) ** 2
        disc = (d2 <= circle[2] ** 2) ^ bool(concave)
    return i, j, wall | disc, disc


class _Exact:
    """The method's time step in FP64 torch: f holds the populations after streaming."""

    def __init__(self, nx, ny, m, walls, drop, bgk=False, interp=False, gx=0.0, gy=0.0, ref=0.0):
        self.m, self.bgk, self.interp, self.g, self.ref = m, bgk, interp, (gx, gy), ref
        i, j, solid, disc = _solid(nx, ny, walls["circle"], walls["concave"])
        near = lambda t: sum(_shift(t, QX[q], QY[q]).int() for q in range(1, 9)) > 0
        self.fluid = ~solid
        inner = (j >= -2) & (j < ny + 2)
        self.l1 = solid & near(self.fluid) & inner
        self.l2 = solid & ~self.l1 & near(self.l1) & inner
        cx, cy, R = walls["circle"]
        full = lambda v: torch.full_like(j, v)
        mu = torch.where(j < 0, full(walls["mu_bottom"]), full(walls["mu_top"]))
        on = full(walls["mu_circle"])
        if walls.get("stripes"):
            k = torch.floor(R * (torch.atan2(j - cy, i - cx) - 0.5 * math.pi) / walls["stripes"][0])
            on = torch.where(k % 2 == 0, on, full(walls["stripes"][1]))
        self.muw = torch.where(disc, on, mu) * (self.l1 | self.l2)
        d = torch.hypot(i - drop[0], j - drop[1])
        rho = 0.5 * (m["rho_g"] + m["rho_l"]) + 0.5 * (m["rho_g"] - m["rho_l"]) * torch.tanh(2 * (d - drop[2]) / drop[3])
        self.rho = rho * self.fluid
        self.f = torch.stack([w * self.rho for w in WQ])
        # per direction: the source is fluid; the sums of neighbour weights of the layers
        self.src = [_shift(self.fluid, -QX[q], -QY[q]) for q in range(9)]
        self.den1 = sum(WQ[q] * _shift(self.fluid.double(), QX[q], QY[q]) for q in range(1, 9)).clamp(min=1e-300)
        self.den2 = sum(WQ[q] * _shift(self.l1.double(), QX[q], QY[q]) for q in range(1, 9)).clamp(min=1e-300)
        M = torch.tensor([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
                          [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
                          [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
                          [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=torch.float64)
        S = torch.diag(torch.tensor([0, m["s_e"], m["s_eps"], 0, m["s_q"], 0, m["s_q"], 1 / m["tau"], 1 / m["tau"]],
                                    dtype=torch.float64))
        A = torch.linalg.inv(M) @ S @ M
        self.A = torch.eye(9, dtype=torch.float64).cuda() / m["tau"] if bgk else A.cuda()
        self.frac = self._fractions(i, j, ny, walls) if interp else None

    def _fractions(self, i, j, ny, walls):
        """Per direction: the share of the link toward the solid source at which the wall surface
        (the circle R + 1/2, the planes y = -1/2 and ny - 1/2) is met; 1/2 without a crossing."""
        cx, cy, R = walls["circle"]
        out = [None]
        for q in range(1, 9):
            vx, vy = QX[OPP[q]], QY[OPP[q]]
            best = torch.full_like(i, 2.0)
            if vy:
                s = (j + 0.5) / -vy if vy < 0 else (ny - 0.5 - j) / vy
                best = torch.where((s >= 0) & (s <= 1), torch.minimum(s, best), best)
            a, b = float(vx * vx + vy * vy), (i - cx) * vx + (j - cy) * vy
            disc = b * b - a * ((i - cx) ** 2 + (j - cy) ** 2 - (R + 0.5) ** 2)
            sq = torch.sqrt(disc.clamp(min=0))
            s = ((sq - b) if walls["concave"] else (-b - sq)) / a
            hit = (disc >= 0) & (s > -1e-12) & (s <= 1)
            best = torch.where(hit, torch.minimum(s.clamp(min=0), best), best)
            out.append(torch.where(best <= 1, best, torch.full_like(best, 0.5)).clamp(min=0.1))
        return out

    def forces(self):
        m, fl = self.m, self.fluid
        rho = self.rho
        num = sum(WQ[q] * _shift(rho * fl, QX[q], QY[q]) for q in range(1, 9))
        rho = torch.where(self.l1, num / self.den1, rho)
        num = sum(WQ[q] * _shift(rho * self.l1, QX[q], QY[q]) for q in range(1, 9))
        rho = torch.where(self.l2, num / self.den2, rho)
        lap = (16 * (_shift(rho, 1, 0) + _shift(rho, -1, 0) + _shift(rho, 0, 1) + _shift(rho, 0, -1)) - 60 * rho
               - (_shift(rho, 2, 0) + _shift(rho, -2, 0) + _shift(rho, 0, 2) + _shift(rho, 0, -2))) / 12
        safe = torch.where(fl, self.rho, torch.full_like(rho, m["rho_g"]))
        mu = torch.where(fl, m["k2"] * _psi_prime(m, safe) - m["kappa"] * lap, self.muw)
        grad = lambda t, x, y: (8 * (_shift(t, x, y) - _shift(t, -x, -y)) - _shift(t, 2 * x, 2 * y) + _shift(t, -2 * x, -2 * y)) / 12
        F = []
        for k, (x, y) in enumerate(((1, 0), (0, 1))):
            F.append(-safe * grad(mu, x, y) + grad(rho, x, y) / 3 + (safe - self.ref) * self.g[k])
        return safe, F[0], F[1]

    def macro(self):
        rho, Fx, Fy = self.forces()
        jx = sum(QX[q] * self.f[q] for q in range(9))
        jy = sum(QY[q] * self.f[q] for q in range(9))
        return rho, Fx, Fy, jx / rho, jy / rho

    def step(self):
        rho, Fx, Fy, ux, uy = self.macro()

        def eq(vx, vy):
            vv = vx * vx + vy * vy
            return torch.stack([WQ[q] * rho * (1 + 3 * (QX[q] * vx + QY[q] * vy) + 4.5 * (QX[q] * vx + QY[q] * vy) ** 2
                                               - 1.5 * vv) for q in range(9)])

        fe = eq(ux, uy)
        post = self.f - torch.einsum("ab,byx->ayx", self.A, self.f - fe) + eq(ux + Fx / rho, uy + Fy / rho) - fe
        post = post * self.fluid
        new, extra = [post[0]], torch.zeros_like(rho)
        for q in range(1, 9):
            back = post[OPP[q]]
            if self.interp:
                D = self.frac[q]
                behind, ok = _shift(post[OPP[q]], QX[q], QY[q]), _shift(self.fluid, QX[q], QY[q])
                lo = torch.where(ok, 2 * D * back + (1 - 2 * D) * behind, back)
                hi = back / (2 * D) + (1 - 1 / (2 * D)) * post[q]
                cut = torch.where(D < 0.5, lo, hi)
                extra = extra + torch.where(self.src[q], torch.zeros_like(rho), back - cut)
                back = cut
            new.append(torch.where(self.src[q], _shift(post[q], -QX[q], -QY[q]), back))
        new[0] = new[0] + extra
        self.f = torch.stack(new) * self.fluid
        self.rho = self.f.sum(0)


def _exact_lattice(c, seed):
    m, walls, drop = _setup(c, seed)
    e = _Exact(c["nx"], c["ny"], m, walls, drop, c["bgk"], c["interp"], c["gx"], c["gy"],
               m["rho_g"] if c["buoyant"] else 0.0)
    for _ in range(c["steps"]):
        e.step()
    if not c["fp64"]:
        return e.rho[4:-4]
    rho, Fx, Fy, ux, uy = e.macro()
    return e.rho[4:-4], *(((u + f / (2 * rho)) * e.fluid)[4:-4] for u, f in ((ux, Fx), (uy, Fy)))


def _exact_measure(c, seed):
    """Both contact angles and the sums, from the field's liquid/gas links near the wall."""
    rho, nx, ny = _field(c, seed), c["nx"], c["ny"]
    circ = _circle(c)
    solid = _solid(nx, ny, circ, c["concave"])[2][4:-4].cpu().numpy()
    rm = 0.5 * (PR["rho_g"] + PR["rho_l"])
    liq = (rho > rm) & ~solid
    jj, ii = np.nonzero(liq)
    qx, qy = ii.mean(), jj.mean()
    Rs = circ[2] + 0.5 if circ else 0.0
    best = [[None, None], [None, None]]
    for sl, (ex, ey) in enumerate(((1, 0), (0, 1), (1, 1), (-1, 1))):
        j, i = np.mgrid[0:ny - ey, 0:nx]
        ti = (i + ex) % nx
        a, b = rho[j, i], rho[j + ey, ti]
        ok = ~solid[j, i] & ~solid[j + ey, ti] & ((a > rm) != (b > rm))
        j, i, a, b = j[ok], i[ok], a[ok], b[ok]
        la = a > rm
        gx, gy = np.where(la, i + ex, i), np.where(la, j + ey, j)
        fr = (rm - np.where(la, b, a)) / (np.where(la, a, b) - np.where(la, b, a))
        s = np.where(la, -1.0, 1.0)
        px, py = gx + fr * s * ex, gy + fr * s * ey
        if circ:
            d = (np.hypot(px - circ[0], py - circ[1]) - Rs) * (-1 if c["concave"] else 1)
            cr = (qx - circ[0]) * (py - circ[1]) - (qy - circ[1]) * (px - circ[0])
            side = np.where((cr < 0) if c["concave"] else (cr > 0), 0, 1)
        else:
            d, side = py + 0.5, np.where(px < qx, 0, 1)
        for k in np.nonzero((d >= 0.5) & (d <= 2.5))[0]:
            ident = (int(j[k]) * nx + int(i[k])) * 4 + sl
            for t in (0, 1):
                key = (abs(d[k] - (t + 1)), ident, px[k], py[k], d[k])
                if best[side[k]][t] is None or key < best[side[k]][t]:
                    best[side[k]][t] = key
    out = []
    for side in (0, 1):
        b1, b2 = best[side]
        if b1 is None or b2 is None or b1[1] == b2[1]:
            return None
        v = np.array([b2[2] - b1[2], b2[3] - b1[3]])
        v /= np.hypot(*v)
        p = np.array([b1[2], b1[3]])
        if circ:
            w = p - np.array(circ[:2])
            disc = (w @ v) ** 2 - (w @ w - Rs * Rs)
            if disc < 0:
                return None
            s = min(-(w @ v) - math.sqrt(disc), -(w @ v) + math.sqrt(disc), key=abs)
            C = p + s * v
            n = (C - np.array(circ[:2])) / np.hypot(*(C - np.array(circ[:2]))) * (-1 if c["concave"] else 1)
            t = np.array([n[1], -n[0]]) * (1 if side == 0 else -1)
        else:
            C = p + (-0.5 - p[1]) / v[1] * v
            t = np.array([1.0 if side == 0 else -1.0, 0.0])
        theta = math.degrees(math.acos(max(-1.0, min(1.0, t @ v))))
        alpha = math.degrees(math.acos(min(1.0, abs(t[0]))))
        beta = theta if not circ else theta + (-alpha if c["concave"] else alpha)
        out.append((np.array([theta, alpha, beta, *C, b1[2], b1[3], b2[2], b2[3], b1[4], b2[4]]), None))
    return out, (float(rho[~solid].sum()), None, float(qx), float(qy))


def _exact_net(c, seed):
    w, x, t, mask = _net(c, seed)
    p = torch.tensor(w, dtype=torch.float64, device="cuda", requires_grad=c["kind"] == "train")
    layers, o = [], 0
    for ci, co in _LAYERS(c["base"]):
        layers.append((p[o:o + co * 9 * ci].reshape(co, 3, 3, ci).permute(0, 3, 1, 2), p[o + co * 9 * ci:o + co * 9 * ci + co]))
        o += co * 9 * ci + co

    def conv(h, k):
        """3 x 3, padding 1, as nine matrix products over the channels (NCHW)."""
        wk, b = layers[k]
        B, C, H, W = h.shape
        hp, z = F.pad(h, (1, 1, 1, 1)), b.view(1, -1, 1, 1)
        for dy in range(3):
            for dx in range(3):
                z = z + torch.einsum("oc,bchw->bohw", wk[:, :, dy, dx], hp[:, :, dy:dy + H, dx:dx + W])
        return F.leaky_relu(z, 0.1)

    pool = lambda h: F.avg_pool2d(h, 2)
    up = lambda h: h.repeat_interleave(2, 2).repeat_interleave(2, 3)
    h = x.double().permute(0, 3, 1, 2)
    s1 = conv(conv(h, 0), 1)
    s2 = conv(conv(pool(s1), 2), 3)
    s3 = conv(conv(pool(s2), 4), 5)
    h = conv(conv(pool(s3), 6), 7)
    for k, skip in ((8, s3), (11, s2), (14, s1)):
        h = conv(conv(torch.cat([conv(up(h), k), skip], 1), k + 1), k + 2)
    phi = torch.sigmoid(torch.einsum("bchw,c->bhw", h, p[o:o + c["base"]]) + p[-1])
    if c["kind"] == "forward":
        return phi.detach()
    m = mask.double()
    loss = ((phi - t.double()) ** 2 * m).sum() / m.sum()
    loss.backward()
    return loss.detach(), p.grad


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind == "lattice":
        return _exact_lattice(c, seed)
    if kind == "batch":
        if c["n"] * c["steps"] > 6000:
            return None
        out = []
        for o, (m, walls, drop) in _batch_sizes(c, seed):
            e = _Exact(o["nx"], o["ny"], m, walls, drop)
            for _ in range(c["steps"]):
                e.step()
            out.append(e.rho[4:-4].reshape(-1))
        return torch.cat(out), None, None
    if kind == "measure":
        return _exact_measure(c, seed)
    return _exact_net(c, seed)
