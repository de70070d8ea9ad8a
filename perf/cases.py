"""The calls that a user of the lattice Boltzmann library spends time in, as
cases with sizes, for timing and for comparing results.

A case is a dict of plain values:
  kind      "run": advance a simulation by `steps` and read it out (`out`:
            "moments", the density and velocity fields; "state", the raw
            populations, as a checkpoint takes them; "both"); "study":
            initialise, advance, reduce and read the droplet statistics and the
            fields;
            "adjoint": initialise at rest, record `steps`, differentiate a loss
            of the final densities
  nz ny nx  lattice cells
  storage   population format; collision, forcing, tau1, tau2, G (the signed
            interaction strength), rho_s1, rho_s2 (wall potential), gx (body
            force along x) as in Lattice
  walls     "none" (periodic), or the wall model at z walls ("mirror",
            "potential") or of a mask of solid sites
  mask      "none", "slab" (inclined staircase wall), "sphere" (one cell of a
            sphere array) or "channel" (inclined staircase channel)
  init      "droplet", "mixture", "hemisphere" (on the wall z = -1/2),
            "uniform"
Every start but those of the adjoint moves: the two-phase states met in earnest
carry flows of a few hundredths of a lattice unit per step.
"""
import math

import torch

from paper_1601_01237_gb300.lattice import Lattice

# The library's direction order (include/lbm.h), opposite directions side by side.
CX = (0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0)
CY = (0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1)
CZ = (0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1)
K36 = (12,) + (2,) * 6 + (1,) * 12          # 36 w_i
BYTES = {"f64": 8, "f32": 4, "f16_dev": 2, "bf16_dev": 2, "f16_rel": 2, "bf16_rel": 2}
# Arithmetic of one two-component cell update (moments 76, interaction sums 80,
# collision 2 x 19 x 20), rounded; of one reverse step, about twice that.
FLOPS_STEP, FLOPS_REVERSE = 900, 1800

DEFAULTS = dict(kind="run", storage="f32", collision="bgk", forcing="edm", tau1=1.0, tau2=1.0, G=-1.8, rho_s1=0.0,
                rho_s2=0.0, gx=0.0, walls="none", mask="none", init="droplet", out="moments", ckpt=0)


def _case(**kw):
    return dict(DEFAULTS, **kw)


def listed():
    return [
        # Watching a quasi-2D droplet step by step (the static-droplet study's
        # side of 5 R with R = 16): one step and its fields, the smallest call.
        _case(name="monitor_2d", nz=1, ny=80, nx=80, steps=1),
        # The quasi-2D droplet in FP64, a stretch of a long run up to its next
        # output and checkpoint.
        _case(name="droplet_2d_f64", nz=1, ny=64, nx=64, storage="f64", steps=100, out="both"),
        # The wetting study: a droplet on a wall in a thin x-z lattice, modified
        # wall model with a wall potential.
        _case(name="wetting_2d", nz=64, ny=1, nx=160, init="hemisphere", walls="mirror", rho_s2=0.2, steps=200,
              out="both"),
        # Flow through the array of touching spheres: FP64, solid sites, driven
        # by a body force, one 34^3 cell.
        _case(name="spheres_f64", nz=34, ny=34, nx=34, storage="f64", collision="regularized", tau1=0.8, tau2=0.8,
              G=0.0, gx=1e-4, walls="mirror", mask="sphere", init="uniform", steps=20, out="both"),
        # One point of the surface-tension study: a 128^3 droplet from its
        # initial fields to its pressure jump and statistics.
        _case(name="tension_128", kind="study", nz=128, ny=128, nx=128, steps=50, out="study"),
        # Spinodal decomposition at 256^3, regularized, tau = 0.7, FP32 with its
        # fields read out.
        _case(name="mixture_256", nz=256, ny=256, nx=256, collision="regularized", tau1=0.7, tau2=0.7, G=-1.2,
              init="mixture", steps=20),
        # The same run in the 16-bit deviation format, checkpointed.
        _case(name="mixture_256_f16", nz=256, ny=256, nx=256, storage="f16_dev", collision="regularized", tau1=0.7,
              tau2=0.7, G=-1.2, init="mixture", steps=20, out="state"),
        # A lattice of odd sizes in the relative 16-bit format, with the other
        # forcing scheme and the third-order filter.
        _case(name="ragged_bf16_rel", nz=131, ny=150, nx=173, storage="bf16_rel", collision="regularized3",
              forcing="guo", tau1=0.8, tau2=0.9, G=-2.4, init="mixture", steps=20, out="state"),
        # Differentiation at 96^3: forward with checkpoints every 25 steps, then
        # the gradient of a loss of the final densities.
        _case(name="adjoint_96", kind="adjoint", nz=96, ny=96, nx=96, steps=50, ckpt=25, out="gradients"),
        # An inclined staircase wall of solid sites across a 256^3 mixture.
        _case(name="mask_256", nz=256, ny=256, nx=256, G=-1.2, init="mixture", walls="mirror", mask="slab", steps=20),
        # The wall-attached droplet on 512 x 512 x 384 (regularized, tau = 0.55).
        _case(name="wall_512", nz=384, ny=512, nx=512, collision="regularized", tau1=0.55, tau2=0.55, G=-1.2,
              walls="mirror", init="hemisphere", steps=10, out="state"),
        # The throughput workload: 512^3, FP32, periodic mixture.
        _case(name="throughput_512", nz=512, ny=512, nx=512, G=-1.2, init="mixture", steps=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: thin and quasi-2D lattices, FP64, walls and masks, 3D
    lattices from 24 to 320 cells a side in every format, and differentiation."""
    what = rng.choice(["plane", "wall2d", "channel", "fp64", "cube", "cube", "half", "mask", "walls", "adjoint", "study"])
    reg = rng.choice(["bgk", "regularized"])
    if what == "plane":
        return _case(nz=1, ny=_log(rng, 40, 700), nx=_log(rng, 40, 700), collision=reg, steps=_log(rng, 1, 300))
    if what == "wall2d":
        return _case(nz=_log(rng, 32, 300), ny=1, nx=_log(rng, 80, 600), init="hemisphere",
                     walls=rng.choice(["mirror", "potential"]), rho_s2=round(rng.uniform(0.0, 0.4), 3),
                     steps=_log(rng, 1, 300))
    if what == "channel":
        return _case(nz=rng.randint(40, 200), ny=1, nx=rng.randint(90, 300), collision="regularized",
                     walls=rng.choice(["mirror", "potential"]), rho_s2=0.4, mask="channel", steps=_log(rng, 1, 300))
    if what == "fp64":
        if rng.random() < 0.5:
            return _case(nz=1, ny=_log(rng, 40, 300), nx=_log(rng, 40, 300), storage="f64", collision=reg,
                         steps=_log(rng, 1, 100))
        L = _log(rng, 20, 100)
        return _case(nz=L, ny=L, nx=L, storage="f64", collision=rng.choice(["bgk", "regularized", "regularized3"]),
                     tau1=0.8, tau2=0.8, G=0.0, gx=1e-4, walls="mirror", mask=rng.choice(["none", "sphere"]),
                     init="uniform", steps=_log(rng, 1, 30))
    n = [_log(rng, 24, 320) for _ in range(3)]
    guo = rng.random() < 0.25
    mix = dict(nz=n[0], ny=n[1], nx=n[2], init="mixture", forcing="guo" if guo else "edm", G=-2.4 if guo else -1.2,
               steps=_log(rng, 2, 20))
    if guo:
        reg = "regularized"
    tau = 1.0 if reg == "bgk" else round(rng.uniform(0.65, 1.0), 3)
    if what == "cube":
        return _case(collision=reg, tau1=tau, tau2=tau, out=rng.choice(["moments", "state"]), **mix)
    if what == "half":
        return _case(storage=rng.choice(["f16_dev", "bf16_dev", "f16_rel", "bf16_rel"]),
                     collision=rng.choice([reg, "regularized"]), tau1=tau, tau2=tau, out="state", **mix)
    if what == "mask":
        return _case(collision=reg, tau1=tau, tau2=tau, walls=rng.choice(["mirror", "potential"]), mask="slab", **mix)
    if what == "walls":
        return _case(nz=n[0], ny=n[1], nx=n[2], collision="regularized", tau1=0.6, tau2=0.6, G=-1.2,
                     walls=rng.choice(["mirror", "potential"]), init="hemisphere", steps=_log(rng, 2, 20), out="state")
    n = [_log(rng, 24, 96) for _ in range(3)]
    if what == "study":
        return _case(kind="study", nz=n[0] + 24, ny=n[1] + 24, nx=n[2] + 24, steps=_log(rng, 10, 50), out="study")
    steps = rng.randint(8, 50)
    return _case(kind="adjoint", nz=n[0], ny=n[1], nx=n[2], collision=rng.choice(["bgk", "regularized"]), steps=steps,
                 ckpt=rng.randint(2, 25), out="gradients")


# --------------------------------------------------------------------------
# inputs

def _grid(c):
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (c["nz"], c["ny"], c["nx"])]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


def _dist(v, c, n):
    d = v - c
    return d - n * torch.round(d / n)


def _solid(c):
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    if c["mask"] == "none":
        return None
    z, y, x = _grid(c)
    if c["mask"] == "slab":          # 8 cells thick at 30 degrees along x
        m = torch.remainder(z - torch.floor(x * math.tan(math.radians(30.0))), nz) < 8
        return m.expand(nz, ny, nx).contiguous()
    if c["mask"] == "sphere":
        r2 = (z - (nz - 1) / 2) ** 2 + (y - (ny - 1) / 2) ** 2 + (x - (nx - 1) / 2) ** 2
        return r2 < (min(nz, ny, nx) / 2.0) ** 2
    # a channel along the lattice's diagonal, of height 16 across it
    L = math.hypot(nx, nz)
    d = -(x - (nx - 1) / 2) * nz / L + (z - (nz - 1) / 2) * nx / L
    P = nx * nz / L
    d = d - P * torch.round(d / P)
    return (d.abs() >= 8.0).expand(nz, ny, nx).contiguous()


def _fields(c, seed):
    """(rho1, rho2, u or None, solid or None) of the start, FP64 on the GPU."""
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    shape = (nz, ny, nx)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 17)
    r = torch.rand(12, dtype=torch.float64, device="cuda", generator=gen).cpu().tolist()
    z, y, x = _grid(c)
    if c["init"] == "mixture":
        rho = [0.5 * (1.0 + 0.01 * (2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0))
               for _ in range(2)]
    elif c["init"] == "uniform":
        rho = [torch.full(shape, 0.5 + 0.01 * r[k], dtype=torch.float64, device="cuda") for k in range(2)]
    else:
        thin = [n for n in shape if n > 1]
        R = min(thin) * (0.2 + 0.05 * r[0])
        if c["init"] == "hemisphere":
            cen = (-0.5, (ny - 1) * r[1], (nx - 1) * r[2])
        else:
            cen = [(n - 1) * (0.45 + 0.1 * v) for n, v in zip(shape, r[1:4])]
        dy = _dist(y, cen[1], ny) if ny > 1 else 0.0 * y
        dz = (z - cen[0]) if c["init"] == "hemisphere" else (_dist(z, cen[0], nz) if nz > 1 else 0.0 * z)
        dist = torch.sqrt(dz ** 2 + dy ** 2 + _dist(x, cen[2], nx) ** 2)
        # near the densities that coexist at the case's interaction strength
        hi, lo = (1.0, 0.03) if abs(c["G"]) >= 1.5 else (0.897, 0.148)
        a = lo + 0.5 * (hi - lo) * (1.0 - torch.tanh((dist - R) / 2.0))
        a = a * (1.0 + 1e-3 * (2.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0))
        rho = [a, hi + lo - a]
    rho = [t.contiguous() for t in rho]
    if c["kind"] == "adjoint":
        return rho[0], rho[1], None, None
    # a shear flow over the lattice, along x and y (and z where that is periodic)
    free_z = c["walls"] == "none" or c["mask"] != "none"
    u = torch.empty(shape + (3,), dtype=torch.float64, device="cuda")
    tz, ty, tx = (2 * math.pi * (t + 0.5) / n for t, n in ((z, nz), (y, ny), (x, nx)))
    u[..., 0] = 0.03 * (0.8 + 0.4 * r[5]) * (1.0 + 0.5 * torch.sin(tz + ty))
    u[..., 1] = 0.02 * (0.8 + 0.4 * r[6]) * (1.0 + 0.5 * torch.cos(tx))
    u[..., 2] = -0.02 * (0.8 + 0.4 * r[7]) * (1.0 + 0.5 * torch.sin(ty + tx)) if free_z else 0.0 * (tx + ty)
    return rho[0], rho[1], u, _solid(c)


def _options(c):
    kw = dict(storage=c["storage"], collision=c["collision"], forcing=c["forcing"], tau=(c["tau1"], c["tau2"]),
              G12=c["G"], rho_s=(c["rho_s1"], c["rho_s2"]), g_ext=(c["gx"], 0.0, 0.0))
    if c["walls"] != "none":
        kw["wall_model"] = c["walls"]
        if c["mask"] == "none":
            kw["periodic"] = (1, 1, 0)
    if c["storage"].endswith("_dev"):
        kw["rho0_dev"] = 0.5
    return kw


def _droplet_frame(c):
    """Centre for the pressure jump and origin for the droplet's centre of mass."""
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    m = min(nz, ny, nx)
    return ((nx - 1) / 2, (ny - 1) / 2, (nz - 1) / 2), 0.1 * m, 0.4 * m, ((nx - 1) / 2 - 5, (ny - 1) / 2 - 7, (nz - 1) / 2 - 9)


class _State:
    pass


def prepare(case, seed):
    c = case
    s = _State()
    s.c = c
    shape = (c["nz"], c["ny"], c["nx"])
    r1, r2, u, solid = _fields(c, seed)
    s.lat = Lattice(shape, **_options(c))
    if solid is not None:
        s.lat.set_solid(solid.to(torch.uint8))
    if c["kind"] == "run":
        s.lat.init_fields(r1, r2, u)
    else:
        s.rho, s.u = (r1, r2), u
    R = torch.float64 if c["storage"] == "f64" else torch.float32
    s.f64 = R == torch.float64
    s.view = []
    if c["out"] in ("state", "both"):
        # the populations, as the storage type, and behind them (relative
        # formats, at the next multiple of 256 bytes) the reference densities
        s.buf = torch.zeros(s.lat.state_bytes(), dtype=torch.uint8, device="cuda")
        T = {"f64": torch.float64, "f32": torch.float32, "f16_dev": torch.float16, "f16_rel": torch.float16,
             "bf16_dev": torch.bfloat16, "bf16_rel": torch.bfloat16}[c["storage"]]
        N = shape[0] * shape[1] * shape[2]
        nb = 38 * N * BYTES[c["storage"]]
        s.view = [s.buf[:nb].view(T)]
        if c["storage"].endswith("_rel"):
            off = (nb + 255) // 256 * 256
            s.view.append(s.buf[off:off + 8 * N].view(torch.float32))
    if c["out"] != "state":
        s.m = [torch.zeros(shape, dtype=R, device="cuda") for _ in range(2)]
        if c["out"] != "gradients":
            s.m.append(torch.zeros(shape + (3,), dtype=R, device="cuda"))
    if c["kind"] == "adjoint":
        s.seed = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2)]
        s.grad = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(2)]
        s.target = _target(c)
    return s


def _target(c):
    """Target density of the differentiation loss: an ellipsoid of component 1."""
    z, y, x = _grid(c)
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    q = torch.sqrt(((z - (nz - 1) / 2) / (0.17 * nz)) ** 2 + ((y - (ny - 1) / 2) / (0.21 * ny)) ** 2 +
                   ((x - (nx - 1) / 2) / (0.25 * nx)) ** 2)
    return 0.03 + 0.485 * (1.0 - torch.tanh((q - 1.0) * 0.1 * min(nz, ny, nx)))


def run(state):
    s, c, lat = state, state.c, state.lat
    if c["kind"] == "run":
        lat.step(c["steps"])
        if s.view:
            lat.get_state(s.buf)
        if c["out"] != "state":
            lat.moments_device(s.m[0], s.m[1], s.m[2], out_f64=s.f64)
        return {"fields": s.m if c["out"] != "state" else [], "state": s.view}
    if c["kind"] == "study":
        lat.init_fields(s.rho[0], s.rho[1], s.u)
        lat.step(c["steps"])
        centre, r_in, r_out, origin = _droplet_frame(c)
        red = lat.reduce()
        jump = lat.pressure_jump(centre, r_in, r_out)
        st = lat.droplet_stats(0.515, origin)
        lat.moments_device(s.m[0], s.m[1], s.m[2], out_f64=s.f64)
        return [s.m, [red["mass1"], red["mass2"], red["max_uF"]] + list(red["momentum"]), list(jump),
                [st["volume"], st["mass"]] + list(st["com"])]
    # adjoint: the loss sum (rho1 - target)^2 + sum rho1 rho2 / 2 of the final densities
    lat.init_fields(s.rho[0], s.rho[1])
    lat.record(c["steps"], c["ckpt"])
    lat.moments_device(s.m[0], s.m[1], None, out_f64=False)
    s.seed[0].copy_(s.m[0]).sub_(s.target).mul_(2.0).add_(s.m[1], alpha=0.5)
    s.seed[1].copy_(s.m[0]).mul_(0.5)
    par = lat.adjoint(s.seed[0], s.seed[1], s.grad[0], s.grad[1])
    return [s.m, [g.float() for g in s.grad], list(par)]


def work(case):
    c = case
    N = c["nz"] * c["ny"] * c["nx"]
    b = BYTES[c["storage"]]
    state = 38 * b * N + (8 * N if c["storage"].endswith("_rel") else 0)
    R = 8 if c["storage"] == "f64" else 4
    out = {"state": 2 * state, "moments": state + 5 * R * N, "both": 2 * state + 5 * R * N, "study": state + 5 * R * N,
           "gradients": state + 2 * R * N}[c["out"]]
    steps = c["steps"]
    bytes_, flops = 2 * state * steps + out, FLOPS_STEP * N * steps
    if c["kind"] == "study":
        bytes_ += (5 * 8 * N + state) + 2 * state     # set-up; reductions of the final state
    if c["kind"] == "adjoint":
        # set-up; per reverse step the forward step it replays, the state it
        # differentiates and the sensitivities in and out
        bytes_ += (2 * 8 * N + state) + steps * (2 * state + state + 2 * 38 * R * N) + 4 * 8 * N
        flops += steps * N * (FLOPS_STEP + FLOPS_REVERSE)
    return {"bytes": float(bytes_), "flops": float(flops)}


# --------------------------------------------------------------------------
# the same update in 64 bits

def _opp(i):
    return 0 if i == 0 else (i + 1 if i & 1 else i - 1)


def _at(t, i, sign=1):
    """t(x + sign c_i), periodic."""
    return torch.roll(t, shifts=(-sign * CZ[i], -sign * CY[i], -sign * CX[i]), dims=(0, 1, 2)) if i else t


def _acc(a, k, t):
    return a if k == 0 else (a + t if k > 0 else a - t)


class _Model:
    def __init__(self, c, solid, G12=None, G21=None, tau1=None, tau2=None):
        self.c, self.solid = c, solid
        self.G = (c["G"] if G12 is None else G12, c["G"] if G21 is None else G21)
        self.tau = (c["tau1"] if tau1 is None else tau1, c["tau2"] if tau2 is None else tau2)
        self.rho_s = (c["rho_s1"], c["rho_s2"])
        self.wallz = c["walls"] != "none" and c["mask"] == "none"
        self.links = None
        if solid is not None:
            self.links = [None] + [_at(solid, i, -1) for i in range(1, 19)]   # x - c_i is solid
            self.den = sum(K36[i] * (~_at(solid, i)).double() for i in range(1, 19))

    def feq(self, i, v):
        """f^eq / rho of direction i and its opposite."""
        vsq = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
        w = K36[i] / 36.0
        if i == 0:
            return w * (1.0 - 1.5 * vsq), None
        cv = CX[i] * v[0] + CY[i] * v[1] + CZ[i] * v[2]
        E, O = 1.0 - 1.5 * vsq + 4.5 * cv * cv, cv * (3.0 - 4.5 * vsq + 4.5 * cv * cv)
        return w * (E + O), w * (E - O)

    def init(self, rho, u):
        f = []
        for a in range(2):
            fa = []
            for i in range(19):
                if u is None:
                    fa.append(rho[a] * (K36[i] / 36.0))
                    continue
                p, m = self.feq(i if i == 0 or i & 1 else i - 1, (u[..., 0], u[..., 1], u[..., 2]))
                fa.append(rho[a] * (p if i == 0 or i & 1 else m))
            f.append(fa)
        if self.solid is not None:
            f = [[torch.where(self.solid, 0.0, t) for t in fa] for fa in f]
        return f

    def rho(self, f):
        r = []
        for fa in f:
            t = fa[0]
            for i in range(1, 19):
                t = t + fa[i]
            r.append(t)
        return r

    def force(self, rho):
        """g^1, g^2 (three components each)."""
        S = []
        for b in range(2):
            r = rho[b]
            if self.solid is not None:
                wall = torch.full_like(r, self.rho_s[b])
                if self.c["walls"] == "mirror":
                    num = sum(K36[i] * _at(torch.where(self.solid, 0.0, r), i) for i in range(1, 19))
                    wall = wall + torch.where(self.den > 0, num / self.den.clamp(min=1.0), 0.0)
                r = torch.where(self.solid, wall, r)
            s = [0.0, 0.0, 0.0]
            for i in range(1, 19):
                v = _at(r, i)
                if self.wallz and CZ[i]:
                    z = 0 if CZ[i] < 0 else -1
                    flat = torch.roll(r[z], shifts=(-CY[i], -CX[i]), dims=(0, 1)) if self.c["walls"] == "mirror" else 0.0 * r[z]
                    wall = (flat + self.rho_s[b])[None]
                    v = torch.cat([wall, v[1:]]) if z == 0 else torch.cat([v[:-1], wall])
                v = v * (K36[i] / 36.0)
                s = [_acc(s[0], CX[i], v), _acc(s[1], CY[i], v), _acc(s[2], CZ[i], v)]
            S.append(s)
        ext = (self.c["gx"], 0.0, 0.0)
        return [[self.G[a] * S[1 - a][d] + ext[d] for d in range(3)] for a in range(2)]

    def velocity(self, f, rho):
        j = [0.0, 0.0, 0.0]
        for i in range(1, 19):
            t = f[0][i] + f[1][i]
            j = [_acc(j[0], CX[i], t), _acc(j[1], CY[i], t), _acc(j[2], CZ[i], t)]
        den = rho[0] + rho[1]
        if self.solid is not None:
            den = torch.where(self.solid, 1.0, den)
        return [t / den for t in j], den

    def moments(self, f):
        rho = self.rho(f)
        u, den = self.velocity(f, rho)
        g = self.force(rho)
        uF = torch.stack([u[d] + 0.5 * (g[0][d] * rho[0] + g[1][d] * rho[1]) / den for d in range(3)], -1)
        if self.solid is not None:
            uF = torch.where(self.solid[..., None], 0.0, uF)
        return rho, uF

    def step(self, f, streamed=True):
        """The next populations (streamed), or the post-collision ones."""
        reg = {"bgk": 0, "regularized": 1, "regularized3": 2}[self.c["collision"]]
        guo = self.c["forcing"] == "guo"
        rho = self.rho(f)
        u, den = self.velocity(f, rho)
        g = self.force(rho)
        if guo:
            u = [u[d] + 0.5 * (g[0][d] * rho[0] + g[1][d] * rho[1]) / den for d in range(3)]
        new = []
        for a in range(2):
            fa, om = f[a], 1.0 / self.tau[a]
            keep = 1.0 - om
            v = u if guo else [u[d] + g[a][d] for d in range(3)]
            F = [rho[a] * g[a][d] for d in range(3)]
            uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2] if guo else None

            def force_term(i):
                cu = CX[i] * u[0] + CY[i] * u[1] + CZ[i] * u[2]
                cF = CX[i] * F[0] + CY[i] * F[1] + CZ[i] * F[2]
                return (K36[i] / 36.0) * (3.0 * (cF - uF) + 9.0 * cu * cF)

            if reg:
                # f^neq (with Guo's forcing, f - f^eq + F/2) projected on the second-
                # and, for reg = 2, third-order Hermite polynomials of the lattice
                P = [[0.0] * 3 for _ in range(3)]
                H = {}
                for i in range(0, 19):
                    e = self.feq(i if i == 0 or i & 1 else i - 1, u)
                    n = fa[i] - rho[a] * (e[0] if i == 0 or i & 1 else e[1])
                    if guo:
                        n = n + 0.5 * force_term(i)
                    cc = (CX[i], CY[i], CZ[i])
                    for p in range(3):
                        for q in range(p, 3):
                            if cc[p] * cc[q]:
                                P[p][q] = P[p][q] + cc[p] * cc[q] * n
                    if reg == 2:
                        for p in range(3):
                            for q in range(3):
                                if p != q:
                                    h = cc[p] * (cc[q] ** 2 - 1.0 / 3.0)
                                    if h:
                                        H[p, q] = H.get((p, q), 0.0) + h * n

            def post(i):
                b = i if i == 0 or i & 1 else i - 1
                k = 0 if i == b else 1
                e = rho[a] * self.feq(b, v)[k]
                if not reg:
                    o = e + keep * (fa[i] - rho[a] * self.feq(b, u)[k])
                    return o + (1.0 - 0.5 * om) * force_term(i) if guo else o
                cc = (CX[i], CY[i], CZ[i])
                n = 0.0
                for p in range(3):
                    n = n + 4.5 * (cc[p] * cc[p] - 1.0 / 3.0) * P[p][p]
                    for q in range(p + 1, 3):
                        if cc[p] * cc[q]:
                            n = n + 9.0 * cc[p] * cc[q] * P[p][q]
                if reg == 2:
                    for p in range(3):
                        q, r = [t for t in range(3) if t != p]
                        hq, hr = cc[p] * (cc[q] ** 2 - 1.0 / 3.0), cc[p] * (cc[r] ** 2 - 1.0 / 3.0)
                        # the sum and the difference of the pair are orthogonal, norms 2/27 and 6/27
                        if hq + hr:
                            n = n + (27.0 / 2.0) * (hq + hr) * (H[p, q] + H[p, r])
                        if hq - hr:
                            n = n + (27.0 / 6.0) * (hq - hr) * (H[p, q] - H[p, r])
                o = e + keep * (K36[i] / 36.0) * n
                return o + 0.5 * force_term(i) if guo else o

            na = [None] * 19
            na[0] = post(0)
            for i in range(1, 19, 2):
                pi, pm = post(i), post(i + 1)
                if self.solid is not None:
                    pi, pm = torch.where(self.solid, 0.0, pi), torch.where(self.solid, 0.0, pm)
                na[i], na[i + 1] = self.stream(i, pi, pm) if streamed else (pi, pm)
            if self.solid is not None:
                na[0] = torch.where(self.solid, 0.0, na[0])
            new.append(na)
        return new

    def stream(self, i, pi, pm):
        a, b = _at(pi, i, -1), _at(pm, i)
        if self.links is not None:
            a, b = torch.where(self.links[i], pm, a), torch.where(self.links[i + 1], pi, b)
            a, b = torch.where(self.solid, 0.0, a), torch.where(self.solid, 0.0, b)
        elif self.wallz and CZ[i]:
            if CZ[i] > 0:
                a, b = torch.cat([pm[:1], a[1:]]), torch.cat([b[:-1], pi[-1:]])
            else:
                a, b = torch.cat([a[:-1], pm[-1:]]), torch.cat([pi[:1], b[1:]])
        return a, b


def exact(case, seed):
    c = case
    r1, r2, u, solid = _fields(c, seed)
    if c["kind"] == "adjoint":
        return _exact_adjoint(c, r1, r2)
    m = _Model(c, solid)
    with torch.no_grad():
        f = m.init((r1, r2), u)
        del u
        for k in range(c["steps"]):
            last = k + 1 == c["steps"]
            g = m.step(f, streamed=not last)
            if not last:
                f = g
        state = []
        if c["out"] in ("state", "both") and not c["storage"].endswith("_rel"):
            # (the relative formats' codes and references mix two time levels: no value of their own)
            N = r1.numel()
            out = torch.empty(19 * N, 2, dtype=torch.float64, device="cuda")
            for a in range(2):
                for i in range(19):
                    ref = 0.5 * K36[i] / 36.0 if c["storage"].endswith("_dev") else 0.0
                    out[i * N:(i + 1) * N, a] = (g[a][i] - ref).reshape(-1)
            state = [out.reshape(-1)]
        elif c["out"] == "state":
            return None
        if c["out"] == "state":
            return {"fields": [], "state": state}
        for a in range(2):
            for i in range(1, 19, 2):
                g[a][i], g[a][i + 1] = m.stream(i, g[a][i], g[a][i + 1])
        del f
        rho, uF = m.moments(g)
        if c["kind"] == "run":
            return {"fields": [rho[0], rho[1], uF], "state": state}
        tot = rho[0] + rho[1]
        red = [float(rho[0].sum()), float(rho[1].sum()), float(uF.square().sum(-1).max().sqrt())]
        red += [float((tot * uF[..., d]).sum()) for d in range(3)]
        centre, r_in, r_out, origin = _droplet_frame(c)
        z, y, x = _grid(c)
        n = (c["nx"], c["ny"], c["nz"])
        d = [_dist(t, o, k) for t, o, k in zip((x, y, z), centre, n)]
        dist = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        p = (rho[0] + rho[1]) / 3.0 - c["G"] / 3.0 * rho[0] * rho[1]
        jump = [float(p[dist < r_in].mean()), float(p[dist > r_out].mean())]
        jump.append(jump[0] - jump[1])
        inside = rho[0] > 0.515
        st = [float(inside.sum()), float(rho[0][inside].sum())]
        st += [float(_dist(t, o, k).expand(inside.shape)[inside].mean()) for t, o, k in zip((x, y, z), origin, n)]
        return [[rho[0], rho[1], uF], red, jump, st]


def _exact_adjoint(c, r1, r2):
    from torch.utils.checkpoint import checkpoint
    if r1.numel() * c["steps"] > 5e7:
        return None
    r1, r2 = r1.requires_grad_(), r2.requires_grad_()
    par = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True)
           for v in (c["G"], c["G"], c["tau1"], c["tau2"])]
    m = _Model(c, None, *par)
    f = m.init((r1, r2), None)

    def step(*flat):
        new = m.step([list(flat[:19]), list(flat[19:])])
        return tuple(new[0] + new[1])

    flat = tuple(f[0] + f[1])
    for _ in range(c["steps"]):
        flat = checkpoint(step, *flat, use_reentrant=False)
    a, b = m.rho([list(flat[:19]), list(flat[19:])])
    loss = ((a - _target(c)) ** 2).sum() + 0.5 * (a * b).sum()
    loss.backward()
    return [[a.detach(), b.detach()], [r1.grad, r2.grad], [float(p.grad) for p in par]]
