"""Performance cases of the kinetic Monte Carlo step library: what users of the
framework have it do, through the public calls of paper_1210_8084_gb300.

A case is one simulation (or an ensemble of them) on the device and a pass of it
is what a driver loop does between two outputs: advance the handle, read the
moments and the state into device buffers.  The handle goes on from pass to pass
as a run does; the blast and implosion cases, whose state would drift away from
the physics they stand for, start every pass from a kept checkpoint
(kmc_set_state).  Initial states follow the recipes of the package's `inputs`
module, drawn on the GPU.
"""
import math

import numpy as np
import torch

import paper_1210_8084_gb300 as kmc
from paper_1210_8084_gb300 import inputs

DEV = "cuda"
PER, WALL, ABSORB = kmc.KMC_BC_PERIODIC, kmc.KMC_BC_WALL, kmc.KMC_BC_ABSORB
MASK = kmc.KMC_MOM_RAW | kmc.KMC_MOM_DERIVED | kmc.KMC_MOM_GLOBAL


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest run there is: a test-sized slab tube, binary64, candidates and pairs recorded;
        # a step is a handful of launches
        dict(name="tube_4k_fp64", kind="slab", n=4_000, nx=20, lam=1e-3, precision=64, steps=1, record=True),
        # closest candidates for a host framework that owns all device memory (no allocation), close
        # to the call's particle limit
        dict(name="partners_250k", kind="partners", n=250_000, nx=22, sub=2, lam=1e-3, precision=32, steps=1),
        # the plain method in binary64: 200k-particle slab Sod tube, ten steps between two outputs
        dict(name="tube_200k_fp64", kind="slab", n=200_000, nx=200, lam=1e-3, precision=64, steps=10, record=False),
        # cylindrical Noh implosion in the paper's 2-D mode (2-D velocities, radial moment), resumed
        # from a checkpoint and run on
        dict(name="noh2d_5M", kind="noh2d", n=5_000_000, nx=500, lam=1e-3, precision=32, steps=4),
        # Sedov-Taylor blast: absorbing walls, adaptive timestep, 8 particles per cubic c-bin, resumed
        dict(name="sedov3d_8M", kind="sedov3d", n=8_000_000, nx=100, lam=1e-3, precision=32, steps=1),
        # the random-partner comparison variant on the slab tube of the accuracy study
        dict(name="dsmc_4M", kind="dsmc", n=4_000_000, nx=2000, lam=1e-3, precision=32, steps=1),
        # slab Sod tube with 2000 c-bins, the middle of the Knudsen sweep
        dict(name="slab_16M", kind="slab", n=16_000_000, nx=2000, lam=1e-3, precision=32, steps=1, record=False),
        # the dense end of the Knudsen sweep (a hundred candidates per particle), sizes no power of two
        dict(name="slab_5M_dense", kind="slab", n=5_000_011, nx=1237, lam=1e-4, precision=32, steps=1, record=False),
        # the paper's Sod geometry: cubic c-bins with about 20 particles each
        dict(name="sod3d_21M", kind="sod3d", n=20 * 1024 * 32 * 32, nx=1024, ny=32, lam=1e-3, precision=32, steps=1),
        # four-quadrant Riemann problem in two dimensions, 240 particles per c-bin
        dict(name="quadrants_64M", kind="quadrants", n=64_000_000, nx=512, lam=5e-4, precision=32, steps=1),
        # batched ensemble: 256 uneven slab tubes in one handle
        dict(name="ensemble_256", kind="ensemble", instances=256, sizes=0, n_min=50_000, n_max=2_000_000, nx=200,
             precision=32, steps=1),
        # the largest run: 3-D Sod tube at scale, 122 particles per cubic c-bin
        dict(name="sod3d_512M", kind="sod3d", n=512_000_000, nx=1024, ny=64, lam=2e-4, precision=32, steps=1),
    ]


def _between(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _drawn(rng):
    kind = rng.choice(["slab", "slab", "sod3d", "sod3d", "quadrants", "noh2d", "sedov3d", "ensemble", "dsmc", "partners"])
    c = dict(kind=kind, precision=32, steps=1, lam=1e-3)
    if kind == "slab":
        c["precision"] = rng.choice([32, 32, 64])
        c["n"] = int(_between(rng, 4e3, 16e6 if c["precision"] == 32 else 1e6))
        c["nx"] = int(_between(rng, 20, min(2000, max(21, c["n"] // 50))))
        c["lam"] = _between(rng, 1e-4, 1.0)
        c["steps"] = rng.choice([1, 1, 10]) if c["n"] < 1_000_000 else 1
        c["record"] = c["n"] < 100_000
    elif kind == "sod3d":
        c["ny"] = int(_between(rng, 8, 64))
        c["nx"] = c["ny"] * rng.choice([8, 16, 32])
        c["n"] = int(_between(rng, 10, 130) * c["nx"] * c["ny"] ** 2)
        c["lam"] = _between(rng, 2e-4, 1e-3)
    elif kind == "quadrants":
        c["n"] = int(_between(rng, 1e5, 32e6))
        c["nx"] = max(8, int(math.sqrt(c["n"] / _between(rng, 20, 250))))
        c["lam"] = _between(rng, 1e-4, 1e-3)
    elif kind == "noh2d":
        c["n"] = int(_between(rng, 2e5, 8e6))
        c["nx"] = int(math.sqrt(c["n"] / 20))
        c["steps"] = rng.choice([1, 4])
    elif kind == "sedov3d":
        c["n"] = int(_between(rng, 2e5, 16e6))
        c["nx"] = int((c["n"] / 8) ** (1 / 3))
    elif kind == "ensemble":
        del c["lam"]
        c.update(instances=rng.randint(8, 64), sizes=rng.randrange(1 << 20), n_min=20_000, n_max=500_000,
                 nx=int(_between(rng, 100, 400)))
    elif kind == "dsmc":
        c["n"] = int(_between(rng, 1e5, 4e6))
        c["nx"] = int(_between(rng, 100, 2000))
        c["lam"] = _between(rng, 2.0, 20.0) / c["nx"]   # collision cells no wider than half a mean free path
    else:
        c["precision"] = rng.choice([32, 32, 64])
        c["n"] = int(_between(rng, 1e3, kmc.KMC_STATIC_MAX_PARTICLES))
        c["nx"] = max(3, int((c["n"] / _between(rng, 10, 40)) ** (1 / 3)))
        c["sub"] = rng.choice([1, 2, 3])
    return c


def draw(rng):
    while True:
        c = _drawn(rng)
        if _particles(c) > 64_000_000:
            continue
        pairs = sum(g["n"] * _window(c, g) for g in _instances(c))
        # a fine tube with a long reach costs more than any listed case: not drawn
        if pairs <= (2e10 if c["precision"] == 32 else 5e8):
            return c


# ------------------------------------------------- geometry, instances, config

def _geometry(c):
    """(position dimensions, cells, lo, hi, bc, flags)"""
    k, nx = c["kind"], c["nx"]
    one = (1.0, 1.0, 1.0)
    if k in ("slab", "ensemble"):
        return 3, (nx, 1, 1), one, (WALL, PER, PER), kmc.KMC_FLAG_RECORD if c.get("record") else 0
    if k == "dsmc":
        return 3, (nx, 1, 1), one, (WALL, PER, PER), kmc.KMC_FLAG_DSMC
    if k == "sod3d":
        return 3, (nx, c["ny"], c["ny"]), (1.0, c["ny"] / nx, c["ny"] / nx), (WALL, PER, PER), 0
    if k == "quadrants":
        return 2, (nx, nx, 1), one, (WALL, WALL, PER), 0
    if k == "noh2d":
        return 2, (nx, nx, 1), one, (WALL, WALL, PER), kmc.KMC_FLAG_VELOCITY_2D | kmc.KMC_FLAG_RADIAL_MOMENT
    if k == "sedov3d":
        return 3, (nx, nx, nx), one, (ABSORB, ABSORB, ABSORB), kmc.KMC_FLAG_ADAPTIVE_DT
    return 3, (nx, nx, nx), one, (PER, PER, PER), 0   # partners: a homogeneous periodic box


def _instances(c):
    """n, mean free path and timestep (0.2 of a c-bin at thermal speed 1) of every instance."""
    dt = 0.2 / c["nx"]
    if c["kind"] != "ensemble":
        return [dict(n=c["n"], lam=c["lam"], dt=1.0 if c["kind"] == "sedov3d" else dt, seed=0)]
    ns, lams = inputs.log_uniform_instances(c["instances"], c["sizes"], n_range=(c["n_min"], c["n_max"]))
    return [dict(n=int(n), lam=float(lam), dt=dt, seed=i) for i, (n, lam) in enumerate(zip(ns, lams))]


def _particles(c):
    return sum(g["n"] for g in _instances(c))


def _window(c, g):
    """About how many candidates lie within the reach of a step, per particle of instance g."""
    dim, cells, hi, _, _ = _geometry(c)
    vol = math.prod(hi[:dim])
    r = math.sqrt(vol / (math.pi * g["lam"] * g["n"])) + 2 * 5.5 * 0.2 / c["nx"]
    w = g["n"] / vol
    for d in range(dim):
        w *= min(2.5 * r, 3 * hi[d] / cells[d], hi[d])
    return 1.6 * w


def _config(c, seed):
    dim, cells, hi, bc, flags = _geometry(c)
    g = _instances(c)
    sub = (c["sub"],) * 3 if c["kind"] == "partners" else (0, 0, 0)
    return kmc.make_config(dim_pos=dim, n_cells=cells, hi=hi, bc=bc, lam=g[0]["lam"], dt=g[0]["dt"], seed=seed,
                           precision=c["precision"], flags=flags, sub_cells=sub,
                           instances=g if c["kind"] == "ensemble" else None)


def _inputs(c, seed):
    """Positions and velocities [n, 3] in the state precision, on the GPU."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    dt = torch.float32 if c["precision"] == 32 else torch.float64
    dim, _, hi, bc, _ = _geometry(c)

    def uniform(x, lo, up):   # in place, never the open upper end of a periodic dimension
        x.uniform_(lo, up, generator=gen)
        x.clamp_(max=float(np.nextafter(np.float32(up), np.float32(0))))

    n = _particles(c)
    pos = torch.empty((n, 3), device=DEV, dtype=dt)
    vel = torch.empty((n, 3), device=DEV, dtype=dt).normal_(generator=gen)
    for d in range(3):
        uniform(pos[:, d], 0.0, hi[d])
    k = c["kind"]
    if k in ("slab", "ensemble", "dsmc", "sod3d"):   # Sod: density 8 : 1, T 1 and 0.8, split at x = 1/2
        a = 0
        for g in _instances(c):
            m, b = a + round(g["n"] * 8 / 9), a + g["n"]
            pos[a:m, 0] *= 0.5
            pos[m:b, 0] = 0.5 + 0.5 * pos[m:b, 0]
            vel[m:b] *= math.sqrt(0.8)
            a = b
    elif k == "quadrants":
        a = 0
        counts = [int(n * w / 1.875) for w in (1.0, 0.5, 0.25, 0.125)]
        counts[0] += n - sum(counts)
        for m, cx, cy in zip(counts, (0.5, 0.0, 0.0, 0.5), (0.5, 0.5, 0.0, 0.0)):
            pos[a:a + m, 0] = cx + 0.5 * pos[a:a + m, 0]
            pos[a:a + m, 1] = cy + 0.5 * pos[a:a + m, 1]
            a += m
    elif k == "noh2d":
        r = pos[:, :2].norm(dim=1, keepdim=True).clamp(min=1e-30)
        vel *= 1e-3
        vel[:, :2] -= pos[:, :2] / r
        vel[:, 2] = 0.0
    elif k == "sedov3d":
        vel /= vel.norm(dim=1, keepdim=True)
        inside = (pos - 0.5).norm(dim=1, keepdim=True) <= 2.0 / c["nx"]
        vel *= torch.where(inside, 85.0, 1e-3).to(dt)
    if dim == 2:
        pos[:, 2] = 0.0
    return pos, vel


# ------------------------------------------------------------- prepare and run

def prepare(c, seed):
    pos, vel = _inputs(c, seed)
    cfg = _config(c, seed)
    torch.cuda.synchronize()   # the handle works on its own stream
    n = pos.shape[0]
    if c["kind"] == "partners":
        return dict(case=c, cfg=cfg, n=n, pos=pos, vel=vel, best=torch.empty(n, device=DEV, dtype=torch.int32))
    sim = kmc.Simulation(cfg, pos, vel, kmc.KMC_WHERE_DEVICE)
    radial = bool(cfg.flags & kmc.KMC_FLAG_RADIAL_MOMENT)
    mask = MASK | (kmc.KMC_MOM_RADIAL if radial else 0)
    nb, ni = sim.n_bins, sim.n_instances
    mom = torch.empty(kmc.kmc_moments_size(sim.h, mask), device=DEV, dtype=torch.float64)
    s = dict(case=c, sim=sim, mask=mask, mom=mom)
    s["out"] = dict(raw=mom[:8 * nb].view(nb, 8), derived=mom[8 * nb:16 * nb].view(nb, 8),
                    glob=mom[16 * nb:16 * nb + 8 * ni].view(ni, 8))
    if radial:
        s["out"]["radial"] = mom[16 * nb + 8 * ni:].view(nb, 2)
    if c["kind"] in ("noh2d", "sedov3d"):
        s["checkpoint"] = (pos, vel)
        pos, vel = torch.empty_like(pos), torch.empty_like(vel)
    s["out"].update(pos=pos, vel=vel)   # the initial arrays are free for the state read back
    if cfg.flags & kmc.KMC_FLAG_RECORD:
        s["out"].update(best=torch.empty(n, device=DEV, dtype=torch.int32),
                        partner=torch.empty(n, device=DEV, dtype=torch.int32))
    return s


def run(s):
    c = s["case"]
    where = kmc.KMC_WHERE_DEVICE
    if c["kind"] == "partners":
        rc = kmc.kmc_find_partners_noalloc(s["cfg"], s["n"], s["pos"], s["vel"], s["best"])
        if rc != kmc.KMC_OK:
            raise kmc.KmcError(rc, "kmc_find_partners_noalloc")
        return dict(best=s["best"])
    h, out = s["sim"].h, s["out"]
    if "checkpoint" in s:
        kmc.kmc_set_state(h, *s["checkpoint"], where, 0)
    kmc.kmc_step(h, c["steps"], 1)
    kmc.kmc_moments(h, s["mom"], where, s["mask"])
    kmc.kmc_get_state(h, out["pos"], out["vel"], where)
    if "best" in out:
        kmc.kmc_get_partners(h, out["best"], out["partner"], where)
    return out


def work(c):
    """One pass: the state read and written once (positions, velocities), the moments written; the
    pair tests (25 operations) of the candidates near enough to meet within the step, each pair once."""
    n, word = _particles(c), c["precision"] // 8
    _, cells, _, _, _ = _geometry(c)
    if c["kind"] == "partners":
        by = n * (6 * word + 4)
    else:
        by = n * 12 * word + math.prod(cells) * len(_instances(c)) * 16 * 8
    fl = 0.0
    for g in _instances(c):
        fl += 25 * 0.5 * g["n"] * (0.0 if c["kind"] == "dsmc" else _near(c, g)) + 100 * g["n"]
    return dict(bytes=float(by), flops=float(fl * c["steps"]))


def _near(c, g):
    """Candidates of the window within contact distance plus one step's thermal relative flight."""
    dim, _, hi, _, _ = _geometry(c)
    vol = math.prod(hi[:dim])
    r = math.sqrt(vol / (math.pi * g["lam"] * g["n"])) + 2.3 * 0.2 / c["nx"]
    return min(g["n"] / vol * (4.19 * r ** 3 if dim == 3 else 3.14 * r ** 2), _window(c, g))


# ----------------------------------------------- the same pass in plain 64 bits

MOST_PAIRS = 2e10   # window pairs a plain torch search goes through in some ten seconds
CHUNK = 1 << 25     # pairs at a time


def exact(c, seed):
    """What run() returns for these inputs, from plain torch: the pair decisions in the state's own
    arithmetic (they define the pairs), everything else in 64 bits.  A binary32 run of several steps
    has no such value: rounding of one step's state decides other pairs in the next."""
    pairs = sum(g["n"] * _window(c, g) for g in _instances(c)) * c["steps"]
    if c["kind"] == "dsmc" or pairs > MOST_PAIRS or (c["steps"] > 1 and c["precision"] == 32):
        return None
    pos, vel = _inputs(c, seed)
    parts, a = [], 0
    for g in _instances(c):
        b = a + g["n"]
        p, v = pos[a:b].contiguous(), vel[a:b].contiguous()
        key = seed if c["kind"] != "ensemble" else g["seed"]
        for step in range(c["steps"]):
            r = _one_step(c, g, p, v, step, key)
            p, v = r["pos"], r["vel"]
        parts.append(r)
        a = b
    r = {k: torch.cat([q[k] for q in parts]) for k in parts[0]}
    if c["kind"] == "partners":
        return dict(best=r["best"])
    if not c.get("record"):
        del r["best"], r["partner"]
    return r


def _fma(a, b, c):
    return (a.double() * b.double() + c.double()).to(a.dtype)


def _dot(a, b):   # a.b, first product rounded, then fused adds; a and b are lists of components
    s = a[0] * b[0]
    for x, y in zip(a[1:], b[1:]):
        s = _fma(x, y, s)
    return s


def _philox(c0, step, key):
    m32 = 0xFFFFFFFF
    x = [c0, torch.full_like(c0, step), torch.zeros_like(c0), torch.zeros_like(c0)]
    k0, k1 = key & m32, (key >> 32) & m32
    m0, m1 = 0xD2511F53, 0xCD9E8D57
    for _ in range(10):
        p0, p1 = x[0] * m0, x[2] * m1   # modulo 2^64
        x = [((p1 >> 32) & m32) ^ x[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ x[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return x


def _one_step(c, g, pos, vel, step, key):
    T = pos.dtype
    dim, cells, hi, bc, flags = _geometry(c)
    n, vol = pos.shape[0], math.prod(hi[:dim])
    plane = bool(flags & kmc.KMC_FLAG_VELOCITY_2D)
    R2 = vol / (g["lam"] * g["n"]) / math.pi
    vv = [vel[:, d] for d in range(3)]
    vmax = math.sqrt(float(_dot(vv, vv).max()))
    dt = g["dt"]
    if flags & kmc.KMC_FLAG_ADAPTIVE_DT:
        dt = min(hi[d] / cells[d] for d in range(dim)) / vmax
    R2t, dtt = torch.tensor(R2, dtype=T, device=DEV), torch.tensor(dt, dtype=T, device=DEV)
    best = _closest(pos, vel, dim, cells, hi, bc, R2t, dtt, math.sqrt(R2) + 2 * vmax * dt)
    me = torch.arange(n, device=DEV)
    partner = torch.where((best >= 0) & (best[best.clamp(min=0)] == me), best, -1)

    x, v, dt = pos.double(), vel.double(), float(dtt)
    i = (partner >= 0).nonzero()[:, 0]
    j = partner[i]
    dr, dv = x[i] - x[j], v[i] - v[j]
    for d in range(dim):
        if bc[d] == PER:
            dr[:, d] -= hi[d] * (dr[:, d] / hi[d]).round()
    dr[:, dim:] = 0.0
    tp = -(dr * dv).sum(1) / (dv[:, :dim] ** 2).sum(1)
    w = _philox(torch.minimum(i, j), step, key)
    if T == torch.float32:
        u1, u2 = ((w[0] >> 8) | 1).double() * 2.0 ** -24, ((w[2] >> 8) | 1).double() * 2.0 ** -24
    else:
        u1 = (2 * ((w[0] << 20) | (w[1] >> 12)) + 1).double() * 2.0 ** -53
        u2 = (2 * ((w[2] << 20) | (w[3] >> 12)) + 1).double() * 2.0 ** -53
    phi = 2 * math.pi * u2
    sth = 2 * (u1 * (1 - u1)).sqrt()
    nh = torch.stack([phi.cos(), phi.sin(), torch.zeros_like(phi)] if plane else
                     [sth * phi.cos(), sth * phi.sin(), 1 - 2 * u1], 1)
    sign = torch.where(i < j, 0.5, -0.5).double()
    vn = 0.5 * (v[i] + v[j]) + (sign * dv.norm(dim=1))[:, None] * nh
    xe, ve = x.clone(), v.clone()
    xe[:, :dim] += v[:, :dim] * dt
    xe[i, :dim] = x[i, :dim] + v[i, :dim] * tp[:, None] + vn[:, :dim] * (dt - tp)[:, None]
    ve[i] = vn
    W = torch.zeros(n, device=DEV, dtype=torch.float64)
    W[i] = ((dr + dv * tp[:, None])[:, :dim] * (vn - v[i])[:, :dim]).sum(1)
    gone = x[:, 0].isnan()
    for d in range(dim):
        if bc[d] == PER:
            xe[:, d] = xe[:, d].remainder(hi[d])
        elif bc[d] == ABSORB:
            gone |= (xe[:, d] < 0) | (xe[:, d] > hi[d])
        else:
            for _ in range(64):
                out = (xe[:, d] < 0) | (xe[:, d] > hi[d])
                if not bool(out.any()):
                    break
                xe[:, d] = torch.where(xe[:, d] < 0, -xe[:, d], torch.where(out, 2 * hi[d] - xe[:, d], xe[:, d]))
                ve[:, d] = torch.where(out, -ve[:, d], ve[:, d])
    r = _moments(xe[~gone], ve[~gone], W[~gone], (partner >= 0)[~gone], dim, cells, hi, dt, plane,
                 bool(flags & kmc.KMC_FLAG_RADIAL_MOMENT))
    xe[gone] = math.nan
    ve[gone] = math.nan
    r.update(pos=xe, vel=ve, best=best.int(), partner=partner.int())
    return r


def _moments(x, v, W, hit, dim, cells, hi, dt, plane, radial):
    nb = math.prod(cells)
    vc = math.prod(hi[:dim]) / nb
    b = torch.zeros(x.shape[0], device=DEV, dtype=torch.int64)
    for d in reversed(range(dim)):
        b = b * cells[d] + (x[:, d] * (cells[d] / hi[d])).long().clamp(0, cells[d] - 1)
    one = torch.ones_like(W)
    cols = [one, v[:, 0], v[:, 1], v[:, 2], v[:, 0] ** 2, v[:, 1] ** 2, v[:, 2] ** 2, W]
    raw = torch.stack([torch.zeros(nb, device=DEV, dtype=torch.float64).index_add_(0, b, q) for q in cols], 1)
    N = raw[:, 0].clamp(min=1)
    u = raw[:, 1:4] / N[:, None]
    temp = (raw[:, 4:7].sum(1) / N - (u ** 2).sum(1)) / (2 if plane else 3)
    pk = raw[:, 0] / vc * temp
    pv = raw[:, 7] / (2 * dim * vc * dt)
    der = torch.cat([(raw[:, 0] / vc)[:, None], u, torch.stack([temp, pk, pv, pk + pv], 1)], 1)
    der[raw[:, 0] == 0] = 0.0
    t = raw.sum(0)
    glob = torch.stack([t[0], 0.5 * t[4:7].sum(), t[1], t[2], t[3], t[7], 0.5 * hit.sum().double(), 0 * t[0]])[None]
    r = dict(raw=raw, derived=der, glob=glob)
    if radial:
        vr = (v[:, :dim] * x[:, :dim]).sum(1) / x[:, :dim].norm(dim=1).clamp(min=1e-300)
        s = torch.zeros(nb, device=DEV, dtype=torch.float64).index_add_(0, b, vr)
        r["radial"] = torch.stack([s, s / N], 1)
    return r


def _closest(pos, vel, dim, cells, hi, bc, R2, dt, reach):
    """Closest candidate of every particle over the neighbouring c-bins: a grid of cells no narrower
    than the step's reach inside each c-bin, all pairs of neighbouring cells tested."""
    n, T = pos.shape[0], pos.dtype
    M, cell = [], []
    for d in range(dim):
        s = max(1, min(400, int(hi[d] / cells[d] / (1.01 * reach + 1e-5 * hi[d]))))
        t = pos[:, d] * torch.tensor(cells[d] / hi[d], dtype=T, device=DEV)
        cb = t.long().clamp(0, cells[d] - 1)
        M.append(cells[d] * s)
        cell.append(cb * s + ((t - cb) * s).long().clamp(0, s - 1))
    flat = cell[0]
    for d in range(1, dim):
        flat = flat * M[d] + cell[d]
    order = torch.argsort(flat)
    start = torch.zeros(math.prod(M) + 1, device=DEV, dtype=torch.int64)
    start[1:] = torch.bincount(flat, minlength=math.prod(M)).cumsum(0)
    steps = [(0,) if m == 1 else (0, 1) if m == 2 and b == PER else (-1, 0, 1) for m, b in zip(M, bc)]
    offsets = [()]
    for d in range(dim):
        offsets = [o + (q,) for o in offsets for q in steps[d]]
    best = torch.full((n,), -1, device=DEV, dtype=torch.int64)
    spans = []   # every particle's candidate ranges, sorted order
    for o in offsets:
        key, ok = torch.zeros(n, device=DEV, dtype=torch.int64), torch.ones(n, device=DEV, dtype=torch.bool)
        for d in range(dim):
            q = cell[d][order] + o[d]
            if bc[d] == PER:
                q = q % M[d]
            ok &= (q >= 0) & (q < M[d])
            key = key * M[d] + q.clamp(0, M[d] - 1)
        a = start[key]
        spans.append((a, torch.where(ok, start[key + 1] - a, 0)))
    total = sum(s[1] for s in spans).cumsum(0)
    ps, vs = pos[order], vel[order]
    lo = 0
    while lo < n:
        done = int(total[lo - 1]) if lo else 0
        up = max(lo + 1, int(torch.searchsorted(total, done + CHUNK)))
        found = []
        for a, m in spans:
            a, m = a[lo:up], m[lo:up]
            k = int(m.sum())
            if not k:
                continue
            i = torch.repeat_interleave(torch.arange(up - lo, device=DEV), m, output_size=k)
            j = torch.arange(k, device=DEV) - (m.cumsum(0) - m)[i] + a[i]
            dr, dv = [], []
            for d in range(dim):
                x = ps[lo:up, d][i] - ps[j, d]
                if bc[d] == PER:
                    L, half = torch.tensor(hi[d], dtype=T, device=DEV), 0.5 * hi[d]
                    x = torch.where(x > half, x - L, torch.where(x < -half, x + L, x))
                dr.append(x)
                dv.append(vs[lo:up, d][i] - vs[j, d])
            r_v, v_v = _dot(dr, dv), _dot(dv, dv)
            t = ((v_v > 0) & (r_v < 0) & (_fma(v_v, dt, r_v) > 0)).nonzero()[:, 0]
            dr, r_v, v_v = [q[t] for q in dr], r_v[t], v_v[t]
            r_r = _dot(dr, dr)
            d2 = r_r - r_v * r_v / v_v
            ok = _fma(r_v, r_v, -(v_v * (r_r - R2))) >= 0
            found.append((i[t][ok], order[j[t][ok]], d2[ok]))
        if found:
            i, j, d2 = (torch.cat(q) for q in zip(*found))
            least = torch.full((up - lo,), math.inf, device=DEV, dtype=T).scatter_reduce_(0, i, d2, "amin")
            tie = d2 == least[i]
            who = torch.full((up - lo,), n, device=DEV, dtype=torch.int64).scatter_reduce_(0, i[tie], j[tie], "amin")
            best[order[lo:up]] = torch.where(who < n, who, -1)
        lo = up
    return best
