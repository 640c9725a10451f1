"""The library's work as its users have it done, as cases that can be timed.

A case is a dict of plain values.  `kind` says which entry points a pass goes
through; every array is on the device and every call is the public binding's.

  run       a segment of a simulation: the compressed store restored from its
            checkpoint, `steps` PM steps (uniform, or each cut by
            cube_next_epoch as the ensembles and the server cut them), the
            particles decoded
  batch     the same for `members` simulations of one geometry, one launch
            per kernel for all of them
  raw       the uncompressed FP32 store of the precision study: particles in,
            `steps` PM steps, particles out
  encode    the initial-condition generator's two passes: float particles to
            the compressed store, written out as a checkpoint
  decode    the store read out as float particles
  field     the density and the potential of the store as plain meshes
  spectrum  the power spectrum of the store

Sizes: `n` particles per side on a mesh of `mesh` fine cells per side, in a
box of `box` Mpc/h.  `disp` is the particles' rms displacement per axis from
their lattice in fine cells (0.27 at z = 49 for the 256^3 workload), `clump`
the fraction of particles that sit in haloes (late epochs).
"""
import math

import numpy as np
import torch

import paper_1712_06121_gb300 as cube

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def _case(name, kind, n, mesh, **over):
    c = {"name": name, "kind": kind, "n": n, "mesh": mesh, "ratio": 4, "xb": 1, "vb": 1, "idb": 4, "deconv": 2,
         "box": 300.0 * n / 256, "om": 0.3, "ol": 0.7, "a0": 0.02, "da": 0.0196, "steps": 0, "adaptive": False,
         "disp": 0.27, "clump": 0.0, "members": 1, "bins": 0, "order": "lattice"}
    c.update(over)
    return c


def listed():
    return [
        # the smallest member of an uneven ensemble, stepped alone: every
        # step's epoch comes from its particles, so latency and launches count
        _case("run 32^3 adaptive", "run", 32, 64, box=80.0, steps=6, adaptive=True),
        # the 64^3 Einstein-de Sitter workload (x1v2), uniform steps
        _case("run 64^3 x1v2", "run", 64, 128, vb=2, box=100.0, om=1.0, ol=0.0, da=0.008, steps=5),
        # an ensemble's members of one size, batched
        _case("batch 12 x 64^3", "batch", 64, 128, steps=5, adaptive=True, members=12),
        # an ordinary simulation: the largest size of the ensembles
        _case("run 128^3", "run", 128, 256, box=300.0, steps=5),
        # the flagship workload: 256^3 particles on a 512^3 mesh, early epochs
        _case("run 256^3", "run", 256, 512, steps=3),
        # the same resolution late: haloes, crowded bricks, adaptive steps
        # (192^3 is a size of the serving stream)
        _case("run 192^3 late", "run", 192, 384, steps=3, adaptive=True, a0=0.6, da=0.0098, disp=3.0,
              clump=0.25),
        # the precision study's 2-byte codes, a ragged particle count
        _case("run 101^3 x2v2", "run", 101, 192, xb=2, vb=2, steps=4, adaptive=True, a0=0.4, da=0.0098,
              disp=2.0, clump=0.1),
        # the precision study's uncompressed arm
        _case("raw 128^3", "raw", 128, 256, xb=4, vb=4, steps=3),
        # initial conditions of the flagship workload into the store
        _case("encode 256^3", "encode", 256, 512),
        # a snapshot of the flagship workload read out
        _case("decode 256^3", "decode", 256, 512),
        # density and potential meshes for analysis
        _case("field 192^3", "field", 192, 384),
        # the flagship's measurement: P(k) up to the mesh's Nyquist wave number
        _case("spectrum 256^3", "spectrum", 256, 512, bins=256),
    ]


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["run", "run", "run", "run", "batch", "raw", "encode", "decode", "field", "spectrum"])
    meshes = [32, 48, 64, 96, 128, 192, 256, 384, 512]
    if kind == "batch":
        meshes = [32, 48, 64, 96, 128]
    elif kind in ("run", "raw"):
        meshes = [32, 48, 64, 96, 128, 192, 256, 384]
    mesh = rng.choice(meshes)
    n = rng.randint(max(8, (3 * mesh) // 8), mesh // 2)              # particles per side, odd ones too
    xb, vb = (4, 4) if kind == "raw" else (rng.choice([1, 1, 2]), rng.choice([1, 1, 2]))
    late = kind != "raw" and rng.random() < 0.4
    eds = rng.random() < 0.25
    c = _case("", kind, n, mesh, xb=xb, vb=vb, ratio=rng.choice([2, 4, 4, 4, 8]),
              idb=rng.choice([0, 4]) if kind == "raw" else rng.choice([0, 1, 2, 4, 4, 4]), deconv=rng.choice([0, 1, 2, 2]),
              om=1.0 if eds else 0.3, ol=0.0 if eds else 0.7, box=round(rng.uniform(1.0, 4.0) * n, 3))
    if late:
        c.update(a0=round(rng.uniform(0.3, 0.9), 4), disp=round(rng.uniform(0.8, 3.5), 3),
                 clump=round(rng.uniform(0.05, 0.3), 3), ratio=max(4, c["ratio"]))
    else:
        c.update(a0=round(rng.uniform(0.02, 0.04), 4), disp=round(rng.uniform(0.15, 0.4), 3))
    if kind in ("run", "batch", "raw"):
        c.update(steps=rng.randint(2, 4), da=round(rng.uniform(0.002, 0.006), 5), adaptive=kind != "raw")
    if kind == "batch":
        c.update(members=rng.randint(2, 12))
    if kind == "spectrum":
        c.update(bins=rng.randint(mesh // 4, mesh // 2))
    if kind in ("encode", "decode"):
        c.update(order=rng.choice(["lattice", "shuffled"]))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _E(c, a):
    return math.sqrt(c["om"] / a ** 3 + (1.0 - c["om"] - c["ol"]) / a ** 2 + c["ol"])


def _particles(c, seed):
    """Zel'dovich particles with a cold-dark-matter spectrum, haloes mixed in
    for late epochs: positions in fine cells, momenta in fine cells x H0."""
    n, N = c["n"], c["mesh"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    noise = torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device=DEV))
    f = torch.fft.fftfreq(n, 1.0 / n, device=DEV)
    fx = torch.arange(n // 2 + 1, device=DEV, dtype=torch.float32)
    kz, ky, kx = f[:, None, None], f[None, :, None], fx[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    k2[0, 0, 0] = 1.0
    k = torch.sqrt(k2) * (2.0 * math.pi / c["box"])                    # h/Mpc
    q = k / (0.3 * 0.7)
    tf = torch.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3
                                               + (6.71 * q) ** 4) ** -0.25
    amp = torch.sqrt(k ** 0.96) * tf / k2
    if c["disp"] > 0.5:                                                # late: streams already mixed on small scales
        amp = amp * torch.exp(-0.5 * k2 * (2.0 * math.pi * c["disp"] / N) ** 2)
    noise *= amp
    noise[0, 0, 0] = 0.0
    psi = torch.stack([torch.fft.irfftn(1j * g * noise, s=(n, n, n)).reshape(-1) for g in (kx, ky, kz)])
    psi *= c["disp"] / psi.square().mean().sqrt()
    site = torch.arange(n, device=DEV, dtype=torch.float32) * (N / n) + 0.5
    x = psi.clone()
    x[0] += site.repeat(n * n)
    x[1] += site.repeat_interleave(n).repeat(n)
    x[2] += site.repeat_interleave(n * n)
    a, om = c["a0"], c["om"]
    growth = (om / a ** 3 / _E(c, a) ** 2) ** 0.55
    p = psi * (a * a * _E(c, a) * growth)
    if c["clump"] > 0.0:
        m = n ** 3
        pick = torch.nonzero(torch.rand(m, generator=gen, device=DEV) < c["clump"]).reshape(-1)
        halos = max(1, m // 4096)
        centre = torch.randint(0, m, (halos,), generator=gen, device=DEV)
        u = torch.rand(pick.numel(), generator=gen, device=DEV)
        host = centre[(halos * u ** 1.3).long().clamp_(max=halos - 1)]
        r = 8.0 * torch.rand(pick.numel(), generator=gen, device=DEV)      # isothermal: rho ~ r^-2
        way = torch.randn((3, pick.numel()), generator=gen, device=DEV)
        x[:, pick] = x[:, host] + r * way / way.norm(dim=0).clamp_(min=1e-6)
        hot = 0.6 * p.square().mean().sqrt()
        p[:, pick] = p[:, host] + hot * torch.randn((3, pick.numel()), generator=gen, device=DEV)
    x = torch.remainder(x, float(N))
    x[x >= float(N)] = 0.0
    ids = torch.arange(n ** 3, device=DEV, dtype=torch.int32)
    if c["order"] == "shuffled":
        s = torch.randperm(n ** 3, generator=gen, device=DEV)
        x, p, ids = x[:, s], p[:, s], ids[s]
    return x.contiguous(), p.contiguous(), ids


def _params(c):
    return cube.make_params(c["mesh"], c["n"] ** 3, ratio=c["ratio"], x_bytes=c["xb"], v_bytes=c["vb"],
                            id_bytes=c["idb"], deconv_power=c["deconv"], box=c["box"], omega_m=c["om"],
                            omega_l=c["ol"])


class _State:
    """A user's handles and buffers; the handles go with it."""

    def __init__(self, c):
        self.c, self.ctx, self.batch = c, None, None

    def outputs(self):
        n3, c = self.c["n"] ** 3, self.c
        return (torch.zeros((3, n3), device=DEV), torch.zeros((3, n3), device=DEV),
                torch.zeros(n3, device=DEV, dtype=torch.int32) if c["idb"] else None)

    def __del__(self):
        if self.batch is not None:
            cube.cube_batch_destroy(self.batch)
        elif self.ctx is not None:
            cube.cube_destroy(self.ctx)


def _checkpoint(c, ctx, x, p, ids, prm):
    """The store of these particles as its checkpoint."""
    cube.cube_encode(ctx, x, p, ids, c["a0"], 0.0)
    buf = torch.zeros(cube.cube_checkpoint_size(prm), device=DEV, dtype=torch.uint8)
    cube.cube_checkpoint_save(ctx, buf)
    return buf


def prepare(case, seed):
    c = dict(case)
    s = _State(c)
    stream = torch.cuda.current_stream()
    prm = _params(c)
    if c["kind"] == "batch":
        s.batch = cube.cube_batch_create([prm] * c["members"], stream)
        s.members = [cube.cube_batch_member(s.batch, i) for i in range(c["members"])]
        s.saved = []
        for i, m in enumerate(s.members):
            x, p, ids = _particles(c, seed * 64 + i)
            s.saved.append(_checkpoint(c, m, x, p, ids, prm))
        s.out = [s.outputs() for _ in s.members]
        return s
    x, p, ids = _particles(c, seed)
    s.ctx = cube.cube_create(prm, stream)
    if c["kind"] == "run":
        s.saved = _checkpoint(c, s.ctx, x, p, ids, prm)
        s.out = s.outputs()
    elif c["kind"] in ("encode", "raw"):
        s.x, s.p, s.ids = x, p, ids
        if c["kind"] == "raw":
            s.out = s.outputs()
        else:
            s.saved = _checkpoint(c, s.ctx, x, p, ids, prm)
    else:
        cube.cube_encode(s.ctx, x, p, ids, c["a0"], 0.0)
        if c["kind"] == "decode":
            s.out = s.outputs()
        elif c["kind"] == "field":
            N = c["mesh"]
            s.out = (torch.zeros((N, N, N), device=DEV), torch.zeros((N, N, N), device=DEV))
        else:
            s.out = tuple(torch.zeros(c["bins"], device=DEV, dtype=torch.float64) for _ in range(3))
    return s


# ---------------------------------------------------------------- a pass
def run(s):
    c = s.c
    if c["kind"] == "run":
        cube.cube_checkpoint_load(s.ctx, s.saved)
        a = c["a0"]
        for _ in range(c["steps"]):
            to = cube.cube_next_epoch(s.ctx, a + c["da"], 0.5) if c["adaptive"] else a + c["da"]
            cube.cube_pm_step(s.ctx, a, to)
            a = to
        cube.cube_decode(s.ctx, *s.out)
        return s.out
    if c["kind"] == "batch":
        for m, b in zip(s.members, s.saved):
            cube.cube_checkpoint_load(m, b)
        a = np.full(c["members"], c["a0"])
        for _ in range(c["steps"]):
            to = cube.cube_batch_next_epochs(s.batch, a + c["da"], 0.5)
            cube.cube_batch_step(s.batch, a, to)
            a = to
        for m, o in zip(s.members, s.out):
            cube.cube_decode(m, *o)
        return s.out
    if c["kind"] == "raw":
        cube.cube_encode(s.ctx, s.x, s.p, s.ids, c["a0"], 0.0)
        a = c["a0"]
        for _ in range(c["steps"]):
            cube.cube_pm_step(s.ctx, a, a + c["da"])
            a += c["da"]
        cube.cube_decode(s.ctx, *s.out)
        return _displacement(s.out[0], s.x, c["mesh"]), s.out[1], s.out[2]
    if c["kind"] == "encode":
        cube.cube_encode(s.ctx, s.x, s.p, s.ids, c["a0"], 0.0)
        cube.cube_checkpoint_save(s.ctx, s.saved)
        return s.saved
    if c["kind"] == "decode":
        cube.cube_decode(s.ctx, *s.out)
        return s.out
    if c["kind"] == "field":
        cube.cube_density(s.ctx, s.out[0])
        cube.cube_potential(s.ctx, s.out[1])
        return s.out
    cube.cube_power_spectrum(s.ctx, c["bins"], *s.out)
    return s.out


def _displacement(x, x0, N):
    """How far the particles have moved: periodic positions as a study compares them."""
    d = x - x0
    return d - N * torch.round(d / N)


# ---------------------------------------------------------------- the least a pass can do
def work(case):
    c = dict(case)
    np_, nm = float(c["n"]) ** 3, float(c["mesh"]) ** 3
    ncc = (c["mesh"] // c["ratio"]) ** 3
    store = (3 * c["xb"] + 3 * c["vb"] + c["idb"]) * np_ + (16 * ncc if c["kind"] != "raw" else 0)
    floats = (24 + (4 if c["idb"] else 0)) * np_
    fft = 2.5 * nm * math.log2(nm)
    if c["kind"] in ("run", "batch", "raw"):
        # a step: the store read and written, and the mesh, larger than the
        # chip's own memory, written and read between the axes of the transforms
        step = 2 * store + 32 * nm
        per = (300.0 * np_ + 2 * fft) * c["steps"]
        first = floats if c["kind"] == "raw" else store
        return {"bytes": c["members"] * (first + c["steps"] * step + floats), "flops": c["members"] * per}
    if c["kind"] == "encode":
        return {"bytes": floats + store, "flops": 60.0 * np_}
    if c["kind"] == "decode":
        return {"bytes": floats + store, "flops": 20.0 * np_}
    if c["kind"] == "field":
        return {"bytes": store + 8 * nm + 24 * nm, "flops": 2 * fft + 60.0 * np_}
    return {"bytes": store + 12 * nm + 24.0 * c["bins"], "flops": fft + 60.0 * np_ + 5 * nm}


# ---------------------------------------------------------------- the same in 64 bits
def _coded(c, x):
    """Positions as the store holds them: the middle of their code's bin."""
    if c["xb"] == 4:
        return x.double()
    scale = 2.0 ** (8 * c["xb"]) / c["ratio"]
    return (torch.floor(x.double() * scale) + 0.5) / scale


def _density(c, x):
    N = c["mesh"]
    rho = torch.zeros(N ** 3, device=DEV, dtype=torch.float64)
    i = torch.floor(x)
    w = x - i
    i = i.long() % N
    for corner in range(8):
        d = [(corner >> b) & 1 for b in range(3)]
        at = ((i[2] + d[2]) % N * N + (i[1] + d[1]) % N) * N + (i[0] + d[0]) % N
        ws = [w[b] if d[b] else 1.0 - w[b] for b in range(3)]
        rho.index_add_(0, at, ws[0] * ws[1] * ws[2])
    return (rho * (N ** 3 / x.shape[1])).reshape(N, N, N)


def _axis(N):
    """Signed integer frequency of each index (N / 2 positive) and sinc(pi f / N)."""
    f = torch.arange(N, device=DEV, dtype=torch.float64)
    f = torch.where(f <= N // 2, f, f - N)
    return f, torch.sinc(f / N)


def _potential(c, rho):
    N = c["mesh"]
    f, w = _axis(N)
    h = N // 2 + 1
    k2 = (2.0 * math.pi * f / N) ** 2
    wd = w ** (-2.0 * c["deconv"])
    rk = torch.fft.rfftn(rho)
    kk = k2[:, None, None] + k2[None, :, None] + k2[None, None, :h]
    kk[0, 0, 0] = 1.0
    rk *= -1.5 * c["om"] / kk * (wd[:, None, None] * wd[None, :, None] * wd[None, None, :h])
    rk[0, 0, 0] = 0.0
    return torch.fft.irfftn(rk, s=(N, N, N))


def _force(phi, x):
    """-grad Phi by 4th-order differences at the nodes, interpolated with CIC weights."""
    N = phi.shape[0]
    i = torch.floor(x)
    w = x - i
    i = i.long() % N
    out = []
    for axis in (2, 1, 0):
        g = (8.0 * (torch.roll(phi, -1, axis) - torch.roll(phi, 1, axis))
             - (torch.roll(phi, -2, axis) - torch.roll(phi, 2, axis))).reshape(-1) / -12.0
        acc = torch.zeros_like(x[0])
        for corner in range(8):
            d = [(corner >> b) & 1 for b in range(3)]
            at = ((i[2] + d[2]) % N * N + (i[1] + d[1]) % N) * N + (i[0] + d[0]) % N
            ws = [w[b] if d[b] else 1.0 - w[b] for b in range(3)]
            acc += ws[0] * ws[1] * ws[2] * g[at]
        out.append(acc)
    return torch.stack(out)


def _integral(fn, a0, a1):
    t, w = np.polynomial.legendre.leggauss(64)
    a = 0.5 * (a0 + a1) + 0.5 * (a1 - a0) * t
    return float(sum(wi * fn(ai) for wi, ai in zip(w, a)) * 0.5 * (a1 - a0))


def _brick(c):
    """The storage brick's side: the largest of 4, 2, 1 that fits the geometry."""
    nc = c["mesh"] // c["ratio"]
    return next(b for b in (4, 2, 1) if nc % b == 0 and nc // b >= 3 and 4 <= b * c["ratio"] <= 16)


def _decoded(c, x, p, ids):
    """The store's particles in its order: bricks, cells and codes from their definitions."""
    nc, b, xd = c["mesh"] // c["ratio"], _brick(c), _coded(c, x)
    cell = torch.floor(xd / c["ratio"]).long()
    home, l = cell // b, cell % b
    nb = nc // b
    rank = ((home[2] * nb + home[1]) * nb + home[0]) * b ** 3 + (l[2] * b + l[1]) * b + l[0]
    order = torch.sort(rank, stable=True).indices
    count = torch.bincount(rank, minlength=nc ** 3).clamp_(min=1)
    vc = []
    for d in range(3):
        fixed = torch.round(p[d].double() * 2.0 ** 24).long()
        vc.append((torch.zeros(nc ** 3, device=DEV, dtype=torch.int64).index_add_(0, rank, fixed).double()
                   / count / 2.0 ** 24).float())
    vc = torch.stack(vc)[:, rank]
    off = (p - vc).double()
    sigma = 2.0 ** (math.floor(16.0 * math.log2(float(off.square().mean().sqrt())) + 0.5) / 16.0)
    m = 2 ** (8 * c["vb"]) - 1
    nu = m / math.pi * torch.atan(off * math.sqrt(math.pi / (2.0 * sigma ** 2)))
    nu = (torch.sign(nu) * torch.floor(nu.abs() + 0.5)).clamp_(-(m // 2), m // 2)
    v = vc.double() + torch.tan(math.pi * nu / m) * math.sqrt(2.0 * sigma ** 2 / math.pi)
    return xd[:, order], v[:, order]


def exact(case, seed):
    c = dict(case)
    if c["kind"] in ("run", "batch", "encode"):       # whole numbers, or particles that such numbers steer
        return None
    x, p, ids = _particles(c, seed)
    if c["kind"] == "decode":
        return (*_decoded(c, x, p, ids), None)
    if c["kind"] == "raw":
        a, ap, q, v = c["a0"], c["a0"], x.double(), p.double()
        for _ in range(c["steps"]):
            b = a + c["da"]
            mid = 0.5 * (a + b)
            g = _force(_potential(c, _density(c, q)), q)
            v = v + g * _integral(lambda t: 1.0 / (t * t * _E(c, t)), ap, mid)
            q = q + v * _integral(lambda t: 1.0 / (t ** 3 * _E(c, t)), a, b)
            a, ap = b, mid
        return q - x.double(), v, None
    rho = _density(c, _coded(c, x))
    if c["kind"] == "field":
        return rho, _potential(c, rho)
    N, h = c["mesh"], c["mesh"] // 2 + 1
    f, w = _axis(N)
    rk = torch.fft.rfftn(rho - 1.0)
    power = (rk.real ** 2 + rk.imag ** 2) * (c["box"] ** 3 / float(N) ** 6)
    del rk
    w4 = w ** -4.0
    power *= w4[:, None, None] * w4[None, :, None] * w4[None, None, :h]
    weight = torch.full((h,), 2.0, device=DEV, dtype=torch.float64)
    weight[0] = weight[-1] = 1.0
    nmax = c["bins"]
    edge = torch.arange(1, nmax + 2, device=DEV, dtype=torch.float64) - 0.5
    out = torch.zeros((3, nmax), device=DEV, dtype=torch.float64)
    for z in range(N):                                     # a plane at a time
        n2 = f[z] ** 2 + f[:, None] ** 2 + f[None, :h] ** 2
        i = torch.bucketize(n2.reshape(-1), edge ** 2, right=True) - 1
        ok = (i >= 0) & (i < nmax)
        i, ww = i[ok], weight.expand(N, h).reshape(-1)[ok]
        out[2].index_add_(0, i, ww)
        out[0].index_add_(0, i, ww * torch.sqrt(n2.reshape(-1)[ok]) * (2.0 * math.pi / c["box"]))
        out[1].index_add_(0, i, ww * power[z].reshape(-1)[ok])
    out[:2] /= out[2]
    return tuple(out)
