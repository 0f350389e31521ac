"""The work that users of the library have it do, as cases that can be timed and compared.

A case is a dict of plain values with a "form":

  run       a lattice advanced by `steps` steps, then its fields (rlbm_step, rlbm_moments);
  sample    one sample of a long run: `steps` steps, the spectrum and the filtered
            velocity (the body of analysis.sample_run), with `fields` set also the fields;
  channel   the current density of an open channel, recorded every step
            (analysis.current_density_run);
  ensemble  lattices of uneven sizes advanced together (rlbm.Batch), then their fields;
  gradient  the gradient of the time-averaged kinetic energy (adjoint.kinetic_energy and
            backward, or rlbm.Lattice.gradient).

Outputs are in the precision of the lattice's storage: the library hands every field out
as doubles, but those of a 32-bit or 16-bit lattice are worth 32 or 16 bits, and a program
that keeps them keeps them so.  BF16 storage is offered for comparison only and has no
case.  `exact` is the same run in 64 bits in plain torch.
"""
import math

import numpy as np
import torch

from paper_2205_04658_gb300 import adjoint, analysis, inputs, rlbm

# Keys that every lattice case has: nx, ny, precision, walls (bounce-back at y = -1 and ny),
# discs (area fraction of impurities of radius 6), stir (shell "kmin-kmax" or ""), amp, eta,
# body (force along x), flow (mean u^x at the start), u (size of the start's fluctuations).
LATTICE = dict(precision="f32", vset=3, walls=False, discs=0.0, stir="", amp=0.0, eta=0.05, body=0.0, flow=0.0, u=3e-3)


def _case(form, **kw):
    return dict(LATTICE, form=form, **kw)


def listed():
    return [
        # the decaying shear wave that the method is checked with: smallest lattice, 64 bits
        dict(_case("run", nx=64, ny=64, precision="f64", eta=0.1, u=0.01, steps=200), name="decay_64_f64"),
        # the same physics on the two-dimensional velocity set, 32 bits
        dict(_case("run", nx=256, ny=256, vset=2, eta=0.1, u=0.01, steps=100), name="decay_256_vset2"),
        # one sample of a stirred run at the paper's smallest size: launches and latency count
        dict(_case("sample", nx=128, ny=128, stir="8-10", amp=1e-4, steps=18, nbins=64, fields=False), name="sample_128"),
        # the same at 512^2
        dict(_case("sample", nx=512, ny=512, stir="8-10", amp=1e-4, steps=18, nbins=256, fields=False), name="sample_512"),
        # sizes that are no multiple of anything
        dict(_case("run", nx=397, ny=251, stir="4-6", amp=1e-4, steps=100), name="stirred_397x251"),
        # the stirred workload as it runs: blocks of steps with a spectrum and the fields after each
        dict(_case("sample", nx=1024, ny=1024, stir="8-10", amp=1e-4, steps=100, nbins=512, fields=True), name="stirred_1024"),
        # the largest stirred lattice of the benchmark
        dict(_case("run", nx=4096, ny=4096, stir="8-10", amp=1e-4, steps=100), name="stirred_4096"),
        # the graphene-like sample between walls, 16-bit storage
        dict(_case("run", nx=2048, ny=512, precision="f16", walls=True, discs=0.15, body=1e-6, flow=2e-3, u=1e-4, steps=200),
             name="graphene_2048x512_f16"),
        # the open channel with one impurity, observed after every step
        dict(_case("channel", nx=1024, ny=256, impurities=1, eta=0.1, flow=0.1, u=1e-3, steps=20), name="channel_1024x256"),
        # an ensemble of stirred realisations of uneven sizes, 16-bit storage
        dict(_case("ensemble", sizes="256,512,768,1024,256,512,768,1024,512,512,768,256,1024,256,768,512", precision="f16",
                   stir="8-10", amp=1e-4, steps=100), name="ensemble_16_f16"),
        # the gradient of a stirred run, checkpointed every sqrt(steps)
        dict(_case("gradient", nx=512, ny=512, stir="4-6", amp=1e-4, eta=0.1, body=1e-6, flow=2e-3, u=0.01, steps=200, autograd=False),
             name="gradient_512"),
        # a small gradient in 64 bits through autograd
        dict(_case("gradient", nx=64, ny=48, precision="f64", stir="4-6", amp=1e-3, eta=0.1, body=1e-6, flow=2e-3, u=0.01, steps=50, autograd=True),
             name="gradient_64x48_f64"),
    ]


def draw(rng):
    def size(lo, hi):  # spread over the logarithm; a third are multiples of 32
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, n // 32 * 32) if rng.random() < 1 / 3 else n

    shell = lambda: rng.choice(["2-4", "4-6", "8-10", "6-12"])  # noqa: E731
    form = rng.choice(["run", "run", "run", "sample", "sample", "channel", "ensemble", "gradient"])
    if form == "run":
        nx, ny = size(32, 3000), size(32, 3000)
        most = 1.5e9 / (nx * ny)  # cell updates of a pass
        precision = rng.choice(["f32", "f32", "f32", "f16", "f64"])
        kw = dict(nx=nx, ny=ny, precision=precision, steps=max(10, min(size(20, 120), int(most / (12 if precision == "f64" else 1)))),
                  eta=rng.choice([0.05, 0.1]))
        kind = rng.choice(["stirred", "stirred", "sample", "decay"])
        if kind == "stirred":
            kw.update(stir=shell(), amp=1e-4)
        elif kind == "sample":
            kw.update(walls=True, discs=rng.choice([0.01, 0.05, 0.15]), body=1e-6, flow=2e-3, u=1e-4)
        else:
            kw.update(u=0.01, vset=rng.choice([2, 3]))
        return _case("run", **kw)
    if form == "sample":
        n = rng.choice([64, 128, 192, 256, 384, 512, 640, 1024, 1536])
        return _case("sample", nx=n, ny=n, stir=shell(), amp=1e-4, steps=rng.choice([9, 18, 36, 100]), nbins=n // 2, fields=False,
                     precision=rng.choice(["f32", "f32", "f16"]))
    if form == "channel":
        return _case("channel", nx=size(200, 1500), ny=size(160, 400), impurities=1, eta=rng.choice([0.05, 0.1]),
                     flow=0.1, u=1e-3, steps=rng.randint(5, 30))
    if form == "ensemble":
        sizes = ",".join(str(size(48, 1024)) for _ in range(rng.randint(3, 20)))
        return _case("ensemble", sizes=sizes, precision=rng.choice(["f32", "f16"]), stir=shell(), amp=1e-4, steps=rng.randint(20, 100))
    precision = rng.choice(["f32", "f32", "f64"])
    n = 128 if precision == "f64" else 640
    return _case("gradient", nx=size(32, n), ny=size(32, n), precision=precision, stir=rng.choice(["2-4", "4-6"]), amp=1e-4,
                 eta=0.1, body=1e-6, flow=2e-3, u=0.01, steps=rng.randint(20, 60 if precision == "f64" else 200), autograd=rng.random() < 0.5)


# ----- inputs ------------------------------------------------------------------------
A, DT = 0.1, 0.05   # lattice spacing and time step of every workload
RADIUS = 6
STORE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}


def _shell(case):
    return tuple(int(v) for v in case["stir"].split("-")) if case["stir"] else (0, 0)


def _mask(case, nx, ny, rng):
    """Solid cells: discs of radius 6 that do not touch, one at a random place of each
    square of a grid as coarse as the area fraction asks for; an impurity of the channel."""
    if case["form"] == "channel":
        return inputs.channel_impurities(nx, ny, 13, count=case["impurities"])
    if not case["discs"]:
        return None
    span = 2 * RADIUS + 1
    area = sum(1 for a in range(-RADIUS, RADIUS + 1) for b in range(-RADIUS, RADIUS + 1) if a * a + b * b <= RADIUS * RADIUS)
    cell = max(span + 2, int(round(math.sqrt(area / case["discs"]))))
    mask = np.zeros((ny, nx), np.uint8)
    cy, cx = np.meshgrid(np.arange(0, ny - cell + 1, cell), np.arange(0, nx - cell + 1, cell), indexing="ij")
    cx = cx + rng.integers(RADIUS + 1, cell - RADIUS, cx.shape)
    cy = cy + rng.integers(RADIUS + 1, cell - RADIUS, cy.shape)
    for a in range(-RADIUS, RADIUS + 1):
        for b in range(-RADIUS, RADIUS + 1):
            if a * a + b * b <= RADIUS * RADIUS:
                mask[cy + b, cx + a] = 1
    return mask


def _fields(case, nx, ny, gen):
    """eps, u^x, u^y: smooth random fields on wave numbers up to 4 about the mean flow."""
    k = torch.arange(-4, 5, dtype=torch.float64)
    ey = torch.exp(2j * math.pi * (torch.arange(ny)[:, None] * k[None, :] / ny)).cuda()
    ex = torch.exp(2j * math.pi * (k[:, None] * torch.arange(nx)[None, :] / nx)).cuda()
    out = []
    for _ in range(3):
        c = torch.randn(9, 9, 2, dtype=torch.float64, generator=gen)
        c[4, 4] = 0.0
        g = ((ey @ torch.view_as_complex(c).cuda()) @ ex).real
        out.append(g / g.abs().max())
    return 1.0 + 0.3 * case["u"] * out[0], case["flow"] + case["u"] * out[1], case["u"] * out[2]


def _inputs(case, nx, ny, seed):
    gen = torch.Generator().manual_seed(seed)
    rng = np.random.default_rng(seed)
    eps, ux, uy = _fields(case, nx, ny, gen)
    kmin, kmax = _shell(case)
    kw = dict(precision=case["precision"], vset=case["vset"], a=A, dt=DT, eta_over_s=case["eta"], walls_y=int(case["walls"]),
              body_force=(case["body"], 0.0), kmin=kmin, kmax=kmax, force_amp=case["amp"], seed=1 + seed,
              solid=_mask(case, nx, ny, rng), init_eps=eps.cpu().numpy(), init_ux=ux.cpu().numpy(), init_uy=uy.cpu().numpy())
    if case["form"] == "channel":
        kw.update(open_x=1, inflow_ux=case["flow"])
    return kw


def _sizes(case):
    return [int(s) for s in case["sizes"].split(",")] if case["form"] == "ensemble" else [(case["nx"], case["ny"])]


class _Fields:
    """Pinned host buffers of the fields of lattices, and the copy that is kept of them."""

    def __init__(self, shapes, precision):
        cells = sum(nx * ny for nx, ny in shapes)
        self.got = [torch.empty(cells, dtype=torch.float64, pin_memory=True) for _ in range(3)]
        self.totals = torch.empty(len(shapes), 4, dtype=torch.float64, pin_memory=True)
        self.kept = None if precision == "f64" else [torch.empty_like(t, dtype=STORE[precision], pin_memory=False) for t in self.got]
        self.at = []
        o = 0
        for i, (nx, ny) in enumerate(shapes):
            self.at.append([t[o:o + nx * ny].numpy() for t in self.got] + [self.totals[i].numpy()])
            o += nx * ny

    def take(self, lattices):
        for lat, to in zip(lattices, self.at):
            rlbm.rlbm_moments(lat.ctx, *to)
        if self.kept is None:
            return dict(eps=self.got[0], ux=self.got[1], uy=self.got[2], totals=self.totals)
        for t, k in zip(self.got, self.kept):
            k.copy_(t)
        return dict(eps=self.kept[0], ux=self.kept[1], uy=self.kept[2], totals=self.totals.float())


def prepare(case, seed):
    form, s = case["form"], dict(case=case)
    if form == "ensemble":
        stream = s["stream"] = torch.cuda.Stream()  # (a stream of its own lets the batch replay graphs)
        s["lattices"] = [rlbm.Lattice(n, n, stream=stream, **_inputs(case, n, n, seed * 64 + i)) for i, n in enumerate(_sizes(case))]
        s["batch"] = rlbm.Batch(s["lattices"], stream=stream)
        s["batch"].autotune(3)
        s["fields"] = _Fields([(n, n) for n in _sizes(case)], case["precision"])
        return s
    nx, ny = case["nx"], case["ny"]
    kw = _inputs(case, nx, ny, seed)
    if form == "gradient" and case["autograd"]:
        lat = rlbm.Lattice(nx, ny, **kw)
        n = lat.num_modes
        lat.close()
        s["spec"] = dict({k: v for k, v in kw.items() if k not in ("eta_over_s", "body_force")}, nx=nx, ny=ny, nsteps=case["steps"])
        s["sigma"] = torch.ones(n, dtype=torch.float64, requires_grad=True)
        s["eta"] = torch.tensor(kw["eta_over_s"], dtype=torch.float64, requires_grad=True)
        s["body"] = torch.tensor(kw["body_force"], dtype=torch.float64, requires_grad=True)
        return s
    lat = s["lattice"] = rlbm.Lattice(nx, ny, **kw)
    if form in ("run", "sample"):
        lat.autotune()
    if form == "run" or form == "sample" and case["fields"]:
        s["fields"] = _Fields([(nx, ny)], case["precision"])
    return s


# ----- one pass ----------------------------------------------------------------------
def run(s):
    case = s["case"]
    form, kind = case["form"], STORE[case["precision"]]
    if form == "run":
        s["lattice"].step(case["steps"])
        return s["fields"].take([s["lattice"]])
    if form == "sample":
        lat = s["lattice"]
        lat.step(case["steps"])
        kind = torch.float32  # (16-bit storage: spectra lie below the 16-bit range)
        out = dict(E=torch.from_numpy(lat.spectrum(case["nbins"])).to(kind),
                   velocity=torch.tensor(lat.filtered_velocity(_shell(case)[0]), dtype=torch.float64).to(kind))
        if case["fields"]:
            out.update(s["fields"].take([lat]))
        return out
    if form == "channel":
        r = analysis.current_density_run(s["lattice"], case["steps"])
        return dict(t=r["t_steps"], j_t=torch.from_numpy(r["j_t"]).to(kind), j_x=torch.from_numpy(r["j_x"]).to(kind))
    if form == "ensemble":
        s["batch"].step(case["steps"])
        return s["fields"].take(s["lattices"])
    if case["autograd"]:
        for t in (s["sigma"], s["eta"], s["body"]):
            t.grad = None
        J = adjoint.kinetic_energy(s["sigma"], s["eta"], s["body"], **s["spec"])
        J.backward()
        out = dict(J=J.detach(), sigma=s["sigma"].grad, eta=s["eta"].grad, body=s["body"].grad)
    else:
        J, gs, ge, gb = s["lattice"].gradient(case["steps"])
        out = dict(J=torch.tensor(J, dtype=torch.float64), sigma=torch.from_numpy(gs), eta=torch.tensor(ge, dtype=torch.float64),
                   body=torch.from_numpy(gb))
    # (d/d(eta/s) is what the equilibrium parts leave over of a sum some thousand times larger: a
    # 32-bit lattice gives three digits of it)
    return {k: v.to(torch.bfloat16 if k == "eta" and kind == torch.float32 else kind) for k, v in out.items()}


def work(case):
    """One pass: the state read and written once (each of the Q populations of a cell), the
    outputs written once, and the arithmetic of a cell update times cells and steps (about 670
    operations with the stirring force, 500 without; the reverse of a step about three times
    a step, with the step itself run twice)."""
    cells = sum(n * n for n in _sizes(case)) if case["form"] == "ensemble" else case["nx"] * case["ny"]
    width = {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
    planes = 17 if case["vset"] == 3 else 8
    per_cell = (670 if case["stir"] else 500) * planes / 17
    flops = per_cell * cells * case["steps"] * (5 if case["form"] == "gradient" else 1)
    out = 3 * width * cells if case["form"] in ("run", "ensemble") or case.get("fields") else 0
    return {"bytes": 2 * planes * width * cells + out, "flops": flops}


# ----- the same in 64 bits -------------------------------------------------------------
class _Exact:
    """The method in plain torch, FP64: pull streaming with bilinear weights, Landau matching
    by Newton's method, the projected equilibrium, Anderson-Witting relaxation and the
    projected force, on the momentum set's directions with v_z folded together."""

    def __init__(self, case, nx, ny, kw):
        d = "cuda"
        self.nx, self.ny, self.walls, self.open = nx, ny, bool(case["walls"]), case["form"] == "channel"
        dirs = {}
        if case["vset"] == 3:  # 26 unit vectors; degree-7 spherical rule
            for a in (-1, 0, 1):
                for b in (-1, 0, 1):
                    for c in (-1, 0, 1):
                        m = a * a + b * b + c * c
                        if m:
                            w = {1: 1 / 21, 2: 4 / 105, 3: 9 / 280}[m]
                            key = (a, b, m)
                            dirs[key] = (a / math.sqrt(m), b / math.sqrt(m), c * c / m, w + dirs.get(key, (0, 0, 0, 0))[3])
            self.dp, self.CA, self.CB, self.CC, self.tau, self.root = 3, 4.0, 10.0, 2.0, 5.0, 0.25
            self.T0 = (math.pi ** 2 / 3) ** 0.25
        else:
            for i in range(8):
                c, s_ = round(math.cos(i * math.pi / 4), 15), round(math.sin(i * math.pi / 4), 15)
                if i % 2:
                    c, s_ = math.copysign(math.sqrt(0.5), c), math.copysign(math.sqrt(0.5), s_)
                dirs[(int(math.copysign(1, c)) if c else 0, int(math.copysign(1, s_)) if s_ else 0, i)] = (c, s_, 0.0, 0.125)
            self.dp, self.CA, self.CB, self.CC, self.tau, self.root = 2, 3.0, 6.0, 1.5, 4.0, 1 / 3
            self.T0 = math.pi ** (1 / 3)
        self.signs = [k[:2] for k in dirs]
        v = list(dirs.values())
        self.opp = [min(range(len(v)), key=lambda p: abs(v[p][0] + v[q][0]) + abs(v[p][1] + v[q][1]) + abs(v[p][2] - v[q][2])) for q in range(len(v))]
        vx, vy, vz2, w = (torch.tensor(c, dtype=torch.float64, device=d) for c in zip(*v))
        self.w = w
        self.mom = torch.stack([w, w * vx, w * vy, w * vx * vx, w * vx * vy, w * vy * vy, w * vx ** 3, w * vx * vx * vy, w * vx * vy * vy, w * vy ** 3])
        one = torch.ones_like(vx)
        self.rel = torch.stack([one, vx, vy], 1)
        self.basis = torch.stack([one, vx, vy, vx * vx, vx * vy, vy * vy, vx ** 3, vx * vx * vy, vx * vy * vy, vy ** 3, vz2], 1)
        solid = None if kw["solid"] is None else torch.from_numpy(np.asarray(kw["solid"])).to(d) != 0
        self.fluid = None if solid is None else ~solid
        self.blocked = None
        if solid is not None or self.walls:
            s_ = solid if solid is not None else torch.zeros(ny, nx, dtype=torch.bool, device=d)
            s_ = torch.cat([s_[-1:], s_, s_[:1]]) if not self.walls else torch.nn.functional.pad(s_, (0, 0, 1, 1), value=True)
            self.blocked = torch.nn.functional.pad(s_, (1, 1), value=False) if self.open else torch.cat([s_[:, -1:], s_, s_[:, :1]], 1)
        C = DT / A
        self.beta = [((1 - C * abs(x)) * (1 - C * abs(y)), C * abs(x) * (1 - C * abs(y)), (1 - C * abs(x)) * C * abs(y), C * C * abs(x * y))
                     for x, y in zip(vx.tolist(), vy.tolist())]
        self.inflow = None
        if self.open:
            u = kw["inflow_ux"]
            self.inflow = self.CA * math.sqrt(1 + u * u) * u * vx + self.CB * (u * vx) ** 2 - self.CC * u * u
        self.eta = torch.tensor(kw["eta_over_s"], dtype=torch.float64, device=d)
        self.body = torch.tensor(kw["body_force"], dtype=torch.float64, device=d)
        self.force_on = case["vset"] == 3 and (bool(case["stir"]) or case["body"] != 0 or case["form"] == "gradient")
        if case["stir"]:
            self._stirring(case, kw["seed"])
        self.sigma = torch.ones(len(self.kx), dtype=torch.float64, device=d) if case["stir"] else None
        e, ux, uy = (torch.from_numpy(kw[k]).to(d) for k in ("init_eps", "init_ux", "init_uy"))
        u2 = ux * ux + uy * uy
        uv = vx[:, None, None] * ux + vy[:, None, None] * uy
        self.h = (e - 1) + self.CA * e * torch.sqrt(1 + u2) * uv + self.CB * e * uv * uv - self.CC * e * u2
        if solid is not None:
            self.h[:, solid] = 0.0
        self.step = 0

    # Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) keyed by the seed, counter (step, mode)
    def _stirring(self, case, seed):
        kmin, kmax = _shell(case)
        self.amp, self.seed = case["amp"], seed
        k = [(x, y) for y in range(kmax + 1) for x in range(-kmax, kmax + 1)
             if (y > 0 or x > 0) and kmin * kmin <= x * x + y * y <= kmax * kmax]
        self.kx, self.ky = np.array([v[0] for v in k]), np.array([v[1] for v in k])
        ph = lambda kk, n: torch.from_numpy(np.exp(2j * np.pi * (np.outer(kk, np.arange(n)) % n) / n)).cuda()  # noqa: E731
        self.ex, self.ey = ph(self.kx, self.nx), ph(self.ky, self.ny)

    def _draws(self, n):
        m = len(self.kx)
        M, mask = [np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)], np.uint64(0xFFFFFFFF)
        c = [np.full(m, n & 0xFFFFFFFF, np.uint64), np.arange(m, dtype=np.uint64), np.full(m, n >> 32, np.uint64), np.zeros(m, np.uint64)]
        k0, k1 = self.seed & 0xFFFFFFFF, self.seed >> 32
        for _ in range(10):
            p0, p1 = M[0] * c[0], M[1] * c[2]
            c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        u = [(v.astype(np.float64) + 0.5) / 2 ** 32 for v in c]
        a = self.amp * np.sqrt(-2 * np.log(u[0])) * np.cos(2 * np.pi * u[1]) * np.exp(2j * np.pi * u[2])
        return torch.from_numpy(np.stack([a * np.cos(2 * np.pi * u[3]), a * np.sin(2 * np.pi * u[3])])).cuda()

    def force(self):
        F = [self.body[0], self.body[1]]
        if self.sigma is not None:
            c = self._draws(self.step) * self.sigma
            for i in (0, 1):
                F[i] = F[i] + ((self.ey.T * c[i]) @ self.ex).real
        return F

    def pull(self, h):
        if self.walls:
            p = torch.nn.functional.pad(h, (0, 0, 1, 1))
        else:
            p = torch.cat([h[:, -1:], h, h[:, :1]], 1)
        if self.open:
            left = self.inflow[:, None, None].expand(-1, p.shape[1], 1)
            p = torch.cat([left, p, p[:, :, -1:]], 2)
        else:
            p = torch.cat([p[:, :, -1:], p, p[:, :, :1]], 2)
        out = []
        for q, (sx, sy) in enumerate(self.signs):
            acc = self.beta[q][0] * h[q]
            for b, ox, oy in ((self.beta[q][1], sx, 0), (self.beta[q][2], 0, sy), (self.beta[q][3], sx, sy)):
                if b:
                    sl = (slice(1 - oy, 1 - oy + self.ny), slice(1 - ox, 1 - ox + self.nx))
                    v = p[q][sl]
                    if self.blocked is not None:
                        v = torch.where(self.blocked[sl], h[self.opp[q]], v)
                    acc = acc.add(v, alpha=b)
            out.append(acc)
        s = torch.stack(out)
        return s if self.fluid is None else s * self.fluid

    def landau(self, M):
        """v of u = gamma (1, v): the residual m - T v - (T00 - m.v) v = 0 by Newton's method
        from m / T00; the last step is the one that is differentiated."""
        e, mx, my, txx, txy, tyy = M[:6]
        Txx, Tyy, T00 = 1 / self.dp + txx, 1 / self.dp + tyy, 1 + e

        def newton(vx, vy):
            E = T00 - (mx * vx + my * vy)
            rx, ry = mx - (Txx * vx + txy * vy) - E * vx, my - (txy * vx + Tyy * vy) - E * vy
            a, b, c, d = -Txx + vx * mx - E, -txy + vx * my, -txy + vy * mx, -Tyy + vy * my - E
            det = a * d - b * c
            return vx + (b * ry - d * rx) / det, vy + (c * rx - a * ry) / det

        with torch.no_grad():
            g = self.dp / (self.dp + 1)
            vx, vy = mx / T00 * g, my / T00 * g
            for _ in range(5):
                vx, vy = newton(vx, vy)
        return newton(vx, vy)

    def macro(self, s):
        M = (self.mom @ s.reshape(len(self.w), -1)).reshape(10, self.ny, self.nx)
        vx, vy = self.landau(M)
        g = 1 / torch.sqrt(1 - vx * vx - vy * vy)
        return M, vx, vy, g, M[0] - (M[1] * vx + M[2] * vy)

    def update(self, h):
        """One step: f*_{n+1} of f*_n, and the v of the state that it collided."""
        s = self.pull(h)
        M, vx, vy, g, em1 = self.macro(s)
        ux, uy, eh = g * vx, g * vy, 1 + em1
        u2 = ux * ux + uy * uy
        om = DT * self.T0 / (self.tau * self.eta) * eh ** self.root
        ca, cb, cc = self.CA * eh * g, self.CB * eh, em1 - self.CC * eh * u2
        p0, p1, p2, p3 = om * g * cc, om * (g * ca - cc), om * (g * cb - ca), -om * cb
        co = [p0, p1 * ux, p1 * uy, p2 * ux * ux, 2 * p2 * ux * uy, p2 * uy * uy,
              p3 * ux ** 3, 3 * p3 * ux * ux * uy, 3 * p3 * ux * uy * uy, p3 * uy ** 3, torch.zeros_like(g)]
        if self.force_on:
            f = -6 * DT / self.T0
            Fx, Fy = self.force()
            mx, my = M[1], M[2]
            Fm = Fx * mx + Fy * my
            Bxx, Bxy, Byy = Fx * M[6] + Fy * M[7], Fx * M[7] + Fy * M[8], Fx * M[8] + Fy * M[9]
            add = [f * Fm / 4, -f * (1 + M[0]) * Fx / 2, -f * (1 + M[0]) * Fy / 2, f * 1.25 * (Bxx - 2 * Fx * mx),
                   f * 2.5 * (Bxy - Fx * my - Fy * mx), f * 1.25 * (Byy - 2 * Fy * my)]
            for i, v in enumerate(add):
                co[i] = co[i] + v
            co[10] = f * 1.25 * (Fm - Bxx - Byy)
        k = torch.stack([1 - om * g, om * ux, om * uy]).reshape(3, -1)
        out = s * (self.rel @ k).reshape(s.shape) + (self.basis @ torch.stack(co).reshape(11, -1)).reshape(s.shape)
        self.step += 1
        return (out if self.fluid is None else out * self.fluid), vx, vy

    def advance(self, n):
        for _ in range(n):
            self.h = self.update(self.h)[0]

    def fields(self):
        s = self.pull(self.h)
        M, vx, vy, g, em1 = self.macro(s)
        f = torch.ones_like(g) if self.fluid is None else self.fluid.double()
        tot = torch.stack([(f * (1 + M[0])).sum(), (f * M[1]).sum(), (f * M[2]).sum(), (f * 0.5 * (vx * vx + vy * vy)).sum()])
        return f * (1 + em1), f * g * vx, f * g * vy, tot, f * vx, f * vy

    def spectrum(self, nbins):
        """E(n) over shells round(|k|), and the modulus squared of the transform by k^2."""
        vx, vy = self.fields()[4:]
        Z = torch.fft.fft2(torch.complex(vx, vy)).abs().square() * (0.5 / (self.nx * self.ny) ** 2)
        kx, ky = (torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda").round() for n in (self.nx, self.ny))
        k2 = ky[:, None] ** 2 + kx[None, :] ** 2
        E = torch.zeros(int(k2.max().sqrt()) + 3, dtype=torch.float64, device="cuda")
        E.index_add_(0, k2.sqrt().round().long().reshape(-1), Z.reshape(-1))
        return E[:nbins], Z, k2

    def gradient(self, steps):
        """J, dJ/dsigma, dJ/d(eta/s), dJ/dF: reverse mode, one step's graph at a time."""
        cells = self.nx * self.ny if self.fluid is None else int(self.fluid.sum())
        par = [self.sigma, self.eta, self.body]
        kept, J = [self.h], 0.0
        with torch.no_grad():
            for n in range(steps):
                h, vx, vy = self.update(kept[-1])
                kept.append(h)
                if n:
                    J = J + (vx * vx + vy * vy).sum() / (2 * cells * steps)
        for p in par:
            p.requires_grad_(True)
        h = kept.pop().requires_grad_(True)
        M, vx, vy, _, _ = self.macro(self.pull(h))
        last = (vx * vx + vy * vy).sum() / (2 * cells * steps)
        J = J + last.detach()
        lam, = torch.autograd.grad(last, h)
        total = [torch.zeros_like(p) for p in par]
        for n in range(steps - 1, -1, -1):
            h = kept.pop().requires_grad_(True)
            self.step = n
            new, vx, vy = self.update(h)
            part = (new * lam).sum()
            if n:
                part = part + (vx * vx + vy * vy).sum() / (2 * cells * steps)
            got = torch.autograd.grad(part, [h] + par, allow_unused=True)
            lam = got[0]
            total = [t if g is None else t + g for t, g in zip(total, got[1:])]
        return [J] + total


def exact(case, seed):
    form = case["form"]
    shapes = [(n, n) for n in _sizes(case)] if form == "ensemble" else _sizes(case)
    # (about 25 ms a step at 4096^2, 1.5 ms at least)
    cost = case["steps"] * sum(max(2.5e-3, 2e-9 * nx * ny) for nx, ny in shapes) * (6 if form == "gradient" else 1)
    if cost > 20:
        return None
    sims = [_Exact(case, nx, ny, _inputs(case, nx, ny, seed * 64 + i if form == "ensemble" else seed)) for i, (nx, ny) in enumerate(shapes)]
    if form == "channel":
        jt = []
        for _ in range(case["steps"]):
            sims[0].advance(1)
            vx = sims[0].fields()[4]
            jt.append(vx[:, -1].mean())
        return dict(t=None, j_t=torch.stack(jt), j_x=vx.mean(0)[case["nx"] // 2:])
    if form == "gradient":
        J, gs, ge, gb = sims[0].gradient(case["steps"])
        return dict(J=J, sigma=gs, eta=ge, body=gb)
    for s in sims:
        s.advance(case["steps"])
    out = {}
    if form == "sample":
        E, Z, k2 = sims[0].spectrum(case["nbins"])
        out = dict(E=E, velocity=torch.sqrt(2 * Z[k2 < _shell(case)[0] ** 2].sum()))
        if not case["fields"]:
            return out
    got = [s.fields() for s in sims]
    out.update({k: torch.cat([f[i].reshape(-1) for f in got]) for i, k in enumerate(("eps", "ux", "uy"))})
    out["totals"] = torch.stack([f[3] for f in got])
    return out
