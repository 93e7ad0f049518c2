"""Cases that stand for the work users give this framework.

A case is one pass of a user's program through the public entry points of
``paper_2007_12266_gb300``: advancing a rock-image domain (`Domain.advance`)
for one reporting interval and reading the analysis and the updated state
back, the same for a batch of independent domains (`Batch`), and serving a few
jobs from submission to completion (`Server`). Images are seeded sphere packs
made on the GPU; wetting maps, initial phases and parameters follow the
framework's workloads (steady state between walls, reservoir displacement,
pressure and flux faces, batched jobs, served jobs).
"""
import math

import numpy as np
import torch

import paper_2007_12266_gb300 as lbm

DEV = "cuda"


def _domain(name, nx, ny, nz, steps, *, precision="fp32", flow="steady", porosity=0.22, radius=10.0, viscosity=1.0,
            report="state"):
    return dict(name=name, kind="domain", nx=nx, ny=ny, nz=nz, steps=steps, precision=precision, flow=flow,
                porosity=porosity, radius=radius, viscosity=viscosity, report=report)


def listed():
    return [
        # monitoring a small sample closely: the parity pack's size, the
        # analysis every ten timesteps; launches and latency are all of it
        _domain("monitor_32_fp32", 32, 32, 32, 10, flow="periodic", porosity=0.35, radius=4.0, report="measures"),
        # a small steady-state run, one reporting interval
        _domain("steady_64_fp32", 64, 64, 64, 400, porosity=0.30, radius=8.0),
        # a ragged crop with fluids of different viscosity, periodic
        _domain("ragged_101x77x131_fp32", 101, 77, 131, 300, flow="periodic", porosity=0.25, radius=8.0, viscosity=2.0),
        # constant-pressure displacement between open faces (the component
        # populations are stored at every step)
        _domain("pressure_128_fp32", 128, 128, 128, 300, flow="pressure", porosity=0.25, radius=8.0),
        # constant-flux injection, reduced storage
        _domain("flux_96x96x160_fp16", 96, 96, 160, 300, flow="flux", precision="fp16", porosity=0.25, radius=8.0),
        # reservoir-slab displacement at the protocol's porosity, reduced storage
        _domain("displace_192_fp16", 192, 192, 192, 200, flow="reservoir", precision="fp16", porosity=0.20),
        # the benchmark workload in both storages: one reporting interval
        _domain("steady_256_fp32", 256, 256, 256, 300),
        _domain("steady_256_fp16", 256, 256, 256, 200, precision="fp16"),
        # a large image, as core-scale runs use
        _domain("steady_512_fp32", 512, 512, 512, 100, report="fields"),
        # a set of independent jobs of mixed sizes advanced together
        dict(name="batch_12_fp32", kind="batch", jobs=12, lo=64, hi=160, steps=200, precision="fp32"),
        dict(name="batch_12_fp16", kind="batch", jobs=12, lo=64, hi=160, steps=200, precision="fp16"),
        # jobs of the three protocols served from submission to their step ceiling
        dict(name="serve_6_fp16", kind="serve", jobs=6, lo=64, hi=128, steps=300, precision="fp16"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["domain", "domain", "domain", "domain", "batch", "serve"])
    precision = rng.choice(["fp32", "fp16"])
    if kind == "batch":
        lo = rng.randint(48, 96)
        return dict(kind="batch", jobs=rng.randint(2, 16), lo=lo, hi=rng.randint(lo + 8, 160),
                    steps=2 * rng.randint(20, 100), precision=precision)
    if kind == "serve":
        lo = rng.randint(48, 80)
        return dict(kind="serve", jobs=rng.randint(2, 8), lo=lo, hi=rng.randint(lo + 8, 128), steps=300,
                    precision=precision)
    edge = _log_uniform(rng, 24, 400)
    nx, ny, nz = (max(16, round(edge * _log_uniform(rng, 0.8, 1.25))) for _ in range(3))
    voxels = nx * ny * nz
    flow = rng.choice(["steady", "steady", "periodic", "reservoir", "pressure", "flux"])
    steps = max(4, min(400 if precision == "fp32" else 200, int(2.0e9 / voxels)))
    steps = rng.randint(max(2, steps // 3), steps)
    return dict(kind="domain", nx=nx, ny=ny, nz=nz, steps=steps, precision=precision, flow=flow,
                porosity=round(rng.uniform(0.15, 0.35), 3), radius=round(min(10.0, edge / 8), 2),
                viscosity=rng.choice([1.0, 1.0, 2.0]), report="state" if voxels < 20_000_000 else "fields")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _sphere_pack(nx, ny, nz, porosity, r_mean, rng, walls):
    """Solid mask (nz, ny, nx) on the GPU: overlapping spheres, lognormal radii
    (sd 0.3 of the mean), periodic, added in order until the porosity is met to
    the voxel (of the last sphere only as many voxels as are wanted). Each
    voxel takes the number of the first sphere that covers it; the cut is the
    number at which the target is reached. `walls`: solid planes at the x and y
    faces."""
    s2 = math.log(1.09)
    V = nx * ny * nz
    vol = 4.0 / 3.0 * math.pi * r_mean ** 3 * math.exp(3.0 * s2)      # mean of r^3
    n = int(1.5 * -math.log(porosity) * V / vol) + 60
    r = np.minimum(rng.lognormal(math.log(r_mean) - 0.5 * s2, math.sqrt(s2), n), 0.49 * min(nx, ny, nz))
    c = rng.uniform(0.0, 1.0, (n, 3)) * np.array([nx, ny, nz])
    first = torch.full((V,), n, dtype=torch.int32, device=DEV)
    order = np.argsort(r)
    at = 0
    while at < n:
        take = max(1, int(4.0e7 / (2 * r[order[min(at + 64, n - 1)]] + 3) ** 3))
        ids = order[at:at + take]
        at += take
        k = int(math.ceil(2 * r[ids].max())) + 2
        ctr = torch.tensor(c[ids], device=DEV, dtype=torch.float32)
        rad = torch.tensor(r[ids], device=DEV, dtype=torch.float32)
        num = torch.tensor(ids, device=DEV, dtype=torch.int32)
        lo = torch.floor(ctr - rad[:, None] - 0.5)
        ax = lo[:, :, None] + torch.arange(k, device=DEV)                 # voxel numbers, [spheres, axis, k]
        d2 = (ax + 0.5 - ctr[:, :, None]) ** 2
        inside = d2[:, 2, :, None, None] + d2[:, 1, None, :, None] + d2[:, 0, None, None, :] <= (rad * rad)[:, None, None, None]
        w = ax.long() % torch.tensor([nx, ny, nz], device=DEV)[None, :, None]
        flat = w[:, 0, None, None, :] + nx * (w[:, 1, None, :, None] + ny * w[:, 2, :, None, None])
        first.scatter_reduce_(0, flat[inside], num[:, None, None, None].expand(inside.shape)[inside], "amin")
    first += 1
    if walls:
        box = first.view(nz, ny, nx)
        box[:, :, 0] = box[:, :, -1] = 0
        box[:, 0, :] = box[:, -1, :] = 0
    want = int((1.0 - porosity) * V)
    count = torch.bincount(first, minlength=n + 2).cumsum(0)
    cut = int(torch.searchsorted(count, want))
    solid = first <= cut
    solid[(first == cut).nonzero()[:int(count[cut]) - want, 0]] = False
    return solid.view(nz, ny, nx)


def _blobs(pore, saturation, gen, sigma=3.0):
    """Initial phase: smoothed noise cut so that `saturation` of the pores is fluid A."""
    nz, ny, nx = pore.shape
    x = torch.fft.rfftn(torch.randn(pore.shape, device=DEV, generator=gen))
    for a, k in ((0, torch.fft.fftfreq(nz)), (1, torch.fft.fftfreq(ny)), (2, torch.fft.rfftfreq(nx))):
        shape = [1, 1, 1]
        shape[a] = -1
        x *= torch.exp(-2.0 * (math.pi * sigma * k.to(DEV)) ** 2).view(shape)
    x = torch.fft.irfftn(x, s=pore.shape)
    v = x[pore]
    cut = v.kthvalue(max(1, min(v.numel(), int((1.0 - saturation) * v.numel())))).values
    return torch.where(x > cut, 1.0, -1.0) * pore


def _walled(flow):
    return flow == "steady"


def _rock(nx, ny, nz, flow, porosity, radius, seed, saturation=0.4, phis=(-0.3, 0.3)):
    """Image, wetting map and initial phase of one domain as host arrays."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    solid = _sphere_pack(nx, ny, nz, porosity, radius, rng, _walled(flow))
    pore = ~solid
    if flow in ("reservoir", "pressure", "flux"):
        aff = -0.7 * solid.float()
        phi = -1.0 * pore
    else:
        aff = (phis[0] + (phis[1] - phis[0]) * torch.rand(solid.shape, device=DEV, generator=gen)) * solid
        phi = _blobs(pore, saturation, gen)
    return solid.to(torch.uint8).cpu().numpy().astype(np.uint16), aff.float().cpu().numpy(), phi.float().cpu().numpy()


def _params(flow, precision, labels, viscosity=1.0, fz=1e-5):
    """Model parameters of a flow kind, as the framework's workloads set them."""
    kw = dict(tau_a=0.7, tau_b=0.5 + 0.2 * viscosity, alpha=0.005, beta=0.95, force=(0.0, 0.0, fz), precision=precision,
              periodic=(0, 0, 1) if _walled(flow) else ((1, 1, 1) if flow == "periodic" else (1, 1, 0)))
    if flow == "reservoir":
        kw.update(reservoir_z=1)
    elif flow == "pressure":
        kw.update(reservoir_z=2, rho_in=1.002, rho_out=0.998, force=(0.0, 0.0, 0.0))
    elif flow == "flux":
        kw.update(reservoir_z=3, rho_out=1.0, force=(0.0, 0.0, 0.0), flux_in=1e-3 * float(np.count_nonzero(labels[0] == 0)))
    return kw


def _edges(case):
    """Edge lengths of a set of jobs, spread over their range in no order."""
    n = case["jobs"]
    return [round(case["lo"] + (case["hi"] - case["lo"]) * ((7 * j + 3) % n) / max(1, n - 1)) for j in range(n)]


def _inputs(case, seed):
    """Host arrays and parameters of every domain of a case: [(labels, affinity, phi0, parameters, protocol)]."""
    if case["kind"] == "domain":
        rock = _rock(case["nx"], case["ny"], case["nz"], case["flow"], case["porosity"], case["radius"], seed)
        return [rock + (_params(case["flow"], case["precision"], rock[0], case["viscosity"]), "steady")]
    rng = np.random.default_rng(seed)
    jobs = []
    for j, edge in enumerate(_edges(case)):
        porosity = 0.15 + 0.2 * ((5 * j + 2) % 11) / 10
        saturation = float(rng.uniform(0.2, 0.8))
        fz, phis, protocol, flow = 1e-5, (-0.3, 0.3), "steady", "steady"
        if case["kind"] == "batch":
            fz = float(rng.uniform(1e-5, 1e-4))
            phis = (float(rng.uniform(-0.9, 0.9)),) * 2
        else:
            protocol = ("steady", "unsteady", "steady", "centrifuge")[j % 4]
            flow = "steady" if protocol == "steady" else "reservoir"
        rock = _rock(edge, edge, edge, flow, porosity, 8.0, seed * 1009 + j, saturation, phis)
        jobs.append(rock + (_params(flow, case["precision"], rock[0], fz=fz), protocol))
    return jobs


# ---------------------------------------------------------------------------
# the pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    jobs = _inputs(case, seed)
    if case["kind"] == "serve":
        return dict(case=case, server=lbm.Server(check_interval=150), jobs=jobs)
    doms = []
    for labels, aff, phi0, kw, _ in jobs:
        d = lbm.Domain(labels, aff, **kw)
        d.init_fluids(phi0)
        doms.append(d)
    if case["kind"] == "domain":
        return dict(case=case, domain=doms[0])
    batch = lbm.Batch()
    for d in doms:
        batch.add(d)
    return dict(case=case, batch=batch, domains=doms)


# of the analysis a run is followed by, the figures that are not a small
# difference of large sums (the velocities are in f)
MEASURES = ("sat_mass", "mass_a", "mass_b", "mass_total", "p_a", "p_b")


def _report(m):
    return {k: m[k] for k in MEASURES}


def run(state):
    case = state["case"]
    if case["kind"] == "domain":
        d = state["domain"]
        d.advance(case["steps"])
        out = dict(analysis=_report(d.measure()))
        if case["report"] == "state":         # the whole state, as a checkpoint takes it; in reduced storage
            out["f"] = d.distributions("f")   # the components as the phase field
            if case["precision"] == "fp32":
                out.update({k: d.distributions(k) for k in ("a", "b")})
            else:
                out["phi"] = d.read_field("phi")
        elif case["report"] == "fields":      # what a large run writes for later study
            out.update({k: d.read_field(k) for k in ("phi", "rho")})
        else:
            out.update(phi=d.read_field("phi"))
        return out
    if case["kind"] == "batch":
        b = state["batch"]
        b.advance(case["steps"])
        return [dict(analysis=[m["sat_mass"], m["mass_total"]], phi=d.read_field("phi"))
                for m, d in zip(b.measure(), state["domains"])]
    s = state["server"]
    tickets = []
    for labels, aff, phi0, kw, protocol in state["jobs"]:
        tickets.append(s.submit(labels, phi0, aff, kind=protocol, max_steps=case["steps"], **kw))
    while True:
        running, queued, _ = s.run()
        if running == 0 and queued == 0:
            break
    out = []
    for t in tickets:
        p = s.poll(t)
        m = p["last"]
        out.append(dict(steps=p["steps"], analysis=[m["sat_mass"], m["mass_total"]], phi=s.job(t).read_field("phi")))
        s.release(t)
    return out


def work(case):
    """Per timestep and pore site the 19 momentum populations and the two
    component densities, read and written once in their storage type (the
    densities in 32 bits); the state is read back once. A domain whose state
    fits the L2 cache needs memory only for its state in and out. About 330
    operations per site and step (moments, collision, recoloring, gradient)."""
    es = 4 if case["precision"] == "fp32" else 2
    if case["kind"] == "domain":
        sizes = [(case["nx"] * case["ny"] * case["nz"], case["porosity"])]
    else:
        sizes = [(edge ** 3, 0.15 + 0.2 * ((5 * j + 2) % 11) / 10) for j, edge in enumerate(_edges(case))]
    sites = sum(v * p for v, p in sizes)
    voxels = sum(v for v, _ in sizes)
    state = sites * (19 * es + 8)
    moved = 2 * state * (case["steps"] if state > 120e6 else 1)
    whole = 33 * 4 * sites if es == 4 else 19 * 4 * sites + 4 * voxels
    back = {"state": whole, "fields": 8 * voxels}.get(case.get("report"), 4 * voxels)
    inputs = 10 * voxels if case["kind"] == "serve" else 0
    return {"bytes": float(moved + back + inputs), "flops": 330.0 * sites * case["steps"]}


# ---------------------------------------------------------------------------
# the same in 64 bits, plainly
# ---------------------------------------------------------------------------

XI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
      (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
T = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
W = [1 / 3] + [1 / 9] * 6
OPP = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]


def _moments():
    rows = []
    for x, y, z in XI:
        s = x * x + y * y + z * z
        rows.append([1, 19 * s - 30, (21 * s * s - 53 * s + 24) / 2, x, (5 * s - 9) * x, y, (5 * s - 9) * y, z,
                     (5 * s - 9) * z, 3 * x * x - s, (3 * s - 5) * (3 * x * x - s), y * y - z * z,
                     (3 * s - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                     (x * x - y * y) * z])
    M = torch.tensor(rows, dtype=torch.float64, device=DEV).T.contiguous()
    return M, (M / (M * M).sum(1, keepdim=True)).T.contiguous()


class _Plain:
    """The color-gradient model on the pore sites of one image, two-array
    streaming, explicit moment-space collision."""

    def __init__(self, labels, aff, phi0, kw):
        self.kw = kw
        lab = torch.from_numpy(labels.astype(np.int32)).to(DEV)
        self.pore = pore = lab == 0
        self.shape = pore.shape
        N = self.N = int(pore.sum())
        ids = torch.full(pore.shape, N, dtype=torch.int64, device=DEV)
        ids[pore] = torch.arange(N, device=DEV)
        phis = torch.from_numpy(aff).to(DEV).double() * ~pore
        self.nbr = torch.empty((19, N), dtype=torch.int64, device=DEV)
        self.wall_c = torch.zeros((3, N), dtype=torch.float64, device=DEV)
        for q, e in enumerate(XI):
            i, p = ids, phis
            for axis, d in ((2, e[0]), (1, e[1]), (0, e[2])):
                if d:
                    i, p = torch.roll(i, -d, axis), torch.roll(p, -d, axis)
                    if not kw["periodic"][2 - axis]:
                        edge = [slice(None)] * 3
                        edge[axis] = -1 if d > 0 else 0
                        i, p = i.clone(), p.clone()
                        i[tuple(edge)] = N
                        p[tuple(edge)] = 0.0
            self.nbr[q] = i[pore]
            for a in range(3):
                if e[a]:
                    self.wall_c[a] += 18 * T[q] * e[a] * p[pore]
        self.z = pore.nonzero()[:, 0]
        self.M, self.Minv = _moments()
        p = torch.from_numpy(phi0).to(DEV).double()[pore].clamp(-1, 1)
        t = torch.tensor(T, dtype=torch.float64, device=DEV)[:, None]
        w = torch.tensor(W, dtype=torch.float64, device=DEV)[:, None]
        self.f = t.repeat(1, N)
        self.a, self.b = w * (1 + p) / 2, w * (1 - p) / 2
        self.boundary()

    def boundary(self):
        kw, nz = self.kw, self.shape[0]
        kind = kw.get("reservoir_z", 0)
        rho_in, rho_out = kw.get("rho_in", 1.0), kw.get("rho_out", 1.0)
        if kind == 1:
            for at, rho, na in ((self.z < 4, rho_in, 1.0), (self.z >= nz - 4, rho_out, 0.0)):
                for q in range(19):
                    self.f[q][at] = T[q] * rho
                for q in range(7):
                    self.a[q][at], self.b[q][at] = W[q] * na, W[q] * (1 - na)
        for face, sgn, rho in ((0, 1, rho_in), (nz - 1, -1, rho_out)) if kind >= 2 else ():
            at = (self.z == face).nonzero()[:, 0]
            g = self.f[:, at]
            still = sum(g[q] for q in range(19) if XI[q][2] == 0)
            leave = sum(g[q] for q in range(19) if XI[q][2] * sgn < 0)
            K = still + 2 * leave
            if kind == 3 and sgn > 0:
                rho = K.sum() / (at.numel() - kw["flux_in"])
            nt = [0.5 * sum(XI[q][a] * g[q] for q in range(19) if XI[q][2] == 0) for a in (0, 1)]
            un = 1.0 - K / rho
            for q in range(1, 19):
                if XI[q][2] * sgn > 0:
                    part = 1 / 6 if XI[q][0] or XI[q][1] else 1 / 3
                    self.f[q, at] = g[OPP[q]] + rho * un * part - XI[q][0] * nt[0] - XI[q][1] * nt[1]
            enter = W[5] * rho * (1 + 4.5 * un)
            q = 5 if sgn > 0 else 6
            self.a[q, at] = enter if sgn > 0 else torch.zeros_like(enter)
            self.b[q, at] = torch.zeros_like(enter) if sgn > 0 else enter

    def step(self):
        kw, N, f = self.kw, self.N, self.f
        Na, Nb = self.a.sum(0), self.b.sum(0)
        Nt = Na + Nb
        phi = torch.where(Nt > 0, (Na - Nb) / Nt, torch.zeros_like(Nt))
        ext = torch.cat([phi, phi.new_zeros(1)])
        C = self.wall_c.clone()
        for q in range(1, 19):
            p = ext[self.nbr[q]]
            for a in range(3):
                if XI[q][a]:
                    C[a] += 18 * T[q] * XI[q][a] * p
        mag = C.square().sum(0).sqrt()
        n = torch.where(mag > 0, C / mag, torch.zeros_like(C))
        ac = kw["alpha"] * mag
        tau = kw["tau_b"] + (kw["tau_a"] - kw["tau_b"]) * (1 + phi) / 2
        s_nu = 1 / tau
        s_m = 8 * (2 - s_nu) / (8 - s_nu)
        m = self.M @ f
        rho, jx, jy, jz = m[0].clone(), m[3].clone(), m[5].clone(), m[7].clone()
        jj = jx * jx + jy * jy + jz * jz
        eq = torch.zeros_like(m)
        eq[1] = -11 * rho + 19 * jj - ac
        eq[2] = 3 * rho - 5.5 * jj
        eq[4], eq[6], eq[8] = -2 / 3 * jx, -2 / 3 * jy, -2 / 3 * jz
        pxx, pww = 2 * jx * jx - jy * jy - jz * jz, jy * jy - jz * jz
        eq[9] = pxx + 0.5 * ac * (2 * n[0] ** 2 - n[1] ** 2 - n[2] ** 2)
        eq[10] = -0.5 * pxx
        eq[11] = pww + 0.5 * ac * (n[1] ** 2 - n[2] ** 2)
        eq[12] = -0.5 * pww
        eq[13] = jx * jy + 0.5 * ac * n[0] * n[1]
        eq[14] = jy * jz + 0.5 * ac * n[1] * n[2]
        eq[15] = jx * jz + 0.5 * ac * n[0] * n[2]
        m = eq - m
        for k in (1, 2, 9, 10, 11, 12, 13, 14, 15):
            m[k] *= s_nu
        for k in (4, 6, 8, 16, 17, 18):
            m[k] *= s_m
        m[0] = m[3] = m[5] = m[7] = 0.0
        post = self.Minv @ m
        del eq, m
        post += f
        F = kw["force"]
        for q in range(1, 19):
            post[q] += 3 * T[q] * sum(XI[q][a] * F[a] for a in range(3))
        fa, fb = torch.where(Nt > 0, Nb / Nt, Nt), torch.where(Nt > 0, Na / Nt, Nt)
        u = (jx, jy, jz)
        self.f = self.stream(post)
        post = post[:14]
        for q in range(7):
            ux = sum(XI[q][a] * u[a] for a in range(3))
            nx = sum(XI[q][a] * n[a] for a in range(3))
            post[q] = W[q] * Na * (1 + 4.5 * ux + kw["beta"] * fa * nx)
            post[7 + q] = W[q] * Nb * (1 + 4.5 * ux - kw["beta"] * fb * nx)
        self.a, self.b = self.stream(post[:7]), self.stream(post[7:])
        self.boundary()

    def stream(self, g):
        out = torch.empty_like(g)
        for q in range(g.shape[0]):
            up = self.nbr[OPP[q]]
            here = up == self.N
            out[q] = torch.where(here, g[OPP[q]], g[q][up.masked_fill(here, 0)])
        return out

    def analysis(self):
        Na, Nb = self.a.sum(0), self.b.sum(0)
        phi = (Na - Nb) / (Na + Nb)
        rho = self.f.sum(0)
        A = phi > 0
        mass_a, mass_b = float(Na.sum()), float(Nb.sum())
        return dict(sat_mass=mass_a / (mass_a + mass_b), mass_a=mass_a, mass_b=mass_b, mass_total=float(rho.sum()),
                    p_a=float(rho[A].mean() / 3), p_b=float(rho[~A].mean() / 3))

    def field(self, which):
        out = torch.full(self.shape, float("nan"), dtype=torch.float64, device=DEV)
        Na, Nb = self.a.sum(0), self.b.sum(0)
        out[self.pore] = (Na - Nb) / (Na + Nb) if which == "phi" else self.f.sum(0)
        return out


def _wide(v):
    """Numbers as 64-bit values."""
    if isinstance(v, dict):
        return {k: _wide(x) for k, x in v.items()}
    if isinstance(v, list):
        return [_wide(x) for x in v]
    return np.float64(v)


def exact(case, seed):
    out = []
    for labels, aff, phi0, kw, _ in _inputs(case, seed):
        p = _Plain(labels, aff, phi0, kw)
        for _ in range(case["steps"]):
            p.step()
        m = p.analysis()
        if case["kind"] == "domain":
            r = dict(analysis=_wide(m))
            if case["report"] == "state":
                r.update(dict(f=p.f, a=p.a, b=p.b) if case["precision"] == "fp32" else dict(f=p.f, phi=p.field("phi")))
            elif case["report"] == "fields":
                r.update(phi=p.field("phi"), rho=p.field("rho"))
            else:
                r.update(phi=p.field("phi"))
            return r
        if case["kind"] == "batch":
            out.append(dict(analysis=_wide([m["sat_mass"], m["mass_total"]]), phi=p.field("phi")))
        else:
            out.append(dict(steps=None, analysis=_wide([m["sat_mass"], m["mass_total"]]), phi=p.field("phi")))
        del p
    return out
