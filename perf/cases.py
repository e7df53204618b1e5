"""The work that users of this framework have it do, as cases that can be timed and checked.

A case is one pass through the public binding: a force evaluation (``Context.forces``), a short
leapfrog run (``P3MRun``), a vector-Jacobian product of the force map (``Context.force_vjp``) or
the gradient of the final emittance through a run (``P3MRun`` and ``Emittance`` under autograd).
The bunches are those of the package's workloads: a Gaussian, a uniform sphere and a Gaussian
core with a halo shell, drawn on the GPU from the seed.

Fields of a case: ``kind`` (forces, run, vjp, grad), ``dist`` (gauss, long_gauss, sphere, halo),
``n`` particles, the mesh ``nx, ny, nz``, the cutoff ``rc`` in spacings, ``precision`` (0 FP64,
1 FP32 mixed), ``order`` (1 CIC, 2 TSC), ``pm_bc`` and ``pp_bc`` (the cathode in the long and in
the short range), ``det`` (the bitwise reproducible mode), ``energy``, and for runs ``steps``,
``dt`` and ``ckpt`` (steps per checkpoint).
"""
import math

import torch

from paper_2103_02046_gb300 import p3m

Q = 1e-15
E_CHARGE = 1.602176634e-19
E_MASS = 9.1093837015e-31
C_LIGHT = 299792458.0
MASS = Q / E_CHARGE * E_MASS
K_E = 1.0 / (4.0 * math.pi * 8.8541878128e-12)
KAPPA = 3.0
GAP = 0.15e-3  # lowest particle above the cathode at z = 0
SIGMA = {"gauss": (1e-3, 1e-3, 1e-3), "long_gauss": (1e-3, 1e-3, 3e-3),
         "halo": (1e-3, 1e-3, 1e-3)}
RADIUS = 1e-3
ROOM = 1.05  # a run's mesh is laid out over the bunch expanded by this much


def _case(name, kind, dist, n, mesh, rc=2.0, precision=1, order=2, pm_bc=0, pp_bc=0, det=0,
          energy=False, steps=0, dt=0.0, ckpt=0):
    nx, ny, nz = (mesh, mesh, mesh) if isinstance(mesh, int) else mesh
    c = {"kind": kind, "dist": dist, "n": n, "nx": nx, "ny": ny, "nz": nz, "rc": rc,
         "precision": precision, "order": order, "pm_bc": pm_bc, "pp_bc": pp_bc, "det": det,
         "energy": energy, "steps": steps, "dt": dt, "ckpt": ckpt}
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest use: one evaluation of a 4096-particle bunch with its energies, the
        # reference precision (a check of a setup, a scan over parameters).
        _case("forces4k_f64", "forces", "gauss", 4096, 16, precision=0, energy=True),
        # The small photo-gun run: ten leapfrog steps above the cathode.
        _case("run4k_f64_cathode", "run", "gauss", 4096, 16, precision=0, pm_bc=1, steps=10,
              dt=1e-12),
        # An odd particle count on a ragged mesh, the cathode in both ranges, cloud-in-cell.
        _case("forces5003_f32_ragged", "forces", "gauss", 5003, (20, 24, 64), order=1, pm_bc=1,
              pp_bc=1),
        # A quick look in mixed precision: a quarter of a million particles, odd count.
        _case("forces261k_f32", "forces", "sphere", 261121, 64),
        # The ordinary production evaluation.
        _case("forces2m_f32", "forces", "sphere", 2097152, 128),
        # The Coulomb-explosion workload at full size, the benchmark's default.
        _case("forces16m_f32", "forces", "sphere", 16777216, 256),
        # The dense long bunch of the energy-drift and gradient studies.
        _case("forces1m_f32_dense", "forces", "long_gauss", 1048576, 64),
        # The boundary stress: core and halo above the cathode, images in both ranges.
        _case("forces4m_f32_halo", "forces", "halo", 4194304, 128, rc=3.0, pm_bc=1, pp_bc=1),
        # The reference precision at production size.
        _case("forces2m_f64", "forces", "sphere", 2097152, 128, precision=0),
        # A few steps of a dense thermal bunch (the shape of a long tracking run).
        _case("run131k_f32_dense", "run", "long_gauss", 131072, 64, steps=4, dt=2.5e-13),
        # The reverse direction of one evaluation on the dense bunch.
        _case("vjp262k_f32_dense", "vjp", "long_gauss", 262144, 64),
        # The gradient of the final emittance with respect to the initial phase space.
        _case("grad4k_f64", "grad", "long_gauss", 4096, 64, precision=0, steps=20, dt=2.5e-13,
              ckpt=5),
    ]


# ------------------------------------------------------------------------------------------
# sizes
# ------------------------------------------------------------------------------------------
def _half_extent(case):
    """Expected half extents of the bunch per axis."""
    n, d = case["n"], case["dist"]
    if d == "sphere":
        return (RADIUS,) * 3
    if d == "halo":
        return (6e-3,) * 3
    t = math.sqrt(2.0 * math.log(n))
    t -= (math.log(math.log(n)) + math.log(4.0 * math.pi)) / (2.0 * t)
    return tuple(t * s for s in SIGMA[d])


def _pairs(case):
    """Expected unordered pairs within the cutoff."""
    n = case["n"]
    room = ROOM if case["kind"] in ("run", "grad") else 1.0
    m = (case["nx"], case["ny"], case["nz"])
    rc = case["rc"] * max(2.0 * room * e / (k - 5) for e, k in zip(_half_extent(case), m))
    if case["dist"] == "sphere":
        p = min(1.0, (rc / RADIUS) ** 3)
    else:
        s = SIGMA[case["dist"]]
        frac = 0.95 ** 2 if case["dist"] == "halo" else 1.0
        p = min(1.0, frac * 4.0 / 3.0 * math.pi * rc ** 3 /
                ((4.0 * math.pi) ** 1.5 * s[0] * s[1] * s[2]))
    return 0.5 * n * n * p


def work(case):
    """Bytes: the positions read and the results written once (per pass, whatever happens
    between). Flops: per evaluation 37 for each unordered pair (the screened force), 27 nodes a
    particle in the deposit and the interpolation, and a forward and an inverse real transform of
    the doubled mesh; a product with the Jacobian takes about three times the pair's work and a
    second transform pair."""
    n = case["n"]
    points = 8.0 * case["nx"] * case["ny"] * case["nz"]
    fft = 2 * 2.5 * points * math.log2(points)
    mesh = 27 * 2 * n + 27 * 6 * n + fft
    force = 37.0 * _pairs(case) + mesh
    vjp = 100.0 * _pairs(case) + 2 * mesh
    if case["kind"] == "forces":
        return {"bytes": 48.0 * n, "flops": force}
    if case["kind"] == "run":
        return {"bytes": 96.0 * n, "flops": (case["steps"] + 1) * force}
    if case["kind"] == "vjp":
        return {"bytes": 72.0 * n, "flops": vjp}
    return {"bytes": 144.0 * n, "flops": case["steps"] * (force + vjp)}


def _seconds(case):
    """A rough cost, to keep drawn cases below the largest listed one."""
    rate = 1.2e11 if case["precision"] else 1.6e10
    if case["det"]:
        rate *= 0.3
    one = _pairs(case) / rate
    if case["kind"] == "vjp":
        return 3.0 * one
    if case["kind"] == "grad":
        return (case["steps"] + 2) * 8.0 * one
    return (case["steps"] + 1) * one


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same bunches, any count between the listed ones, meshes with and
    without powers of two, the cutoffs, precisions and boundary options in use."""
    while True:
        kind = rng.choice(("forces", "forces", "forces", "run", "vjp", "grad"))
        dist = rng.choice(("sphere", "gauss", "long_gauss", "halo"))
        precision = rng.choice((1, 1, 0))
        pm_bc = rng.choice((0, 0, 1))
        kw = dict(rc=rng.choice((1.0, 2.0, 3.0)), precision=precision, order=rng.choice((2, 2, 1)),
                  pm_bc=pm_bc, pp_bc=pm_bc and rng.choice((0, 1)))
        if kind == "forces":
            n = _log_int(rng, 4096, 16777216 if precision else 4194304)
            kw["energy"] = rng.random() < 0.25
            kw["det"] = int(not precision and rng.random() < 0.2)
        elif kind == "run":
            n = _log_int(rng, 4096, 1048576)
            kw.update(steps=rng.randint(2, 6), dt=2.5e-13)
        elif kind == "vjp":
            n = _log_int(rng, 4096, 1048576)
        else:
            n = _log_int(rng, 4096, 65536)
            kw.update(steps=rng.randint(4, 12), dt=2.5e-13, ckpt=rng.randint(2, 5))
        # between one and eight particles a node in the mean, as in the listed cases' range
        side = (n / math.exp(rng.uniform(math.log(0.5), math.log(8.0)))) ** (1.0 / 3.0)
        side = max(16, min(256, int(round(side))))
        shape = rng.random()
        if shape < 0.5:  # a power of two
            mesh = 1 << max(4, min(8, round(math.log2(side))))
        elif shape < 0.8:
            mesh = side
        else:  # another number of nodes along each axis
            mesh = tuple(max(16, min(256, int(round(side * rng.uniform(0.8, 1.25)))))
                         for _ in range(3))
        case = _case(None, kind, dist, n, mesh, **kw)
        if _seconds(case) <= 0.12:
            return case


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _bunch(case, seed):
    """Positions and momenta of the case, and the cotangent of a vector-Jacobian product."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))

    def normal(k):
        return torch.randn((k, 3), generator=g, device=dev, dtype=torch.float64)

    def uniform(k):
        return torch.rand((k, 1), generator=g, device=dev, dtype=torch.float64)

    def direction(k):
        v = normal(k)
        return v / v.norm(dim=1, keepdim=True)

    n = case["n"]
    if case["dist"] == "sphere":
        x = direction(n) * (RADIUS * uniform(n) ** (1.0 / 3.0))
    else:
        sigma = torch.tensor(SIGMA[case["dist"]], device=dev, dtype=torch.float64)
        x = normal(n) * sigma
        if case["dist"] == "halo":
            k = int(round(0.05 * n))
            r3 = (4e-3) ** 3 + uniform(k) * ((6e-3) ** 3 - (4e-3) ** 3)
            x[:k] = direction(k) * r3 ** (1.0 / 3.0)
            x = x[torch.randperm(n, generator=g, device=dev)].contiguous()
    if case["pm_bc"] == 1:
        x[:, 2] += GAP - x[:, 2].min()
    p = normal(n) * (1e-4 * MASS * C_LIGHT)  # thermal
    w = normal(n) if case["kind"] == "vjp" else None
    return x.contiguous(), p.contiguous(), w


def _mesh_points(case, x):
    """The positions over whose bounding box the mesh is laid out."""
    if case["kind"] not in ("run", "grad"):
        return x
    mid = 0.5 * (x.min(dim=0).values + x.max(dim=0).values)
    return (mid + ROOM * (x - mid)).contiguous()


def prepare(case, seed):
    x, p, w = _bunch(case, seed)
    slots = -(-case["steps"] // case["ckpt"]) if case["kind"] == "grad" else 0
    prm = p3m.Params(n=(case["nx"], case["ny"], case["nz"]), rc_over_h=case["rc"], kappa=KAPPA,
                     assign_order=case["order"], pm_bc=case["pm_bc"], pp_bc=case["pp_bc"],
                     z_cathode=0.0, precision=case["precision"], deterministic=case["det"], q=Q,
                     mass=MASS, adj_slots=slots, adj_segment=case["ckpt"])
    prm = p3m.auto_mesh(_mesh_points(case, x), prm)
    return {"case": case, "ctx": p3m.Context(prm, case["n"]), "x": x, "p": p, "w": w}


def run(state):
    case, ctx, x, p = state["case"], state["ctx"], state["x"], state["p"]
    kind = case["kind"]
    if kind == "forces":
        return ctx.forces(x, energy=case["energy"])
    if kind == "run":
        return p3m.P3MRun.apply(x, p, ctx, case["dt"], case["steps"])
    if kind == "vjp":
        return ctx.force_vjp(x, state["w"])
    x0, p0 = x.detach().requires_grad_(True), p.detach().requires_grad_(True)
    x1, p1 = p3m.P3MRun.apply(x0, p0, ctx, case["dt"], case["steps"])
    j = p3m.Emittance.apply(x1, p1, ctx)
    gx, gp = torch.autograd.grad(j, (x0, p0))
    return {"x": x1.detach(), "p": p1.detach(), "emittance": j.detach(), "gx": gx, "gp": gp}


# ------------------------------------------------------------------------------------------
# the same in 64 bits with torch alone
# ------------------------------------------------------------------------------------------
class _Exact:
    """Forces and their vector-Jacobian products in FP64: the short range from a list of the
    candidates in the 27 cells around each particle, the long range from a transform of the
    doubled mesh."""

    CHUNK = 1 << 25  # candidate pairs at a time

    def __init__(self, case, points):
        self.case = case
        self.n = (case["nx"], case["ny"], case["nz"])
        dev = points.device
        nn = torch.tensor(self.n, device=dev, dtype=torch.float64)
        a, b = points.min(dim=0).values, points.max(dim=0).values
        self.h = (b - a) / (nn - 5)
        self.lo = a - 2.0 * self.h
        self.rc = float(case["rc"] * self.h.max())
        self.alpha = KAPPA / self.rc
        self.dev = dev
        self.kernels = self._kernels()

    def _kernels(self):
        """Spectra of erf(alpha r)/r at the offsets between nodes and to their images."""
        m = []
        for d in range(3):
            k = torch.arange(2 * self.n[d], device=self.dev)
            m.append((torch.where(k < self.n[d], k, k - 2 * self.n[d]).double(), k == self.n[d]))
        unused = m[2][1][:, None, None] | m[1][1][None, :, None] | m[0][1][None, None, :]
        xy2 = ((m[1][0] * self.h[1]) ** 2)[None, :, None] + ((m[0][0] * self.h[0]) ** 2)[None, None]

        def spectrum(z):
            r = torch.sqrt(xy2 + (z ** 2)[:, None, None])
            k = torch.where(r > 0, torch.erf(self.alpha * r) / r.clamp_min(1e-300),
                            torch.full_like(r, 2.0 * self.alpha / math.sqrt(math.pi)))
            k[unused] = 0.0
            return torch.fft.rfftn(k)

        out = [spectrum(m[2][0] * self.h[2])]
        if self.case["pm_bc"] == 1:
            out.append(spectrum(2.0 * self.lo[2] + (m[2][0] + self.n[2] - 1) * self.h[2]))
        return out

    def _weights(self, x):
        """First node, weights and their derivatives per axis (in mesh units)."""
        s = (x - self.lo) / self.h
        if self.case["order"] == 2:
            c = torch.floor(s + 0.5).detach()
            u = s - c
            w = torch.stack((0.5 * (0.5 - u) ** 2, 0.75 - u ** 2, 0.5 * (0.5 + u) ** 2), 2)
            dw = torch.stack((u - 0.5, -2.0 * u, u + 0.5), 2)
            return c.long() - 1, w, dw
        c = torch.floor(s).detach()
        u = s - c
        return c.long(), torch.stack((1.0 - u, u), 2), torch.stack((-torch.ones_like(u),
                                                                    torch.ones_like(u)), 2)

    def _nodes(self, c):
        s = 3 if self.case["order"] == 2 else 2
        for k in range(s):
            for j in range(s):
                for i in range(s):
                    yield i, j, k, ((c[:, 2] + k) * self.n[1] + c[:, 1] + j) * self.n[0] + c[:, 0] + i

    def _long(self, x):
        """Long-range force and energy (differentiable in x)."""
        nx, ny, nz = self.n
        c, w, dw = self._weights(x)
        q = torch.zeros(nx * ny * nz, device=self.dev, dtype=torch.float64)
        for i, j, k, at in self._nodes(c):
            q = q.index_add(0, at, w[:, 0, i] * w[:, 1, j] * w[:, 2, k])
        q = Q * q.reshape(nz, ny, nx)
        size = (2 * nz, 2 * ny, 2 * nx)

        def pad(v):
            return torch.fft.rfftn(v, s=size)

        spec = self.kernels[0] * pad(q)
        if len(self.kernels) > 1:
            spec = spec - self.kernels[1] * pad(q.flip(0))
        phi = K_E * torch.fft.irfftn(spec, s=size)[:nz, :ny, :nx]
        flat = phi.reshape(-1)
        g = [0.0, 0.0, 0.0]
        for i, j, k, at in self._nodes(c):
            v = flat[at]
            g[0] = g[0] + v * dw[:, 0, i] * w[:, 1, j] * w[:, 2, k]
            g[1] = g[1] + v * w[:, 0, i] * dw[:, 1, j] * w[:, 2, k]
            g[2] = g[2] + v * w[:, 0, i] * w[:, 1, j] * dw[:, 2, k]
        f = -Q * torch.stack(g, 1) / self.h
        return f, 0.5 * (q * phi).sum()

    def _lists(self, x):
        """The particles in cell order, and chunks (i, j) of candidate pairs of sorted ones."""
        cell = torch.floor((x - self.lo) / (self.rc * (1.0 + 1e-9))).long()
        nc = cell.max(dim=0).values + 1
        key = (cell[:, 2] * nc[1] + cell[:, 1]) * nc[0] + cell[:, 0]
        key, order = torch.sort(key)
        xs, cs = x[order], cell[order]
        base = torch.arange(len(x), device=self.dev)

        def chunks():
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    cy, cz = cs[:, 1] + dy, cs[:, 2] + dz
                    ok = (cy >= 0) & (cy < nc[1]) & (cz >= 0) & (cz < nc[2])
                    row = (cz * nc[1] + cy) * nc[0]
                    a = torch.searchsorted(key, row + (cs[:, 0] - 1).clamp_min(0))
                    b = torch.searchsorted(key, row + torch.minimum(cs[:, 0] + 1, nc[0] - 1),
                                           right=True)
                    count = torch.where(ok, b - a, torch.zeros_like(a))
                    ends = torch.cumsum(count, 0)
                    total, done, first = int(ends[-1]), 0, 0
                    while done < total:
                        last = int(torch.searchsorted(ends, done + self.CHUNK, right=True))
                        last = max(last, first + 1)
                        k = count[first:last]
                        i = torch.repeat_interleave(base[first:last], k)
                        off = torch.arange(len(i), device=self.dev) - torch.repeat_interleave(
                            torch.cumsum(k, 0) - k, k)
                        yield i, a[i] + off
                        done, first = int(ends[last - 1]), last

        return xs, order, chunks()

    def _images(self, xs):
        """Pairs of sorted particles with images within reach, and the separations."""
        if not self.case["pp_bc"]:
            return
        near = torch.nonzero(xs[:, 2] < self.rc).flatten()
        mirror = torch.tensor((1.0, 1.0, -1.0), device=self.dev, dtype=torch.float64)
        step = max(1, self.CHUNK // max(1, len(near)))
        for s in range(0, len(near), step):
            i = near[s:s + step].repeat_interleave(len(near))
            j = near.repeat(len(near[s:s + step]))
            d = xs[i] - xs[j] * mirror
            r2 = (d * d).sum(1)
            ok = r2 < self.rc ** 2
            yield i[ok], j[ok], d[ok], r2[ok]

    def _hits(self, xs, chunks):
        for i, j in chunks:
            r2 = ((xs[i] - xs[j]) ** 2).sum(1)
            ok = (r2 < self.rc ** 2) & (r2 > 0)
            i, j = i[ok], j[ok]
            yield i, j, xs[i] - xs[j], r2[ok]

    def _terms(self, r2):
        """Force over separation, potential (both without k_e q^2), and the Gaussian term."""
        r = torch.sqrt(r2)
        pot = torch.erfc(self.alpha * r) / r
        ex = 2.0 * self.alpha / math.sqrt(math.pi) * torch.exp(-self.alpha ** 2 * r2)
        return (pot + ex) / r2, pot, ex

    def forces(self, x):
        f, long_energy = self._long(x)
        xs, order, chunks = self._lists(x)
        short = torch.zeros_like(x)
        energy = torch.zeros((), device=self.dev, dtype=torch.float64)
        for i, j, d, r2 in self._hits(xs, chunks):
            fco, pot, _ = self._terms(r2)
            short.index_add_(0, i, fco[:, None] * d)
            energy += pot.sum()
        for i, j, d, r2 in self._images(xs):
            fco, pot, _ = self._terms(r2)
            short.index_add_(0, i, -fco[:, None] * d)
            energy -= pot.sum()
        f = f.clone()
        f[order] += K_E * Q * Q * short
        return f, torch.stack((0.5 * K_E * Q * Q * energy, long_energy))

    def vjp(self, x, w):
        """(dF/dx)^T w."""
        y = x.detach().clone().requires_grad_(True)
        (long,) = torch.autograd.grad((self._long(y)[0] * w).sum(), y)
        xs, order, chunks = self._lists(x)
        ws = w[order]
        short = torch.zeros_like(x)

        def product(d, r2, v):
            """H(d) v with H the Jacobian of the pair force."""
            fco, pot, ex = self._terms(r2)
            # f(r) = A / r^2 with A = pot + ex; A' = -(pot + ex)/r - 2 alpha^2 r ex
            r = torch.sqrt(r2)
            slope = (-(pot + ex) / r - 2.0 * self.alpha ** 2 * r * ex) / r2 - 2.0 * fco / r
            return fco[:, None] * v + (slope / r * (d * v).sum(1))[:, None] * d

        for i, j, d, r2 in self._hits(xs, chunks):
            short.index_add_(0, i, product(d, r2, ws[i] - ws[j]))
        mirror = torch.tensor((1.0, 1.0, -1.0), device=self.dev, dtype=torch.float64)
        for i, j, d, r2 in self._images(xs):
            short.index_add_(0, i, -product(d, r2, ws[i] - ws[j] * mirror))
        long = long.clone()
        long[order] += K_E * Q * Q * short
        return long


def _emittance(x, p):
    n = len(x)
    dx, dp = x - x.mean(dim=0), p - p.mean(dim=0)
    a, b, c = (dx * dx).sum(0) / n, (dp * dp).sum(0) / n, (dx * dp).sum(0) / n
    return (torch.sqrt(a * b - c * c) / (MASS * C_LIGHT)).sum()


def exact(case, seed):
    if case["n"] * case["n"] and _pairs(case) * max(1, case["steps"]) > 4e9:
        return None  # minutes of elementwise FP64
    x, p, w = _bunch(case, seed)
    ref = _Exact(case, _mesh_points(case, x))
    with torch.no_grad():
        if case["kind"] == "forces":
            f, e = ref.forces(x)
            return (f, e) if case["energy"] else f
    if case["kind"] == "vjp":
        return ref.vjp(x, w)
    dt, steps = case["dt"], case["steps"]
    trail = [x]
    with torch.no_grad():
        f = ref.forces(x)[0]
        for _ in range(steps):
            p = p + 0.5 * dt * f
            x = x + dt / MASS * p
            f = ref.forces(x)[0]
            p = p + 0.5 * dt * f
            trail.append(x)
    if case["kind"] == "run":
        return x, p
    xe, pe = x.requires_grad_(True), p.requires_grad_(True)
    j = _emittance(xe, pe)
    lx, lp = torch.autograd.grad(j, (xe, pe))
    lx = lx + ref.vjp(trail[-1], 0.5 * dt * lp)
    for k in range(steps - 1, -1, -1):
        lp = lp + dt / MASS * lx
        lx = lx + ref.vjp(trail[k], (dt if k else 0.5 * dt) * lp)
    return {"x": x.detach(), "p": p.detach(), "emittance": j.detach(), "gx": lx, "gp": lp}
