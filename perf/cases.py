"""What the library is timed on: minimisations, hysteresis sweeps, field, energy
and differentiation calls of a user's program, through the public binding
(paper_1405_2728_gb300.mm and .autograd).

A case is a dict of plain values:

* kind: "minimize" (mm_minimize), "sweep" (mm_hysteresis_sweep), "batch"
  (mm_batch_sweep over `films` uneven films), "heff" (mm_heff), "energy"
  (autograd.Energy forward and backward) or "hvp" (mm_hessian_vec);
* nx, ny, nz: cells; material "film" (soft film on 3.90625 x 3.90625 x 5 nm
  cells, uniform axis), "film_K" (the same with a per-cell anisotropy) or
  "grains" (hard magnet on 2 nm cells, an easy axis per grain);
* precision: "fp64", "fp32" or "f32x2";
* steps: cap on the minimiser steps of a field value; fields: field values.

Minimiser calls keep the default tolerance and stop at a cap that lies well
before convergence, as a capped benchmark or a polling driver does: every pass
then takes the same number of field evaluations.
"""
import math

import numpy as np
import torch

from paper_1405_2728_gb300 import autograd, mm

MU0 = 4e-7 * math.pi
PRECISION = {"fp64": mm.MM_FP64, "fp32": mm.MM_FP32, "f32x2": mm.MM_F32X2}
MATERIAL = {"film": dict(cell=(3.90625e-9, 3.90625e-9, 5e-9), Ms=8.0e5, A=1.3e-11, K=500.0),
            "grains": dict(cell=(2e-9, 2e-9, 2e-9), Ms=1.28e6, A=7.7e-12, K=4.3e6)}
MATERIAL["film_K"] = MATERIAL["film"]
GRAINS = 64
MT = 1e-3 / MU0  # one millitesla in A/m


def _case(name, kind, size, precision, material="film", **more):
    return dict({"kind": kind, "nx": size[0], "ny": size[1], "nz": size[2], "precision": precision,
                 "material": material, "name": name}, **more)


def listed():
    return [
        # the smallest film of the workloads: a field value's minimisation, bound by latency and launches
        _case("small_film_fp64", "minimize", (32, 16, 1), "fp64", steps=20),
        # one field evaluation of a small odd-sized film: an LLG or string-method code that calls the field alone
        _case("small_heff_fp32", "heff", (50, 35, 1), "fp32"),
        # part of a hysteresis loop of the 10 nm convergence study film (200 x 100 x 2 cells, not powers of two)
        _case("study_sweep_fp64", "sweep", (200, 100, 2), "fp64", steps=6, fields=3),
        # the 5 nm convergence study film in double-word precision
        _case("study_min_f32x2", "minimize", (400, 200, 4), "f32x2", steps=8),
        # the headline film in each precision
        _case("film_min_fp64", "minimize", (512, 256, 4), "fp64", steps=10),
        _case("film_min_f32x2", "minimize", (512, 256, 4), "f32x2", steps=10),
        _case("film_min_fp32", "minimize", (512, 256, 4), "fp32", steps=6),
        # the energy and its gradient through autograd (a gradient-based outer loop), ragged sizes
        _case("energy_grad_fp64", "energy", (333, 97, 3), "fp64"),
        # one product of the tangent-plane Hessian with per-cell anisotropy (the adjoint's inner operation)
        _case("hessian_vec_fp64", "hvp", (128, 64, 2), "fp64", material="film_K"),
        # uneven films swept together in one call
        _case("batch_films_fp64", "batch", (300, 160, 3), "fp64", films=8, steps=6, fields=2),
        # granular cubes: three-dimensional grids
        _case("cube_min_fp64", "minimize", (64, 64, 64), "fp64", material="grains", steps=6),
        _case("cube_min_fp32", "minimize", (160, 160, 160), "fp32", material="grains", steps=4),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["minimize", "minimize", "minimize", "sweep", "heff", "energy", "hvp", "batch"])
    if kind == "minimize" and rng.random() < 0.35:
        n = _log_size(rng, 12, 150)
        size = (n, max(6, int(n * rng.uniform(0.6, 1.0))), max(6, int(n * rng.uniform(0.6, 1.0))))
        return {"kind": kind, "nx": size[0], "ny": size[1], "nz": size[2], "precision": rng.choice(["fp64", "fp32"])
                if n <= 80 else "fp32", "material": "grains", "steps": rng.randint(2, 5)}
    nx = _log_size(rng, 16, 512)
    ny = max(8, min(256, int(nx / rng.uniform(1.0, 4.0))))
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": rng.randint(1, 4), "material": "film",
         "precision": rng.choice(["fp64", "fp64", "fp32", "f32x2"])}
    if kind in ("minimize", "sweep"):
        c["material"] = rng.choice(["film", "film", "film_K"])
        c["steps"] = rng.randint(3, 6) if c["precision"] == "fp32" else rng.randint(4, 12)
        if kind == "sweep":
            c["fields"] = 2 if c["precision"] == "fp32" else rng.randint(2, 3)
            c["steps"] = min(c["steps"], 3 if c["precision"] == "fp32" else 6)
    elif kind in ("energy", "hvp"):
        c["precision"] = rng.choice(["fp64", "fp32"])
        c["material"] = rng.choice(["film", "film_K"])
    elif kind == "batch":
        c.update(nx=_log_size(rng, 64, 300), ny=_log_size(rng, 32, 160), precision=rng.choice(["fp64", "fp32"]),
                 films=rng.randint(3, 8), steps=3, fields=1)
    return c


# --- inputs ------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _unit(v):
    return v / v.square().sum(0, keepdim=True).sqrt()


def _smooth(gen, shape):
    """Three smooth fields of unit size over the grid: a few random plane waves each (the long-range part of a
    magnetisation on its way to equilibrium)."""
    nz, ny, nx = shape
    z, y, x = (torch.linspace(0.0, 1.0, n, dtype=torch.float64, device="cuda") for n in shape)
    r = torch.rand((3, 4, 4), dtype=torch.float64, device="cuda", generator=gen)
    out = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    for w in range(4):
        k = (2.0 * math.pi) * (2.0 * r[:, w, :3] - 1.0)
        ph = (k[:, 0].view(3, 1, 1, 1) * x.view(1, 1, 1, nx) + k[:, 1].view(3, 1, 1, 1) * y.view(1, 1, ny, 1) +
              k[:, 2].view(3, 1, 1, 1) * z.view(1, nz, 1, 1))
        out += torch.cos(ph + 2.0 * math.pi * r[:, w, 3].view(3, 1, 1, 1))
    return out


def _state(gen, shape, kind, u):
    """A magnetisation: near saturation along +x (films) or along each grain's easy axis, as a field step of a loop
    finds it, with smooth deviations and a small random tilt; larger ones for single field, energy and Hessian
    calls."""
    xi = 2.0 * torch.rand((3,) + shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    smooth = _smooth(gen, shape)
    a, b = (0.1, 1e-2) if kind in ("minimize", "sweep", "batch") else (0.5, 0.2)
    m = a * smooth + b * xi
    if u is None:
        m[0] += 1.0
    else:
        m += torch.where(u[0:1] < 0.0, -u, u)
    return _unit(m).contiguous()


def _grain_axes(gen, shape):
    """An easy axis per cell: Voronoi grains of random points, each with a random axis."""
    nz, ny, nx = shape
    pts = torch.rand((GRAINS, 3), dtype=torch.float64, device="cuda", generator=gen)
    axes = _unit(torch.randn((3, GRAINS), dtype=torch.float64, device="cuda", generator=gen))
    z, y, x = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n for n in shape)
    best = torch.full(shape, math.inf, dtype=torch.float64, device="cuda")
    grain = torch.zeros(shape, dtype=torch.int64, device="cuda")
    for i in range(GRAINS):
        d = ((x - pts[i, 0]).square().view(1, 1, nx) + (y - pts[i, 1]).square().view(1, ny, 1) +
             (z - pts[i, 2]).square().view(nz, 1, 1))
        grain = torch.where(d < best, i, grain)
        best = torch.minimum(best, d)
    return axes[:, grain].contiguous()


def _films(case):
    """Sizes of the films of a batch (uneven, the first the largest) or the one grid of the other kinds."""
    if case["kind"] != "batch":
        return [(case["nx"], case["ny"], case["nz"])]
    out = []
    for i in range(case["films"]):
        f = 1.0 - 0.75 * i / case["films"]
        out.append((max(8, int(case["nx"] * f)), max(8, int(case["ny"] * f * f)), 1 + (case["nz"] - 1 + i) % 4))
    return out


def _inputs(case, seed):
    """Per film: size, the magnetisation in float64, per-cell K and axes or None, a second field; and the external
    field values (A/m)."""
    gen = _generator(seed)
    films = []
    for nx, ny, nz in _films(case):
        shape = (nz, ny, nx)
        K = u = v = None
        if case["material"] == "film_K":
            K = 300.0 + 400.0 * torch.rand(shape, dtype=torch.float64, device="cuda", generator=gen)
        if case["material"] == "grains":
            u = _grain_axes(gen, shape)
        m = _state(gen, shape, case["kind"], u)
        if case["kind"] == "hvp":
            v = torch.randn((3,) + shape, dtype=torch.float64, device="cuda", generator=gen)
        if case["precision"] == "fp32":  # what a single-precision program holds
            m = m.float().double()
            v = None if v is None else v.float().double()
        if v is not None:
            v = v - (m * v).sum(0, keepdim=True) * m
            v = v.float().double() if case["precision"] == "fp32" else v
        films.append({"size": (nx, ny, nz), "m": m, "K": K, "u": u, "v": v})
    top = 20.0 if case["material"] != "grains" else 500.0
    t = math.radians(1.0)
    H = [[b * MT * math.cos(t), b * MT * math.sin(t), 0.0] for b in
         (top * (0.5 - 0.25 * i) for i in range(case.get("fields", 1)))]
    return films, np.array(H)


# --- the calls -----------------------------------------------------------------

def prepare(case, seed):
    films, H = _inputs(case, seed)
    mat = MATERIAL[case["material"]]
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    probs, ms = [], []
    for f in films:
        grid = mm.make_grid(*f["size"], *mat["cell"])
        m = mm.make_material(mat["Ms"], mat["A"], mat["K"], K_cell=f["K"], u_cell=f["u"])
        torch.cuda.synchronize()
        probs.append(mm.mm_setup_geometry(grid, m, PRECISION[case["precision"]]))
        ms.append(f["m"].to(dtype).contiguous())
    s = {"kind": case["kind"], "probs": probs, "m": ms, "H": H,
         "opts": mm.make_opts(max_iter=case.get("steps", 0))}
    if case["kind"] == "hvp":
        s["v"] = films[0]["v"].to(dtype).contiguous()
    if case["kind"] == "batch":
        s["batch"] = mm.mm_batch_create(probs)
    if case["kind"] == "energy":
        s["m"][0].requires_grad_(True)
    return s


def run(s):
    kind, H = s["kind"], s["H"]
    prob, m0 = s["probs"][0], s["m"][0]
    real = prob.dtype  # a single-precision program keeps its averages and energies in single precision too
    if kind == "heff":
        out = torch.empty_like(m0)
        return mm.mm_heff(prob, m0, H[0], out)
    if kind == "energy":
        m0.grad = None
        E = autograd.Energy.apply(m0, prob, H[0])
        E.backward()
        return {"E": E.detach().to(m0.dtype), "grad": m0.grad}
    if kind == "hvp":
        return mm.mm_hessian_vec(prob, m0, H[0], s["v"], torch.empty_like(m0))
    if kind == "minimize":
        m = m0.clone()
        _, r = mm.mm_minimize(prob, m, H[0], s["opts"])
        return {"m": m, "energy": r.energy, "max_torque": r.max_torque, "evals": int(r.heff_evals)}
    if kind == "sweep":
        m = m0.clone()
        _, mavg, rs = mm.mm_hysteresis_sweep(prob, m, H, opts=s["opts"])
        return {"m": m, "mavg": mavg.astype(real), "energy": np.array([r.energy for r in rs], dtype=real),
                "evals": np.array([r.heff_evals for r in rs])}
    ms = [x.clone() for x in s["m"]]
    _, mavg, rs = mm.mm_batch_sweep(s["batch"], ms, H, opts=s["opts"])
    return {"m": ms, "mavg": mavg.astype(real), "energy": np.array([[r.energy for r in x] for x in rs], dtype=real),
            "evals": np.array([[r.heff_evals for r in x] for x in rs])}


def work(case):
    """Per field evaluation: the magnetisation read and one field written, the tensor's six components of the first
    octant read; the three forward and three inverse real transforms of the doubled grid (2.5 P log2 P each), the
    product (36 per frequency) and 100 operations a cell of local terms."""
    s = 4 if case["precision"] == "fp32" else 8
    evals = {"heff": 1, "energy": 2, "hvp": 2}.get(case["kind"])
    if evals is None:
        evals = (case["steps"] + 1) * case.get("fields", 1)
    b = f = 0
    for nx, ny, nz in _films(case):
        N = nx * ny * nz
        P = math.prod(2 * n if n > 1 else 1 for n in (nx, ny, nz))
        b += evals * (6 + 6) * N * s
        f += evals * (15 * P * math.log2(max(2, P)) + 18 * P + 100 * N)
    return {"bytes": b, "flops": f}


# --- the same in 64 bits with plain torch and numpy ------------------------------------

def _newell_near(n, cell):
    """The cell-averaged demagnetisation tensor (Newell, Williams and Dunlop 1993) at the offsets 0 <= i < n per
    axis, from the closed form in extended precision: [6][nz][ny][nx]."""
    ld = np.longdouble
    h = max(cell)
    d = [ld(c) / ld(h) for c in cell]
    ax = [ld(1) * np.arange(-1, k + 1) * s for k, s in zip(n, d)]
    Z, Y, X = np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")

    def f(x, y, z):
        x2, y2, z2 = x * x, y * y, z * z
        r = np.sqrt(x2 + y2 + z2)
        with np.errstate(all="ignore"):
            a = np.where(x2 + z2 > 0, y / 2 * (z2 - x2) * np.arcsinh(y / np.sqrt(x2 + z2)), 0)
            b = np.where(x2 + y2 > 0, z / 2 * (y2 - x2) * np.arcsinh(z / np.sqrt(x2 + y2)), 0)
            c = np.where((x != 0) & (r > 0), x * y * z * np.arctan(y * z / (x * r)), 0)
        return a + b - c + (2 * x2 - y2 - z2) * r / 6

    def g(x, y, z):
        x2, y2, z2 = x * x, y * y, z * z
        r = np.sqrt(x2 + y2 + z2)

        def at(num, den, w):
            return np.where(den != 0, w * np.arctan(num / den), 0)

        with np.errstate(all="ignore"):
            a = np.where(x2 + y2 > 0, x * y * z * np.arcsinh(z / np.sqrt(x2 + y2)), 0)
            b = np.where(y2 + z2 > 0, y / 6 * (3 * z2 - y2) * np.arcsinh(x / np.sqrt(y2 + z2)), 0)
            c = np.where(x2 + z2 > 0, x / 6 * (3 * z2 - x2) * np.arcsinh(y / np.sqrt(x2 + z2)), 0)
            t = at(x * y, z * r, z * z2 / 6) + at(x * z, y * r, z * y2 / 2) + at(y * z, x * r, z * x2 / 2)
        return a + b + c - t - x * y * r / 3

    def stencil(T):
        for axis in range(3):
            s = [slice(None)] * 3
            lo, mid, hi = list(s), list(s), list(s)
            lo[axis], mid[axis], hi[axis] = slice(0, -2), slice(1, -1), slice(2, None)
            T = 2 * T[tuple(mid)] - T[tuple(lo)] - T[tuple(hi)]
        return T / (4 * ld(math.pi) * _pi_fix() * d[0] * d[1] * d[2])

    return np.stack([stencil(t) for t in (f(X, Y, Z), f(Y, X, Z), f(Z, Y, X), g(X, Y, Z), g(X, Z, Y), g(Y, Z, X))])


def _pi_fix():
    """pi over its nearest double, so that the scale is exact in extended precision."""
    return np.longdouble(4) * np.arctan(np.longdouble(1)) / np.longdouble(math.pi)


def _triangle_rule(n=5):
    """Gauss rule for the weight 1 - |t| on [-1, 1]: the density of the difference of two points of unit cells."""
    moment = [2.0 / ((k + 1) * (k + 2)) if k % 2 == 0 else 0.0 for k in range(2 * n)]
    t = np.polynomial.legendre.leggauss(20)
    nodes = np.concatenate([0.5 * (t[0] + 1), -0.5 * (t[0] + 1)])
    weights = np.concatenate([0.5 * t[1], 0.5 * t[1]]) * (1 - np.abs(nodes))
    a, b, p0, p1, norm0 = [], [], np.zeros_like(nodes), np.ones_like(nodes), 1.0
    for k in range(n):  # the three-term recurrence of the orthogonal polynomials (Stieltjes)
        norm = float(np.sum(weights * p1 * p1))
        a.append(float(np.sum(weights * nodes * p1 * p1)) / norm)
        b.append(norm / norm0)
        p0, p1, norm0 = p1, (nodes - a[k]) * p1 - (b[k] if k else 0.0) * p0, norm
    J = np.diag(a) + np.diag(np.sqrt(b[1:]), 1) + np.diag(np.sqrt(b[1:]), -1)
    x, V = np.linalg.eigh(J)
    return x, V[0] ** 2 * moment[0]


def _newell(n, cell):
    """The first octant [6][nz][ny][nx]: the closed form near the origin (where its cancellation is harmless in
    extended precision), beyond it the average of the dipole kernel over both cells by a Gauss rule."""
    near = [min(k, 20) for k in n]
    z, y, x = (torch.arange(k, dtype=torch.float64, device="cuda") * c for k, c in zip(n[::-1], cell[::-1]))
    out = torch.zeros((6, n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    t, w = _triangle_rule()
    vol = cell[0] * cell[1] * cell[2] / (4 * math.pi)
    for iz in range(len(t)):
        for iy in range(len(t)):
            for ix in range(len(t)):
                X = (x + float(t[ix]) * cell[0]).view(1, 1, -1)
                Y = (y + float(t[iy]) * cell[1]).view(1, -1, 1)
                Z = (z + float(t[iz]) * cell[2]).view(-1, 1, 1)
                r2 = X * X + Y * Y + Z * Z
                q = (vol * float(w[ix] * w[iy] * w[iz])) / (r2 * r2.sqrt())
                q3 = 3 * q / r2
                out[0] += q - q3 * X * X
                out[1] += q - q3 * Y * Y
                out[2] += q - q3 * Z * Z
                out[3] -= q3 * X * Y
                out[4] -= q3 * X * Z
                out[5] -= q3 * Y * Z
    c = _newell_near(near, cell).astype(np.float64)
    out[:, :near[2], :near[1], :near[0]] = torch.from_numpy(c).cuda()
    return out


class _Exact:
    """Field and energy of one film in float64."""

    def __init__(self, case, film):
        mat = MATERIAL[case["material"]]
        self.n, self.cell, self.Ms, self.A = film["size"], mat["cell"], mat["Ms"], mat["A"]
        self.V = math.prod(self.cell)
        shape = tuple(self.n[::-1])
        self.K = film["K"] if film["K"] is not None else torch.full(shape, mat["K"], dtype=torch.float64, device="cuda")
        ex = torch.zeros((3, 1, 1, 1), dtype=torch.float64, device="cuda")
        ex[0] = 1.0
        self.u = film["u"] if film["u"] is not None else ex
        self.P = tuple(2 * k if k > 1 else 1 for k in shape)
        octant = _newell(self.n, self.cell)
        odd = [(0, 0, 0), (0, 0, 0), (0, 0, 0), (0, 1, 1), (1, 0, 1), (1, 1, 0)]  # along z, y, x
        self.N = []
        for c in range(6):
            full = octant[c]
            for axis, k in enumerate(shape):
                if k == 1:
                    continue
                tail = torch.flip(full.narrow(axis, 1, k - 1), (axis,))
                gap = torch.zeros_like(full.narrow(axis, 0, 1))
                full = torch.cat([full, gap, -tail if odd[c][axis] else tail], axis)
            self.N.append(torch.fft.rfftn(full))

    def demag(self, m):
        N, (nx, ny, nz) = self.N, self.n
        a, b, c = (torch.fft.rfftn(m[i], s=self.P) for i in range(3))
        rows = ((N[0], N[3], N[4]), (N[3], N[1], N[5]), (N[4], N[5], N[2]))
        return torch.stack([torch.fft.irfftn(-self.Ms * (r[0] * a + r[1] * b + r[2] * c), s=self.P)[:nz, :ny, :nx]
                            for r in rows])

    def terms(self, m):
        ex = torch.zeros_like(m)
        for axis, d in ((3, self.cell[0]), (2, self.cell[1]), (1, self.cell[2])):
            k = m.shape[axis]
            if k < 2:
                continue
            diff = (m.narrow(axis, 1, k - 1) - m.narrow(axis, 0, k - 1)) * (2 * self.A / (MU0 * self.Ms * d * d))
            ex.narrow(axis, 0, k - 1).add_(diff)
            ex.narrow(axis, 1, k - 1).sub_(diff)
        an = (2 / (MU0 * self.Ms)) * self.K * (m * self.u).sum(0, keepdim=True) * self.u
        return self.demag(m), ex, an

    def heff(self, m, H):
        d, e, a = self.terms(m)
        return d + e + a + torch.as_tensor(H, dtype=torch.float64, device="cuda").view(3, 1, 1, 1)

    def energy(self, m, H):
        d, e, _ = self.terms(m)
        c = MU0 * self.Ms * self.V
        h = torch.as_tensor(H, dtype=torch.float64, device="cuda").view(3, 1, 1, 1)
        an = (self.K * (1 - (m * self.u).sum(0).square())).sum() * self.V
        return -0.5 * c * (m * (d + e)).sum() + an - c * (m * h).sum()

    def minimize(self, m, H, steps):
        """`steps` midpoint steps with alternating Barzilai-Borwein sizes: m, energy, max |m x H| / Ms."""
        tau, mp, gp = 1e-2 / self.Ms, None, None
        for k in range(steps + 1):
            h = self.heff(m, H)
            g = (m * h).sum(0, keepdim=True) * m - m.square().sum(0, keepdim=True) * h
            if k == steps:
                break
            if k:
                s, y = m - mp, g - gp
                ss, sy, yy = (float((p * q).sum()) for p, q in ((s, s), (s, y), (y, y)))
                tau = ss / sy if k % 2 else sy / yy
                if not (math.isfinite(tau) and tau > 0):
                    tau = math.sqrt(ss / yy)
            mp, gp = m, g
            q = 0.25 * tau * tau * g.square().sum(0, keepdim=True)
            m = ((1 - q) * m - tau * g) / (1 + q)
        return m, float(self.energy(m, H)), float(g.square().sum(0).max().sqrt()) / self.Ms


def exact(case, seed):
    films, H = _inputs(case, seed)
    kind = case["kind"]
    single = case["precision"] == "fp32"  # a difference of large terms: no value to hold a single-precision energy to
    out = []
    for f in films:
        p = _Exact(case, f)
        if kind == "heff":
            return p.heff(f["m"], H[0])
        if kind == "energy":
            return {"E": p.energy(f["m"], H[0]), "grad": -MU0 * p.Ms * p.V * p.heff(f["m"], H[0])}
        if kind == "hvp":
            h, Lv = p.heff(f["m"], H[0]), p.heff(f["v"], np.zeros(3))
            w = (f["m"] * h).sum(0, keepdim=True) * f["v"] - Lv
            return w - (f["m"] * w).sum(0, keepdim=True) * f["m"]
        m, energy, mavg = f["m"], [], []
        for h in H:
            m, e, t = p.minimize(m, h, case["steps"])
            energy.append(e)
            mavg.append([float(x.mean()) for x in m])
        if kind == "minimize":
            return {"m": m, "energy": None if single else energy[0], "max_torque": t, "evals": None}
        out.append((m, mavg, energy))
    if kind == "sweep":
        return {"m": out[0][0], "mavg": np.array(out[0][1]),
                "energy": None if single else np.array(out[0][2]), "evals": None}
    return {"m": [o[0] for o in out], "mavg": np.array([o[1] for o in out]),
            "energy": None if single else np.array([o[2] for o in out]), "evals": None}
