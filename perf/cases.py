"""What this library is used for, as cases that can be timed and checked.

Three kinds, all through the public calls of ``paper_2003_03130_gb300``:

* ``coupled``: cells in a lattice-Boltzmann flow. One pass puts the cells at
  their start positions, advances ``steps`` coupled steps
  (``cf_step_exchange``) and, with ``field``, reads the velocity field. The
  fluid of a prepared state is at rest; it keeps developing from pass to pass,
  as in a run that reports every ``steps`` steps.
* ``elastic``: one cell without fluid, as a quasi-static solver or a report
  uses it: forces, energy, the force Jacobian along a direction, the gradient
  with respect to the moduli, Taylor deformation and cell strain.
* ``compress``: cells compressed between plates (``adjoint.Compression``), the
  force curve alone or with its gradient with respect to the moduli.

The library computes in 32 bits and widens what it hands out (positions are
the 64-bit reference plus a 32-bit displacement), so displacements, forces
and fields are returned in the 32 bits that they were computed in, and so are
plate forces and gradients, whose terms are 32-bit.
"""
import functools
import math

import numpy as np
import torch

import paper_2003_03130_gb300 as P
from paper_2003_03130_gb300.adjoint import Compression, CompressionCurve
from workloads.configs import plate_schedule
from workloads.mesh import sphere_tet_mesh


# ---------------------------------------------------------------- cases
def _coupled(name, nx, ny, nz, steps, **kw):
    c = dict(kind="coupled", nx=nx, ny=ny, nz=nz, cells=1, r_min=16.0, r_max=16.0, h=1.72, fmt="f32", delta="trilinear",
             spread="float", u_wall=0.05, u_max=0.0, mu=0.0, kappa_mu=50.0, w=0.5, noise=0.05, tune=False, field=True,
             steps=steps)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _compress(name, cells, radius, h, levels, steps, ramp, gradient):
    c = dict(kind="compress", cells=cells, radius=radius, h=h, levels=levels, steps=steps, ramp=ramp, gradient=gradient)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest coupled run: a cell in a 32^3 box, the size that the 64-bit
        # oracle checks, nearly incompressible; every launch is short
        _coupled("shear_32", 32, 32, 32, 100, r_min=8.0, r_max=8.0, h=1.4, u_wall=0.01, mu=5e-5, kappa_mu=100.0),
        # a program that drives the cells itself: positions in, one step, positions out
        _coupled("exchange_128", 128, 128, 128, 1, field=False),
        # the production shear run, up to its next report
        _coupled("shear_128", 128, 128, 128, 500, tune=True),
        # eight cells in the 5 x 8 x 4 R box of the multiple-cell runs (22 % by volume)
        _coupled("multicell_8", 80, 128, 64, 300, cells=8, tune=True),
        # pressure-driven channel with 16-bit populations, stochastically rounded
        _coupled("channel_f16sr", 256, 128, 128, 200, fmt="f16sr", u_wall=0.0, u_max=0.02, tune=True),
        # the paper's 10 x 15 x 5 R box with the four-point delta kernel, runs that have
        # to repeat bit for bit
        _coupled("box_peskin_fixed", 160, 240, 80, 200, delta="peskin4", spread="fixed", w=1.0),
        # the largest: 400 cells of uneven size in a 512 x 256 x 256 channel
        _coupled("suspension_400", 512, 256, 256, 100, cells=400, r_min=6.0, r_max=20.0, h=1.64, u_wall=0.0, u_max=0.02,
                 tune=True),
        # one iteration and one report of a solver without fluid: a single production cell
        dict(name="elastic_16", kind="elastic", radius=16.0, h=1.72, kappa_mu=50.0),
        # the same for a fine, nearly incompressible cell
        dict(name="elastic_fine", kind="elastic", radius=24.0, h=1.2, kappa_mu=500.0),
        # fitting two small cells: a short protocol, its curve and gradient
        _compress("fit_2", 2, 5.0, 1.4, 3, 60, 3, True),
        # 64 cells of ~8k tets: the force curve alone
        _compress("curve_64", 64, 10.0, 1.45, 3, 400, 10, False),
        # the same cells: curve and gradient, one step of a fit
        _compress("fit_64", 64, 10.0, 1.45, 1, 200, 2, True),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["coupled", "coupled", "coupled", "compress", "elastic"])
    if kind == "elastic":
        h = round(rng.uniform(1.2, 2.0), 2)
        return dict(kind="elastic", radius=round(h * _log(rng, 3.0, 20.0), 1), h=h, kappa_mu=rng.choice([20.0, 50.0, 100.0, 500.0]))
    if kind == "compress":
        h = round(rng.uniform(1.3, 1.6), 2)
        return _compress("", int(round(_log(rng, 1, 64))), round(h * rng.uniform(3.0, 7.0), 1), h, rng.randint(1, 3),
                         rng.randint(40, 240), rng.choice([2, 3]), rng.random() < 0.6)
    nodes = _log(rng, 3.0e4, 8.0e6)
    side = nodes ** (1.0 / 3.0)
    ny = max(28, int(side * rng.uniform(0.8, 1.3)))
    nx = max(24, int(math.sqrt(nodes / ny) * rng.uniform(0.7, 1.4)))
    nz = max(24, int(nodes / ny / nx))
    nx += nx % 2 if rng.random() < 0.6 else 0
    r_max = round(rng.uniform(5.0, min(16.0, (ny - 9) / 2.0, (nx - 3) / 2.0, (nz - 3) / 2.0)), 1)
    most = max(1, int(0.12 * nx * ny * nz / (4.2 * r_max**3)))
    walls = rng.random() < 0.5
    u_wall = rng.choice([0.02, 0.05]) if walls else 0.0
    n = nx * ny * nz
    steps = int(min(_log(rng, 1, 400), 1.5e9 / (n + 1.0e5), 0.3 * ny / (2 * u_wall) if walls else 400))
    kappa_mu = rng.choice([20.0, 50.0, 200.0]) if steps <= 40 else rng.choice([20.0, 50.0])
    return _coupled("", nx, ny, nz, max(1, steps), cells=int(round(_log(rng, 1, most))), r_min=max(5.0, round(r_max * rng.uniform(0.5, 1.0), 1)),
                    r_max=max(5.0, r_max), h=round(rng.uniform(1.5, 1.8), 2), fmt=rng.choice(["f32", "f32", "f16", "f16sr", "bf16sr"]),
                    delta=rng.choice(["trilinear", "trilinear", "peskin4"]), spread=rng.choice(["float", "float", "fixed"]),
                    u_wall=u_wall, u_max=0.0 if walls else 0.02, kappa_mu=kappa_mu,
                    w=round(rng.uniform(0.0, 1.0), 2), tune=rng.random() < 0.3)


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _mesh(radius, h):
    return sphere_tet_mesh(radius, h)


TAU = 1.0


def _flow(case):
    """Wall speeds, body force and the shear modulus: Ca = 0.5 at the shear rate 0.1 / 128 (stiffer cells become unstable
    in the thousands of steps that a prepared state is advanced while it is timed)."""
    nu = (TAU - 0.5) / 3.0
    g = 8.0 * nu * case["u_max"] / case["ny"] ** 2
    return -case["u_wall"], case["u_wall"], g, case["mu"] or nu * (0.1 / 128.0) / 0.5


@functools.lru_cache(maxsize=4)
def _layout(key):
    """Radii and centres of the cells: one cell in the middle, or without overlap (gap 2) and off the walls, largest first."""
    nx, ny, nz, cells, r_min, r_max = key
    if cells == 1:
        return [(r_max, np.array([(nx - 1) / 2.0, (ny - 1) / 2.0, (nz - 1) / 2.0]))]
    rng = np.random.Generator(np.random.PCG64(400))
    size = np.array([nx, ny, nz], np.float64)
    radii = np.sort(np.round(rng.uniform(r_min, r_max, cells) * 2.0) / 2.0)[::-1]
    at, got = np.zeros((0, 3)), []
    for r in radii:
        for _ in range(200):
            c = np.stack([rng.uniform(0, nx, 256), rng.uniform(r + 3.0, max(r + 3.0, ny - 4.0 - r), 256), rng.uniform(0, nz, 256)], 1)
            ok = np.ones(256, bool)
            if len(at):
                d = np.abs(c[:, None] - at[None])
                d[..., [0, 2]] = np.minimum(d[..., [0, 2]], size[[0, 2]] - d[..., [0, 2]])
                ok = (np.sqrt((d * d).sum(-1)) >= r + np.array([q for q, _ in got])[None] + 2.0).all(1)
            if ok.any():
                c = c[np.argmax(ok)]
                at = np.concatenate([at, c[None]])
                got.append((float(r), c))
                break
    return got


def _cells(case, seed):
    """Reference positions, tets, start positions and moduli of every cell: the start positions, off the rest shape, come from the seed."""
    rng = np.random.Generator(np.random.PCG64([seed, 1]))
    if case["kind"] == "coupled":
        lay = _layout((case["nx"], case["ny"], case["nz"], case["cells"], case["r_min"], case["r_max"]))
        mu = np.full(len(lay), _flow(case)[3])
        if len(lay) > 8:  # a suspension: moduli of their own
            mu = np.exp(rng.uniform(math.log(2.6e-4), math.log(1.3e-3), len(lay)))
        kappa, w = case["kappa_mu"] * mu, np.full(len(lay), case["w"])
        noise = case["noise"]
    elif case["kind"] == "elastic":
        lay = [(case["radius"], np.array([30.0, 30.0, 30.0]))]
        mu, w, noise = np.exp(rng.uniform(-1.0, 1.0, 1)), rng.uniform(0.2, 0.9, 1), 0.05
        kappa = case["kappa_mu"] * mu
    else:
        r = case["radius"]
        lay = [(r, 3.0 * r * np.array([k % 4, (k // 4) % 4, k // 16])) for k in range(case["cells"])]
        mu = np.exp(rng.uniform(math.log(0.7), math.log(1.4), len(lay)))
        kappa, w = 20.0 * mu * rng.uniform(0.8, 1.25, len(lay)), rng.uniform(0.2, 0.9, len(lay))
        noise = 0.02
    xs, ts = [], []
    for r, c in lay:
        x, t = _mesh(r, case["h"])
        xs.append(x + c)
        ts.append(t)
    stretch = np.eye(3) + 0.03 * rng.uniform(-1.0, 1.0, (3, 3)) if case["kind"] == "elastic" else np.eye(3)
    ys = [c + (x - c) @ stretch.T + noise * rng.uniform(-1.0, 1.0, x.shape) for x, (_, c) in zip(xs, lay)]
    return xs, ts, ys, mu, kappa, w


def _protocol(case, xs):
    z_lo = np.array([x[:, 2].min() for x in xs])
    radius = np.array([0.5 * (x[:, 2].max() - x[:, 2].min()) for x in xs])
    return dict(z_lo=z_lo, radius=radius, strains=[0.05 * (k + 1) for k in range(case["levels"])], steps=case["steps"], ramp=case["ramp"])


DT, DAMPING, K_PLATE = 0.03, 0.95, 50.0


def prepare(case, seed):
    xs, ts, ys, mu, kappa, w = _cells(case, seed)
    rng = np.random.Generator(np.random.PCG64([seed, 2]))
    ctx = P.cf_create(0)
    s = dict(case=case, ctx=ctx, x=torch.from_numpy(np.concatenate(xs)), y=np.concatenate(ys))
    s["out"] = np.empty_like(s["y"])
    ids = P.cf_mesh_init_batch(ctx, xs, ts, ys)
    P.cf_set_materials(ctx, ids, mu, kappa, w)
    if case["kind"] == "coupled":
        lo, hi, g, _ = _flow(case)
        box = (case["nx"], case["ny"], case["nz"], TAU, lo, hi, (g, 0.0, 0.0))
        P.cf_set_population_format(ctx, case["fmt"])
        P.cf_set_delta(ctx, case["delta"])
        P.cf_set_spread(ctx, case["spread"])
        P.cf_lbm_init(ctx, *box)
        if case["tune"]:  # the launch shape, found once; then the fluid starts at rest
            P.cf_autotune(ctx, 10)
            P.cf_set_positions(ctx, P.CF_ALL_CELLS, s["y"])
            P.cf_lbm_init(ctx, *box)
        P.cf_prepare_steps(ctx, case["steps"])
        if case["field"]:
            s["field"] = np.zeros((case["nz"], case["ny"], case["nx"], 3))
    elif case["kind"] == "elastic":
        s["v"], s["lam"] = rng.normal(size=s["y"].shape), rng.normal(size=s["y"].shape)
        s["id"] = ids[0]
    else:
        p = _protocol(case, xs)
        s["run"] = Compression(ctx, ids, s["y"], p["z_lo"], p["radius"], p["strains"], p["steps"], DT, K_PLATE, p["ramp"], DAMPING)
        s["theta"] = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (mu, kappa, w)]
        s["dF"] = torch.from_numpy(rng.uniform(0.5, 1.5, (len(xs), case["levels"])))
    return s


def _moved(s):
    return (torch.from_numpy(s["out"]) - s["x"]).float()


def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "coupled":
        P.cf_step_exchange(ctx, case["steps"], s["y"], out=s["out"])
        if not case["field"]:
            return {"u": _moved(s)}
        return {"u": _moved(s), "velocity": torch.from_numpy(P.cf_get_velocity(ctx, out=s["field"])).float()}
    if case["kind"] == "elastic":
        P.cf_set_positions(ctx, s["id"], s["y"])
        P.cf_compute_forces(ctx)
        f = P.cf_get_forces(ctx, s["id"], out=s["out"])
        return {"force": torch.from_numpy(f).float(), "energy": torch.tensor(P.cf_get_energy(ctx, s["id"])).float(),
                "jvp": torch.from_numpy(P.cf_force_jvp(ctx, s["v"])).float(),
                "moduli": torch.from_numpy(P.cf_force_param_vjp(ctx, s["lam"])).float(),
                "taylor": P.cf_get_taylor(ctx, s["id"]),
                "strain": torch.tensor(P.cf_get_cell_strain(ctx, s["id"], 2.0 * case["radius"])["d_max"]).float()}
    if not case["gradient"]:
        F = s["run"].run(*(t.detach().numpy() for t in s["theta"]), record=False)
        P.cf_get_positions(ctx, P.CF_ALL_CELLS, out=s["out"])
        return {"F": torch.from_numpy(F).float(), "u": _moved(s)}
    for t in s["theta"]:
        t.grad = None
    F = CompressionCurve.apply(*s["theta"], s["run"])
    F.backward(s["dF"])
    return {"F": F.detach().float(), **{k: t.grad.float() for k, t in zip(("mu", "kappa", "w"), s["theta"])}}


def _sizes(case):
    if case["kind"] == "coupled":
        lay = _layout((case["nx"], case["ny"], case["nz"], case["cells"], case["r_min"], case["r_max"]))
        m = [_mesh(r, case["h"]) for r, _ in lay]
    else:
        m = [_mesh(case["radius"], case["h"])] * case.get("cells", 1)
    return sum(len(x) for x, _ in m), sum(len(t) for _, t in m)


def work(case):
    """Per coupled step every population read and written once, per force evaluation the mesh read once (indices, B, V_0: 56 bytes a
    tet) and positions read and written; about 300 operations a tet and 250 a node."""
    nv, nt = _sizes(case)
    if case["kind"] == "coupled":
        n = case["nx"] * case["ny"] * case["nz"]
        pop = 4 if case["fmt"] == "f32" else 2
        nodes = (4 if case["delta"] == "peskin4" else 2) ** 3
        per = n * 38 * pop + nt * 56 + nv * 24
        io = nv * 48 + (24 * n if case["field"] else 0)
        return {"bytes": case["steps"] * per + io, "flops": case["steps"] * (250 * n + 300 * nt + 14 * nodes * nv)}
    if case["kind"] == "elastic":  # forces, energy, Jacobian product, moduli gradient, Taylor moments; positions, forces, directions in and out
        return {"bytes": 4 * nt * 56 + nt * 16 + 5 * nv * 24, "flops": nt * (300 + 150 + 700 + 400 + 80)}
    steps = case["levels"] * case["steps"]
    evals = steps * (3 if case["gradient"] else 1)  # forward, recomputed, and the reverse step (twice the operations)
    return {"bytes": evals * (nt * 56 + nv * 48) + nv * 48, "flops": (steps * 300 + (steps * 1400 if case["gradient"] else 0)) * nt}


# ---------------------------------------------------------------- 64 bits
def _mm(a, b, t=False):
    """a b, or a^T b, of 3 x 3 matrices in the last two axes."""
    return sum((a[:, k, :, None] if t else a[:, :, k, None]) * b[:, k, None, :] for k in range(3))


class _Mesh64:
    """Mooney-Rivlin cells in 64 bits: oriented tets, B = J^-1, V_0 and moduli per tet."""

    def __init__(self, xs, ts, mu, kappa, w, dev):
        off = np.cumsum([0] + [len(x) for x in xs])
        x = torch.tensor(np.concatenate(xs), dtype=torch.float64, device=dev)
        t = torch.tensor(np.concatenate([t + o for t, o in zip(ts, off)]).astype(np.int64), device=dev)
        J = (x[t[:, :3]] - x[t[:, 3:]]).transpose(1, 2)
        flip = torch.linalg.det(J) < 0
        t[flip] = t[flip][:, [1, 0, 2, 3]]
        J = (x[t[:, :3]] - x[t[:, 3:]]).transpose(1, 2)
        self.x, self.t, self.V0, self.B = x, t, torch.linalg.det(J) / 6.0, torch.linalg.inv(J)
        self.corner = [t[:, k].contiguous() for k in range(4)]
        self.cell = torch.tensor(np.repeat(np.arange(len(ts)), [len(q) for q in ts]), device=dev)
        self.vcell = torch.tensor(np.repeat(np.arange(len(xs)), [len(q) for q in xs]), device=dev)
        self.theta = [torch.tensor(np.asarray(q), dtype=torch.float64, device=dev) for q in (mu, kappa, w)]

    def _parts(self, y):
        p = [y.index_select(0, k) for k in self.corner]
        F = sum((p[k] - p[3])[:, :, None] * self.B[:, k, None, :] for k in range(3))
        r = [F[:, k].roll(-1, 1) for k in range(3)], [F[:, k].roll(-2, 1) for k in range(3)]
        cof = torch.stack([r[0][(k + 1) % 3] * r[1][(k + 2) % 3] - r[1][(k + 1) % 3] * r[0][(k + 2) % 3] for k in range(3)], 1)
        J = (F[:, 0] * cof[:, 0]).sum(1)
        return F, cof, J, (F * F).sum((1, 2)), _mm(F, F, True)

    def energy(self, y):
        mu, k, w = (q[self.cell] for q in self.theta)
        F, _, J, TC, C = self._parts(y)
        I, K = TC * J ** (-2.0 / 3.0), 0.5 * (TC**2 - (C * C).sum((1, 2))) * J ** (-4.0 / 3.0)
        return (self.V0 * (0.5 * w * mu * (I - 3.0) + 0.5 * (1.0 - w) * mu * (K - 3.0) + 0.5 * k * (J - 1.0) ** 2)).sum()

    def forces(self, y):
        """-dE/dy, written out."""
        mu, k, w = (q[self.cell][:, None, None] for q in self.theta)
        F, cof, J, TC, C = self._parts(y)
        J, TC = J[:, None, None], TC[:, None, None]
        T2 = TC**2 - (C * C).sum((1, 2))[:, None, None]
        G = cof / J  # F^-T
        S = w * mu * J ** (-2.0 / 3.0) * (F - TC / 3.0 * G) + (1.0 - w) * mu * J ** (-4.0 / 3.0) * (TC * F - _mm(F, C) - T2 / 3.0 * G)
        S = (S + k * (J - 1.0) * cof) * -self.V0[:, None, None]
        f = [(S * self.B[:, k, None, :]).sum(2) for k in range(3)]
        f, out = [*f, -f[0] - f[1] - f[2]], torch.zeros_like(y)
        for k in range(4):
            out = out.index_add(0, self.corner[k], f[k])
        return out


_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
_C += [c for c in ((a, b, d) for a in (-1, 0, 1) for b in (-1, 0, 1) for d in (-1, 0, 1)) if sum(map(abs, c)) == 2]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _stream_collide(d, F, g, lo, hi):
    """Pull, bounce back off the moving walls, collide (BGK, Guo forcing); populations less their weights, [19, nz, ny, nx]."""
    new = torch.empty_like(d)
    for q, c in enumerate(_C):
        s = torch.roll(d[q], (c[2], c[0]), (0, 2))
        back = d[_C.index(tuple(-a for a in c))]
        if c[1] == 1:
            new[q][:, 1:], new[q][:, 0] = s[:, :-1], back[:, 0] + 6.0 * _W[q] * c[0] * lo
        elif c[1] == -1:
            new[q][:, :-1], new[q][:, -1] = s[:, 1:], back[:, -1] + 6.0 * _W[q] * c[0] * hi
        else:
            new[q] = s
    F = [F[0] + g, F[1], F[2]]
    drho = new.sum(0)
    u = [(sum(c[a] * new[q] for q, c in enumerate(_C) if c[a]) + 0.5 * F[a]) / (1.0 + drho) for a in range(3)]
    uu, uF = sum(a * a for a in u), sum(a * b for a, b in zip(u, F))
    for q, c in enumerate(_C):
        zero = torch.zeros((), dtype=d.dtype, device=d.device)
        cu, cF = sum((c[a] * u[a] for a in range(3) if c[a]), zero), sum((c[a] * F[a] for a in range(3) if c[a]), zero)
        eq = _W[q] * (drho + (1.0 + drho) * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))
        new[q] += (eq - new[q]) / TAU + (1.0 - 0.5 / TAU) * _W[q] * (3.0 * (cF - uF) + 9.0 * cu * cF)
    return new, torch.stack(u, -1)


def _phi(r, width):
    r = r.abs()
    if width == 2:
        return (1.0 - r).clamp(min=0.0)
    near = (3.0 - 2.0 * r + (1.0 + 4.0 * r - 4.0 * r * r).clamp(min=0.0).sqrt()) / 8.0
    far = (5.0 - 2.0 * r - (-7.0 + 12.0 * r - 4.0 * r * r).clamp(min=0.0).sqrt()) / 8.0
    return torch.where(r <= 1.0, near, torch.where(r <= 2.0, far, torch.zeros_like(r)))


def _exact_coupled(case, seed):
    xs, ts, ys, mu, kappa, w = _cells(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    nx, ny, nz, steps = case["nx"], case["ny"], case["nz"], case["steps"]
    if steps * (nx * ny * nz + 2e5) > 4.0e9:  # over some 20 seconds
        return None
    m = _Mesh64(xs, ts, mu, kappa, w, dev)
    y = torch.tensor(np.concatenate(ys), dtype=torch.float64, device=dev)
    lo, hi, g, _ = _flow(case)
    d = torch.zeros((19, nz, ny, nx), dtype=torch.float64, device=dev)
    width = 4 if case["delta"] == "peskin4" else 2
    k = torch.arange(width, device=dev) - (width // 2 - 1)
    for _ in range(steps):
        f = m.forces(y)
        base = torch.floor(y)
        at = [base[:, a : a + 1].long() + k for a in range(3)]
        wt = [_phi(y[:, a : a + 1] - at[a], width) for a in range(3)]
        node = (at[0] % nx)[:, None, None, :] + nx * (at[1][:, None, :, None] + ny * (at[2] % nz)[:, :, None, None])
        wgt = wt[2][:, :, None, None] * wt[1][:, None, :, None] * wt[0][:, None, None, :]
        node, wgt = node.reshape(len(y), -1), wgt.reshape(len(y), -1)
        F = [torch.zeros(nx * ny * nz, dtype=torch.float64, device=dev).index_add(0, node.reshape(-1), (wgt * f[:, a : a + 1]).reshape(-1)).reshape(nz, ny, nx)
             for a in range(3)]
        d, u = _stream_collide(d, F, g, lo, hi)
        y = y + (u.reshape(-1, 3)[node] * wgt[:, :, None]).sum(1)
    out = {"u": (y - m.x).cpu()}
    if case["field"]:
        out["velocity"] = u.cpu()
    return out


def _exact_elastic(case, seed):
    xs, ts, ys, mu, kappa, w = _cells(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    m = _Mesh64(xs, ts, mu, kappa, w, dev)
    rng = np.random.Generator(np.random.PCG64([seed, 2]))
    y = torch.tensor(np.concatenate(ys), dtype=torch.float64, device=dev)
    v, lam = (torch.tensor(rng.normal(size=tuple(y.shape)), device=dev) for _ in range(2))
    for q in m.theta:
        q.requires_grad_(True)
    y.requires_grad_(True)
    f = m.forces(y)
    jvp, = torch.autograd.grad((f * v).sum(), y, retain_graph=True)  # the Jacobian is symmetric
    moduli = torch.stack([q.reshape(()) for q in torch.autograd.grad((f * lam).sum(), m.theta)])[None]
    y = y.detach()
    p = y[m.t]
    vol = torch.linalg.det(p[:, :3] - p[:, 3:]).abs() / 6.0
    c = p.mean(1)
    c = c - (vol[:, None] * c).sum(0) / vol.sum()
    S = torch.einsum("l,li,lj->ij", vol, c, c)
    th, vec = np.linalg.eigh((torch.eye(3, dtype=S.dtype, device=dev) * S.trace() - S).cpu().numpy())
    th, M = th[::-1], float(vol.sum())
    a2 = 2.5 / M * np.array([-th[0] + th[1] + th[2], th[0] - th[1] + th[2], th[0] + th[1] - th[2]])
    a = np.sqrt(a2)
    ang = math.degrees(math.atan2(vec[1, 0], vec[0, 0]))
    ang += 180.0 if ang <= -90.0 else -180.0 if ang > 90.0 else 0.0
    far = max(float(torch.cdist(q, y).max()) for q in y.split(4096))
    return {"force": f.detach().cpu(), "energy": float(m.energy(y).detach()), "jvp": jvp.cpu(), "moduli": moduli.detach().cpu(), "strain": far,
            "taylor": {"D": (a[2] - a[0]) / (a[2] + a[0]), "D_literal": (a2[2] - a2[0]) / (a2[2] + a2[0]), "inclination": ang, "a1": a[0], "a2": a[1],
                       "a3": a[2], "theta1": th[0], "theta2": th[1], "theta3": th[2], "volume": M}}


def _exact_compress(case, seed):
    xs, ts, ys, mu, kappa, w = _cells(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    m = _Mesh64(xs, ts, mu, kappa, w, dev)
    rng = np.random.Generator(np.random.PCG64([seed, 2]))
    dF = torch.tensor(rng.uniform(0.5, 1.5, (len(xs), case["levels"])), device=dev)
    p = _protocol(case, xs)
    y = torch.tensor(np.concatenate(ys), dtype=torch.float64, device=dev)
    v, z_lo = torch.zeros_like(y), torch.tensor(p["z_lo"], device=dev)[m.vcell]
    trail, F = [], []
    for z_hi, n, measured in plate_schedule(p["z_lo"], p["radius"], p["strains"], p["steps"], p["ramp"]):
        top = torch.tensor(z_hi, device=dev)[m.vcell]
        for k in range(n):
            trail.append((y, top, False))
            f = m.forces(y)
            f[:, 2] += K_PLATE * ((z_lo - y[:, 2]).clamp(min=0.0) - (y[:, 2] - top).clamp(min=0.0))
            v = DAMPING * v + DT * f
            y = y + DT * v
        if measured:
            trail.append((y, top, True))
            F.append(torch.zeros(len(xs), dtype=y.dtype, device=dev).index_add(0, m.vcell, K_PLATE * (y[:, 2] - top).clamp(min=0.0)))
    out = {"F": torch.stack(F, 1).cpu()}
    if not case["gradient"]:
        return {**out, "u": (y - m.x).cpu()}
    for q in m.theta:
        q.requires_grad_(True)
    ly, lv = torch.zeros_like(y), torch.zeros_like(y)
    grad, level = [torch.zeros_like(q) for q in m.theta], case["levels"]
    for y, top, measured in reversed(trail):
        if measured:
            level -= 1
            ly[:, 2] += dF[m.vcell, level] * K_PLATE * (y[:, 2] > top)
            continue
        mm = DT * ly + lv
        y = y.detach().requires_grad_(True)
        gy, *gt = torch.autograd.grad((m.forces(y) * mm).sum(), [y, *m.theta])
        gy[:, 2] -= K_PLATE * mm[:, 2] * ((y < z_lo[:, None])[:, 2] | (y[:, 2] > top))
        grad = [a + DT * b for a, b in zip(grad, gt)]
        ly, lv = ly + DT * gy, DAMPING * mm
    return {**out, **{k: q.cpu() for k, q in zip(("mu", "kappa", "w"), grad)}}


def exact(case, seed):
    return {"coupled": _exact_coupled, "elastic": _exact_elastic, "compress": _exact_compress}[case["kind"]](case, seed)
