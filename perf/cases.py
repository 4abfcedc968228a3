"""The measured work of the wall-stress stage: what a time step asks of the library, over its sizes,
precisions and options.

`listed` gives the cases, `draw` more of the same ranges; `prepare` makes the device fields, the terrain's
handle and the plans a solver keeps; `run` is one pass through the package's calls; `work` is the least
that a pass moves and computes; `exact` is the same result in 64-bit torch arithmetic, written from the
equations alone.  Grid sizes and flow parameters are those of the package's seeded workloads
(paper_2006_03343_gb300/inputs.py) and of its tests.

All fields are [nz, ny, nx] with x fastest; uv-nodes at (i dx, j dy, (k + 1/2) dz), w-nodes at
(i dx, j dy, k dz), dz = lz/(nz - 1); x and y are periodic.
"""
import math
import random

import numpy as np
import torch

from paper_2006_03343_gb300 import autograd, wmibm

KAPPA = 0.4
Z0 = 1e-4
SMAGORINSKY = 0.16
DT = 1e-3
ENSEMBLE_SHAPES = ((64, 64, 64), (128, 64, 64), (192, 96, 96), (256, 128, 64))
TORCH_TYPE = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}
UV, W = (0, 1, 2, 3), (4, 5)            # stress components on uv-nodes (txx, txy, tyy, tzz), on w-nodes (txz, tyz)
MAX_NODES = 512 * 256 * 256


def _case(name, kind, shape, terrain, dtype="f32", vel="", **more):
    nx, ny, nz = shape
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "terrain": terrain, "dtype": dtype,
            "vel": vel or dtype, **more}


def listed():
    return [
        # a small two-dimensional ridge in double precision with the band statistics a solver logs each
        # step: the smallest call, launches and latency
        _case("step_ridge_f64", "step", (32, 32, 32), "ridge", "f64", stats=True),
        # a grid whose rows are no multiple of a vector, with the pressure gradient of Eq. 27 and statistics
        _case("step_ragged_f32", "step", (150, 90, 75), "hills", stats=True, gradp=True),
        # the wall-mounted cube array: an ordinary single-terrain step in single precision
        _case("step_cubes_f32", "step", (256, 128, 128), "cubes"),
        # the large hill with per-cell roughness and the velocity stored in 16 bits
        _case("step_hill_bf16", "step", (512, 256, 256), "hill", "f32", "bf16", z0_field=True),
        # the same stage in double precision on rolling terrain
        _case("step_hills_f64", "step", (256, 128, 128), "hills", "f64"),
        # 64 terrains of uneven grids stepped together
        {"name": "batch_ensemble_f32", "kind": "batch", "members": 64, "mix": 4000, "dtype": "f32", "vel": "f32"},
        # the forcing with the paper's pseudo-spectral horizontal derivatives, both precisions
        _case("spectral_hill_f32", "spectral", (512, 256, 256), "hill"),
        _case("spectral_hills_f64", "spectral", (256, 128, 128), "hills", "f64"),
        # from the velocity to the forcing: sub-grid stress, wall model, divergence
        _case("sgs_chain_cubes_f32", "sgs_chain", (256, 128, 128), "cubes"),
        # the same with the sub-grid stress formed inside the divergence, large terrain
        _case("sgs_fused_hill_f32", "sgs_fused", (512, 256, 256), "hill"),
        # forward and backward of the stage as a differentiable layer (velocity and log-roughness gradients)
        _case("adjoint_hills_f32", "adjoint", (256, 128, 128), "hills", z0_field=True),
        # the exact signed distance of a terrain's height field, computed when the terrain is set
        _case("sdf_hill_f64", "sdf", (512, 256, 256), "hill", "f64", reach=4.0),
    ]


def _size(rng, lo, hi, step=1):
    """A whole number in [lo, hi], a multiple of step, spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "batch", "spectral", "sgs_chain", "sgs_fused", "adjoint", "sdf"))
    dtype = rng.choice(("f32", "f32", "f32", "f64"))
    vel = rng.choice(("f32", "f32", "bf16")) if dtype == "f32" else "f64"
    if kind == "batch":
        return {"kind": kind, "members": _size(rng, 2, 64 if dtype == "f32" else 12), "mix": rng.randrange(1 << 20),
                "dtype": dtype, "vel": vel}
    if kind == "spectral":
        most = MAX_NODES if dtype == "f32" else MAX_NODES // 8
        nx, ny = 1 << rng.randrange(5, 11), 1 << rng.randrange(5, 10)
        nz = _size(rng, 17, max(17, min(256, most // (nx * ny))))
        return _drawn(kind, nx, ny, nz, rng.choice(("hill", "hills")), dtype, dtype)
    if kind == "sdf":
        nx, ny = _size(rng, 32, 512), _size(rng, 32, 256)
        nz = _size(rng, max(32, nx // 4), 256)      # the window within reach stays a few cells wide
        return _drawn(kind, nx, ny, nz, rng.choice(("ridge", "hill", "hills")), "f64", "f64",
                      reach=round(rng.uniform(2.0, 5.0), 2))
    most = MAX_NODES if dtype == "f32" else MAX_NODES // 8
    if kind == "adjoint":
        most //= 4
    step = rng.choice((1, 2, 4, 32))                # any row length, or rows of whole vectors or lines
    nx, ny = _size(rng, 32, 512, step), _size(rng, 17, 256)
    nz = _size(rng, 17, max(17, min(256, most // (nx * ny))))
    terrain = rng.choice(("ridge", "hill", "hills", "cubes"))
    if kind == "step":
        return _drawn(kind, nx, ny, nz, terrain, dtype, vel, stats=dtype == "f64" and rng.random() < 0.5,
                      gradp=rng.random() < 0.5, z0_field=rng.random() < 0.3)
    if kind == "adjoint":
        return _drawn(kind, nx, ny, nz, "hills", dtype, dtype, z0_field=True)
    return _drawn(kind, nx, ny, nz, terrain, dtype, vel)


def _drawn(kind, nx, ny, nz, terrain, dtype, vel, **more):
    case = _case("", kind, (nx, ny, nz), terrain, dtype, vel, **more)
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------------------- #
# inputs
# ---------------------------------------------------------------------------------------------------- #
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Draws:
    """Normal deviates on the device from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=_device())
        self.g.manual_seed(int(seed) * 7919 + 17)

    def normal(self, shape, sigma=1.0, dtype=torch.float32):
        x = torch.empty(shape, dtype=dtype, device=_device())
        return x.normal_(0.0, sigma, generator=self.g)


def _grid(case):
    lx, ly = (4.0, 2.0) if case["terrain"] == "cubes" else (2 * math.pi, math.pi)
    return case["nx"], case["ny"], case["nz"], lx, ly, 1.0


def _near(d, period):
    return d - period * torch.round(d / period)


def _heights(grid, terrain, rng):
    """h[ny, nx] of a ridge, a round hill or one to eight Gaussian hills (Eqs. 31, 32), at a place drawn by rng."""
    nx, ny, nz, lx, ly, lz = grid
    x = torch.arange(nx, dtype=torch.float64, device=_device()) * (lx / nx)
    y = torch.arange(ny, dtype=torch.float64, device=_device()) * (ly / ny)
    cx, cy = rng.randrange(nx) * (lx / nx), rng.randrange(ny) * (ly / ny)
    if terrain == "ridge":
        r = _near(x - cx, lx).abs()
        h = torch.where(r < 0.3, 0.1 * torch.cos(math.pi * r / 0.6) ** 2, torch.zeros_like(r))
        return h[None, :].expand(ny, nx).contiguous()
    if terrain == "hill":
        r = torch.sqrt(_near(x - cx, lx)[None, :] ** 2 + _near(y - cy, ly)[:, None] ** 2)
        return torch.where(r < 0.5, 0.13 * torch.cos(math.pi * r) ** 2, torch.zeros_like(r))
    h = torch.zeros((ny, nx), dtype=torch.float64, device=_device())
    for _ in range(rng.randint(1, 8)):
        a, wd = rng.uniform(0.02, 0.2) / 2, rng.uniform(0.05, 0.4)
        cx, cy = rng.uniform(0.0, lx), rng.uniform(0.0, ly)
        h += a * torch.exp(-(_near(x - cx, lx)[None, :] ** 2 + _near(y - cy, ly)[:, None] ** 2) / (2 * wd * wd))
    return h


def _levels(grid):
    nz, dz = grid[2], grid[5] / (grid[2] - 1)
    k = torch.arange(nz, dtype=torch.float64, device=_device())
    return (k + 0.5) * dz, k * dz


def _distance(grid, terrain, rng):
    """phi on the uv-grid and the w-grid: z - h, or the distance to 4 x 4 wall-mounted cubes of side 0.25."""
    z = _levels(grid)
    if terrain != "cubes":
        h = _heights(grid, terrain, rng)
        return [t[:, None, None] - h[None] for t in z]
    nx, ny, nz, lx, ly, lz = grid
    side, sx, sy = 0.25, rng.randrange(nx) * (lx / nx), rng.randrange(ny) * (ly / ny)
    x = torch.arange(nx, dtype=torch.float64, device=_device()) * (lx / nx)
    y = torch.arange(ny, dtype=torch.float64, device=_device()) * (ly / ny)
    # the nearest cube in x and in y: centres at 0.5, 1.5, ... and 0.25, 0.75, ..., shifted together
    qx = (_near(x - 0.5 - sx, 1.0).abs() - side / 2)[None, None, :]
    qy = (_near(y - 0.25 - sy, 0.5).abs() - side / 2)[None, :, None]
    out = []
    for t in z:
        qz = (t - side)[:, None, None]
        far = torch.sqrt(qx.clamp(min=0) ** 2 + qy.clamp(min=0) ** 2 + qz.clamp(min=0) ** 2)
        out.append(far + torch.maximum(torch.maximum(qx, qy), qz).clamp(max=0))
    return out


class _Terrain:
    """One terrain's geometry and fields, made from the seed alone."""

    def __init__(self, case, seed, grid=None, terrain=None, phi_c_cells=1.5, z0=Z0):
        rng = random.Random(int(seed) * 104729 + 5)
        d = _Draws(seed)
        self.grid = grid or _grid(case)
        nx, ny, nz = self.grid[:3]
        self.shape = (nz, ny, nx)
        self.dz = self.grid[5] / (nz - 1)
        self.phi_c, self.phi_b = phi_c_cells * self.dz, 0.5 * self.dz
        self.phi = _distance(self.grid, terrain or case["terrain"], rng)
        self.z0 = z0
        if case.get("z0_field"):
            self.z0 = Z0 * torch.exp(d.normal(self.shape, 0.5, torch.float64))
        self.type, self.vel_type = TORCH_TYPE[case["dtype"]], TORCH_TYPE[case["vel"]]
        self.gradp = [d.normal(self.shape, 1.0, self.type) for _ in range(3)] if case.get("gradp") else None
        # log profile (Eq. 29) plus noise
        sigma = 0.15 if (terrain or case["terrain"]) == "cubes" else 0.1
        far = torch.maximum(self.phi[0], torch.as_tensor(self.z0, dtype=torch.float64, device=_device()))
        u = (1.0 / KAPPA) * torch.log(far / self.z0)
        vel = [u, 0.0, 0.0]
        for c in range(3):
            x = d.normal(self.shape, sigma, torch.float32).double() + vel[c]
            if case["kind"] in ("step", "batch"):
                # inside the body the velocity already holds the condition of Eq. 27, as after the last step
                body = self.phi[1 if c == 2 else 0] <= 0
                x = torch.where(body, 1.5 * DT * self.gradp[c].double() if self.gradp else 0.0, x)
            vel[c] = x.to(self.vel_type).contiguous()
        self.vel = vel
        self.tau = [d.normal(self.shape, 0.1, self.type) for _ in range(6)]

    def handle(self, case):
        z0 = self.z0 if isinstance(self.z0, float) else self.z0.cpu().numpy()
        return wmibm.Handle(self.grid, self.phi[0].cpu().numpy(), self.phi[1].cpu().numpy(), z0, self.phi_c, self.phi_b,
                            dtype=case["dtype"], vel_dtype=case["vel"] if case["vel"] == "bf16" else None)


def _members(case):
    r = random.Random(case["mix"])
    return [(r.choice(ENSEMBLE_SHAPES), r.uniform(1.0, 2.0), 10.0 ** r.uniform(-5.0, -3.0))
            for _ in range(case["members"])]


def _member(case, seed, m, spec):
    (nx, ny, nz), cells, z0 = spec
    return _Terrain(case, seed * 1009 + m, (nx, ny, nz, 2 * math.pi, math.pi, 1.0), "hills", cells, z0)


def _empty(t, n):
    return [torch.empty(t.shape, dtype=t.type, device=_device()) for _ in range(n)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sdf":
        grid = _grid(case)
        h = _heights(grid, case["terrain"], random.Random(int(seed) * 104729 + 5))
        phi = [torch.empty(case["nz"], case["ny"], case["nx"], dtype=torch.float64, device=_device()) for _ in range(2)]
        return {"kind": kind, "grid": grid, "h": h, "reach": case["reach"] / (case["nz"] - 1), "phi": phi}
    if kind == "batch":
        return _prepare_batch(case, seed)
    t = _Terrain(case, seed)
    s = {"kind": kind, "handle": t.handle(case), "vel": t.vel, "tau": t.tau, "f": _empty(t, 3)}
    h = s["handle"]
    if kind == "step":
        stats = h.new_stats() if case.get("stats") else None
        s["step"] = h.prepare_step(*t.vel, t.tau, s["f"], stats, t.gradp, DT if t.gradp else 0.0)
        s["out"] = {"vel": t.vel, "tau": t.tau, "f": s["f"]}
        if stats is not None:
            # counts, then sum tau_w, sum tau_w^2, min tau_w, max |U_r| of each band
            s["stats"] = stats.view(2, 6)[:, 1:5]
            s["out"]["count"] = stats.view(torch.int64).view(2, 6)[:, ::5]
            # a solver in single precision keeps its history of them in single precision
            s["log"] = torch.empty(2, 4, dtype=t.type, device=_device())
            s["out"]["stats"] = s["log"]
    elif kind == "spectral":
        s["step"] = h.prepare_step(*t.vel, t.tau, s["f"])
    elif kind in ("sgs_chain", "sgs_fused"):
        s["wt"] = h.sgs_wall_terms(t.phi[0].cpu().numpy(), t.phi[1].cpu().numpy(), t.z0)
        s["step"] = h.prepare_step(*t.vel, t.tau, s["f"])
    elif kind == "adjoint":
        s["vel"] = [x.requires_grad_() for x in t.vel]
        s["logz0"] = torch.log(t.z0).to(t.type).requires_grad_()
        s["g"] = [_Draws(seed + 501 + c).normal(t.shape, 1.0, t.type) for c in range(3)]
    return s


def _prepare_batch(case, seed):
    """The members' fields are views into one packed buffer for each kind of field."""
    members = [_member(case, seed, m, spec) for m, spec in enumerate(_members(case))]
    handles = [t.handle(case) for t in members]
    pack = lambda arrays: torch.cat([a.reshape(-1) for a in arrays])  # noqa: E731
    flat = [pack([t.vel[c] for t in members]) for c in range(3)] + [pack([t.tau[c] for t in members]) for c in range(6)]
    flat += [torch.empty(flat[3].numel(), dtype=flat[3].dtype, device=_device()) for _ in range(3)]
    fields, at = [], 0
    for t in members:
        n = t.vel[0].numel()
        v = [f[at:at + n].view(t.shape) for f in flat]
        fields.append((v[0], v[1], v[2], v[3:9], v[9:12]))
        at += n
    batch = wmibm.Batch(handles)
    batch.set_fields(fields)
    return {"kind": "batch", "handles": handles, "batch": batch, "fields": fields,
            "out": {"vel": flat[:3], "tau": flat[3:9], "f": flat[9:]}}


def run(state):
    kind = state["kind"]
    if kind == "step":
        state["step"].step()
        if "log" in state:
            state["log"].copy_(state["stats"])
        return state["out"]
    if kind == "batch":
        state["batch"].step()
        return state["out"]
    if kind == "spectral":
        state["step"].force_spectral()
        return state["f"]
    if kind == "sgs_chain":
        state["handle"].sgs_stress(*state["vel"], state["wt"], state["tau"], SMAGORINSKY)
        state["step"].wall_stress_force()
        return {"tau": state["tau"], "f": state["f"]}
    if kind == "sgs_fused":
        state["step"].wall_stress()
        state["handle"].sgs_force(*state["vel"], state["wt"], state["tau"], state["f"], SMAGORINSKY)
        return {"tau": state["tau"], "f": state["f"]}
    if kind == "adjoint":
        wrt = [*state["vel"], state["logz0"]]
        f = autograd.wall_stress_force(state["handle"], *wrt, state["tau"])
        return {"f": f, "grad": torch.autograd.grad(f, wrt, state["g"])}
    return wmibm.heightfield_sdf(state["grid"], state["h"], state["reach"], *state["phi"])


# ---------------------------------------------------------------------------------------------------- #
# least work of a pass
# ---------------------------------------------------------------------------------------------------- #
def work(case):
    """Bytes: each whole field that the pass reads or writes, once; the band's few percent are left out."""
    e = 8 if case["dtype"] == "f64" else 4
    ve = {"f64": 8, "f32": 4, "bf16": 2}[case["vel"]]
    kind = case["kind"]
    if kind == "batch":
        n = sum(nx * ny * nz for (nx, ny, nz), _, _ in _members(case))
        return {"bytes": 9.0 * e * n, "flops": 18.0 * n}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "step":                              # six stresses in, three forcing components out
        return {"bytes": 9.0 * e * n, "flops": 18.0 * n}
    if kind == "spectral":                          # and six transforms there and back, two real lines in each
        lines = 3 * (math.log2(case["nx"]) + math.log2(case["ny"]))
        return {"bytes": 9.0 * e * n, "flops": n * (5.0 * lines + 18.0)}
    if kind == "sgs_chain":                         # velocity and wall terms in, stresses and forcing out
        return {"bytes": (3.0 * ve + 11.0 * e) * n, "flops": 110.0 * n}
    if kind == "sgs_fused":                         # the stresses are never written
        return {"bytes": (3.0 * ve + 5.0 * e) * n, "flops": 110.0 * n}
    if kind == "adjoint":                           # forward as above; four gradients written
        return {"bytes": (9.0 * e + 3.0 * ve + e) * n, "flops": 18.0 * n}
    return {"bytes": 16.0 * n + 8.0 * case["nx"] * case["ny"], "flops": 2.0 * n}


# ---------------------------------------------------------------------------------------------------- #
# the same results in 64 bits
# ---------------------------------------------------------------------------------------------------- #
def _dx(a, grid):
    return (torch.roll(a, -1, 2) - torch.roll(a, 1, 2)) * (grid[0] / (2.0 * grid[3]))


def _dy(a, grid):
    return (torch.roll(a, -1, 1) - torch.roll(a, 1, 1)) * (grid[1] / (2.0 * grid[4]))


def _spectral(a, length, dim):
    """Eq. 13's derivative along one direction; the Nyquist mode has none."""
    n = a.shape[dim]
    k = torch.fft.rfftfreq(n, d=length / n, dtype=torch.float64, device=a.device) * (2 * math.pi)
    if n % 2 == 0:
        k[-1] = 0.0
    shape = [1, 1, 1]
    shape[dim] = k.numel()
    return torch.fft.irfft(torch.fft.rfft(a, dim=dim) * (1j * k.view(shape)), n=n, dim=dim)


def _divergence(tau, grid, dx=_dx, dy=_dy):
    """f = -div tau (Eq. 18): zero on the ghost uv-level and on the floor and lid w-levels."""
    txx, txy, tyy, tzz, txz, tyz = tau
    rdz = (grid[2] - 1) / grid[5]
    up = lambda a: torch.nn.functional.pad((a[1:] - a[:-1]) * rdz, (0, 0, 0, 0, 0, 1))  # noqa: E731
    uv = torch.ones(grid[2], 1, 1, dtype=torch.float64, device=txx.device)
    uv[-1] = 0.0
    w = uv.clone()
    w[0] = 0.0
    down = torch.nn.functional.pad((tzz[1:] - tzz[:-1]) * rdz, (0, 0, 0, 0, 1, 0))
    return [-(dx(txx, grid) + dy(txy, grid) + up(txz)) * uv, -(dx(txy, grid) + dy(tyy, grid) + up(tyz)) * uv,
            -(dx(txz, grid) + dy(tyz, grid) + down) * w]


def _normals(phi, grid, at):
    """grad(phi)/|grad(phi)| at the nodes `at`: central differences, one-sided at the first and last level."""
    nx, ny, nz, lx, ly, lz = grid
    k, j, i = at
    p = phi.reshape(-1)
    idx = lambda kk, jj, ii: p[(kk * ny + jj % ny) * nx + ii % nx]  # noqa: E731
    gx = (idx(k, j, i + 1) - idx(k, j, i - 1)) * (nx / (2.0 * lx))
    gy = (idx(k, j + 1, i) - idx(k, j - 1, i)) * (ny / (2.0 * ly))
    k1, k0 = (k + 1).clamp(max=nz - 1), (k - 1).clamp(min=0)
    gz = (idx(k1, j, i) - idx(k0, j, i)) / ((k1 - k0).double() * (lz / (nz - 1)))
    size = torch.sqrt(gx * gx + gy * gy + gz * gz)
    flat = size == 0
    size = torch.where(flat, torch.ones_like(size), size)
    return torch.where(flat, 0.0, gx / size), torch.where(flat, 0.0, gy / size), torch.where(flat, 1.0, gz / size)


def _sample(field, grid, x, y, level, top):
    """Trilinear value at (x, y) and the fractional level, clamped to 0 .. top."""
    nx, ny, nz, lx, ly, lz = grid
    fx, fy, fz = x * (nx / lx), y * (ny / ly), level.clamp(0.0, float(top))
    i, j, k = fx.floor(), fy.floor(), fz.floor().clamp(max=top - 1)
    ax, ay, az = fx - i, fy - j, fz - k
    i, j, k = i.long(), j.long(), k.long()
    p, total = field.reshape(-1), 0.0
    for c in range(8):
        a, b, e = c & 1, (c >> 1) & 1, c >> 2
        wt = (ax if a else 1 - ax) * (ay if b else 1 - ay) * (az if e else 1 - az)
        total = total + wt * p[((k + e) * ny + (j + b) % ny) * nx + (i + a) % nx]
    return total


def _wall(t, vel, tau, logz0=None):
    """The wall model (Sec. 3.3) over all band nodes; returns the new stresses and the band statistics."""
    nx, ny, nz, lx, ly, lz = t.grid
    dx, dy, dz = lx / nx, ly / ny, t.dz
    tau, rows, counts = list(tau), [], []
    for on_w in (True, False):
        phi = t.phi[1 if on_w else 0]
        band = (phi.abs() <= t.phi_b) if on_w else (phi >= 0) & (phi <= 2 * t.phi_b)
        solid = phi < (-t.phi_b if on_w else 0.0)
        at = torch.nonzero(band, as_tuple=True)
        k, j, i = at
        n = _normals(phi, t.grid, at)
        s = t.phi_c - phi[band]
        z = (k.double() + (0.0 if on_w else 0.5)) * dz
        x, y, z = i.double() * dx + s * n[0], j.double() * dy + s * n[1], z + s * n[2]
        vals = [_sample(vel[0], t.grid, x, y, z / dz - 0.5, nz - 2), _sample(vel[1], t.grid, x, y, z / dz - 0.5, nz - 2),
                _sample(vel[2], t.grid, x, y, z / dz, nz - 1)]
        un = vals[0] * n[0] + vals[1] * n[1] + vals[2] * n[2]
        ur = [vals[c] - un * n[c] for c in range(3)]
        speed = torch.sqrt(ur[0] ** 2 + ur[1] ** 2 + ur[2] ** 2)
        if logz0 is not None:
            ln = math.log(t.phi_c) - logz0[band]
        elif isinstance(t.z0, float):
            ln = math.log(t.phi_c / t.z0)
        else:
            ln = torch.log(t.phi_c / t.z0[band])
        c = (KAPPA / ln) ** 2
        tw = -c * speed ** 2
        pairs = ((4, 0, 2), (5, 1, 2)) if on_w else ((0, 0, 0), (1, 0, 1), (2, 1, 1), (3, 2, 2))
        for comp, a, b in pairs:
            v = -c * speed * (ur[a] * n[b] + n[a] * ur[b])
            flat = torch.where(solid, 0.0, tau[comp]).reshape(-1)
            tau[comp] = flat.index_put((torch.nonzero(band.reshape(-1))[:, 0],), v).reshape(t.shape)
        some = tw.numel() > 0
        rows.append([tw.sum(), (tw * tw).sum(), tw.min() if some else tw.sum(), speed.max() if some else tw.sum()])
        over = (z / dz - 0.5 < 0) | (z / dz - 0.5 > nz - 2) | (z / dz < 0) | (z / dz > nz - 1)
        counts.append([tw.numel(), int(over.sum())])
    return tau, torch.stack([torch.stack(r) for r in rows]).detach(), counts


def _step(t, case):
    vel = [v.double() for v in t.vel]
    tau, stats, counts = _wall(t, vel, [x.double() for x in t.tau])
    f = _divergence(tau, t.grid)
    for c in range(3):
        body = t.phi[1 if c == 2 else 0] <= 0
        vel[c] = torch.where(body, 1.5 * DT * t.gradp[c].double() if t.gradp else 0.0, vel[c])
    out = {"vel": vel, "tau": tau, "f": f}
    if case.get("stats"):
        out["count"] = torch.tensor(counts)
        out["stats"] = stats
    return out


def _sgs(t):
    """Smagorinsky's stress with Mason's damping (Eqs. 4-7) at fluid nodes, the given stress elsewhere."""
    nx, ny, nz, lx, ly, lz = t.grid
    g, rdz = t.grid, 1.0 / t.dz
    u, v, w = (x.double() for x in t.vel)
    lam0 = 1.0 / (SMAGORINSKY * (lx / nx * ly / ny * t.dz) ** (1.0 / 3.0)) ** 2
    s11, s22, s12 = _dx(u, g)[:-1], _dy(v, g)[:-1], 0.5 * (_dy(u, g) + _dx(v, g))[:-1]
    s33 = (w[1:] - w[:-1]) * rdz                    # uv-levels 0 .. nz-2
    s13 = 0.5 * ((u[1:-1] - u[:-2]) * rdz + _dx(w, g)[1:-1])
    s23 = 0.5 * ((v[1:-1] - v[:-2]) * rdz + _dy(w, g)[1:-1])
    ends = lambda a: torch.cat([a[:1], a, torch.zeros_like(a[:1])])  # noqa: E731   w-levels 0 .. nz-1
    s13, s23 = ends(s13), ends(s23)
    mean = lambda a: 0.5 * (a[1:] + a[:-1])  # noqa: E731
    nu = lambda a, b, c, d, e, f, wt: -2.0 * torch.sqrt(2.0 * (a * a + b * b + c * c) + 4.0 * (d * d + e * e + f * f)) / (lam0 + wt)  # noqa: E731
    wt = [1.0 / (KAPPA * (p + t.z0)) ** 2 for p in t.phi]
    tau = [x.double().clone() for x in t.tau]
    m = nu(s11, s22, s33, s12, mean(s13), mean(s23), wt[0][:-1])
    fluid = (t.phi[0] > 2 * t.phi_b)[:-1]
    for c, s in zip(UV, (s11, s12, s22, s33)):
        tau[c][:-1] = torch.where(fluid, m * s, tau[c][:-1])
    m = nu(mean(s11), mean(s22), mean(s33), mean(s12), s13[1:-1], s23[1:-1], wt[1][1:-1])
    fluid = t.phi[1] > t.phi_b
    for c, s in zip(W, (s13, s23)):
        tau[c][1:-1] = torch.where(fluid[1:-1], m * s[1:-1], tau[c][1:-1])
        tau[c][-1] = torch.where(fluid[-1], 0.0, tau[c][-1])
    return tau


def _triangle2(p, a, b, c):
    """Squared distance of the points p to the triangles a, b, c (tuples of coordinates)."""
    sub = lambda x, y: (x[0] - y[0], x[1] - y[1], x[2] - y[2])  # noqa: E731
    dot = lambda x, y: x[0] * y[0] + x[1] * y[1] + x[2] * y[2]  # noqa: E731

    def segment(q, r):
        e, d = sub(r, q), sub(p, q)
        s = (dot(d, e) / dot(e, e)).clamp(0.0, 1.0)
        m = (d[0] - s * e[0], d[1] - s * e[1], d[2] - s * e[2])
        return dot(m, m)

    ab, ac, ap = sub(b, a), sub(c, a), sub(p, a)
    d00, d01, d11 = dot(ab, ab), dot(ab, ac), dot(ac, ac)
    d20, d21 = dot(ap, ab), dot(ap, ac)
    den = d00 * d11 - d01 * d01
    v, w = (d11 * d20 - d01 * d21) / den, (d00 * d21 - d01 * d20) / den
    inside = (v >= 0) & (w >= 0) & (v + w <= 1)
    m = tuple(ap[c] - v * ab[c] - w * ac[c] for c in range(3))
    edges = torch.minimum(torch.minimum(segment(a, b), segment(b, c)), segment(a, c))
    return torch.where(inside, dot(m, m), edges)


def _sdf(case, seed):
    grid = _grid(case)
    nx, ny, nz, lx, ly, lz = grid
    dx, dy, reach = lx / nx, ly / ny, case["reach"] / (nz - 1)
    h = _heights(grid, case["terrain"], random.Random(int(seed) * 104729 + 5))
    wx, wy = math.ceil(reach / dx), math.ceil(reach / dy)
    lo, hi = h.clone(), h.clone()
    for dim, reachable in ((1, wx), (0, wy)):       # height range over the window
        low, high = lo, hi
        for s in range(-reachable, reachable + 1):
            low, high = torch.minimum(low, torch.roll(lo, s, dim)), torch.maximum(high, torch.roll(hi, s, dim))
        lo, hi = low, high
    out = []
    for z in _levels(grid):
        phi = z[:, None, None] - h[None]
        near = (z[:, None, None] >= lo[None] - reach) & (z[:, None, None] <= hi[None] + reach)
        k, j, i = torch.nonzero(near, as_tuple=True)
        best = phi[near] ** 2
        p = (torch.zeros_like(best), torch.zeros_like(best), z[k])
        for b in range(-wy, wy):
            for a in range(-wx, wx):
                corner = lambda da, db: (torch.full_like(best, (a + da) * dx), torch.full_like(best, (b + db) * dy),  # noqa: E731
                                         h[(j + b + db) % ny, (i + a + da) % nx])
                A, B, C, D = corner(0, 0), corner(1, 0), corner(1, 1), corner(0, 1)
                best = torch.minimum(best, torch.minimum(_triangle2(p, A, B, C), _triangle2(p, A, C, D)))
        d = torch.sqrt(best)
        vert = phi[near]
        phi[near] = torch.where(d <= reach, torch.copysign(d, vert), vert)
        out.append(phi)
    return tuple(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sdf":
        return _sdf(case, seed)
    if kind == "batch":
        parts = []
        for m, spec in enumerate(_members(case)):
            parts.append(_step(_member(case, seed, m, spec), case))
        join = lambda key, n: [torch.cat([p[key][c].reshape(-1) for p in parts]) for c in range(n)]  # noqa: E731
        return {"vel": join("vel", 3), "tau": join("tau", 6), "f": join("f", 3)}
    t = _Terrain(case, seed)
    if kind == "step":
        return _step(t, case)
    vel, tau = [v.double() for v in t.vel], [x.double() for x in t.tau]
    if kind == "spectral":
        dx = lambda a, g: _spectral(a, g[3], 2)  # noqa: E731
        dy = lambda a, g: _spectral(a, g[4], 1)  # noqa: E731
        return _divergence(tau, t.grid, dx, dy)
    if kind in ("sgs_chain", "sgs_fused"):
        full, _, _ = _wall(t, vel, _sgs(t))
        f = _divergence(full, t.grid)
        return {"tau": full if kind == "sgs_chain" else _wall(t, vel, tau)[0], "f": f}
    wrt = [v.requires_grad_() for v in vel] + [torch.log(t.z0).to(t.type).double().requires_grad_()]
    f = _divergence(_wall(t, wrt[:3], tau, wrt[3])[0], t.grid)
    g = [_Draws(seed + 501 + c).normal(t.shape, 1.0, t.type).double() for c in range(3)]
    return {"f": [x.detach() for x in f], "grad": torch.autograd.grad(f, wrt, g)}
