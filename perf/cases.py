"""Performance cases: the solves a user of this library runs, through its public Python entry points.

A case names a problem (sizes, grid stretching, boundary pairs, coefficients), the arithmetic of its plan and the entry
point.  `listed` gives the fixed cases, `draw` further ones of the same ranges, `prepare` the plan and buffers that a
program keeps between calls, `run` one call, `work` the bytes and operations that the call cannot do without, and
`exact` the result in plain float64 torch (three dense eigenbases and refinement), without the library.

Fields are flat float64 CUDA tensors, x fastest: (nz, ny, nx) as a torch shape.
"""
import math
import random

import numpy as np
import torch

import paper_2603_09528_gb300 as tpt

DEVICE = "cuda:0"
PRECISION = {"fp64": tpt.FP64, "bf16x3": tpt.MIXED_BF16X3, "tf32": tpt.MIXED_TF32, "ozaki": 4}
PAIRS = {"periodic": (tpt.PERIODIC,) * 2, "neumann": (tpt.NEUMANN,) * 2, "dirichlet": (tpt.DIRICHLET,) * 2,
         "mixed": (tpt.DIRICHLET, tpt.NEUMANN)}
# sizes of the batched workload (many independent instances of uneven size)
BATCH_SIZES = ((64, 64, 64), (96, 128, 160), (128, 128, 128), (192, 192, 96), (256, 256, 256))


def _case(kind, n, stretch, bc, precision, alpha=0.0, beta=1.0, name=None, **more):
    c = {} if name is None else {"name": name}
    c.update(kind=kind, nx=n[0], ny=n[1], nz=n[2], sx=stretch[0], sy=stretch[1], sz=stretch[2], bx=bc[0], by=bc[1],
             bz=bc[2], precision=precision, alpha=alpha, beta=beta)
    c.update(more)
    return c


def listed():
    wall = ("neumann",) * 3
    return [
        # the smallest everyday solve: channel-like 32^3, periodic uniform x (FFT), two stretched wall directions; latency
        _case("solve", (32, 32, 32), (0.0, 1.5, 1.5), ("periodic", "neumann", "neumann"), "fp64", name="fp64_32_channel"),
        # a small implicit-diffusion solve on sizes that divide no tile, with Dirichlet walls
        _case("solve", (61, 97, 75), (1.5, 2.0, 1.2), ("dirichlet", "neumann", "mixed"), "fp64", 1.0, -5e-4,
              name="fp64_61x97x75_helmholtz"),
        # the float64 production solve: stretched pressure Poisson, eigenbasis transforms in x and y
        _case("solve", (256, 256, 256), (2.0, 2.0, 2.0), wall, "fp64", name="fp64_256_poisson"),
        # the same grid made uniform: cosine transforms in x and y, implicit diffusion
        _case("solve", (256, 256, 256), (0.0, 0.0, 0.0), wall, "fp64", 1.0, -5e-4, name="fp64_256_uniform_helmholtz"),
        # the full-size stretched Poisson solve in float64, against which the mixed path is quoted
        _case("solve", (512, 512, 512), (1.5, 2.0, 2.5), wall, "fp64", name="fp64_512_poisson"),
        # float64 accuracy asked for from the tensor cores, three different sizes
        _case("solve", (384, 320, 256), (1.5, 2.0, 2.5), wall, "ozaki", name="ozaki_384x320x256_poisson"),
        # the smallest request of a batch or a server: split bf16 corrections to 1e-10; launches count
        _case("solve", (64, 64, 64), (2.0, 1.5, 2.5), wall, "bf16x3", name="bf16x3_64_poisson"),
        # a served implicit-diffusion request of ragged size
        _case("solve", (150, 277, 133), (1.25, 2.0, 3.0), wall, "bf16x3", 1.0, -2.5e-3, name="bf16x3_150x277x133_helmholtz"),
        # the headline: full-size stretched Poisson, refined to 1e-10, tiles tuned as a long run does
        _case("solve", (512, 512, 512), (1.5, 2.0, 2.5), wall, "bf16x3", name="bf16x3_512_poisson", tune=True),
        # corrections with float32-like operands (tf32), implicit diffusion
        _case("solve", (192, 192, 96), (1.5, 2.5, 2.0), wall, "tf32", 1.0, -5e-3, name="tf32_192x192x96_helmholtz"),
        # many uneven instances at once, Poisson and Helmholtz mixed
        dict(name="batch_24_uneven", kind="batch", count=24, members=5, precision="bf16x3"),
        # one fractional-step pressure projection: divergence, refined solve, gradient correction
        _case("project", (256, 256, 256), (0.0, 2.0, 1.5), ("periodic", "neumann", "neumann"), "bf16x3",
              name="project_256_duct"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("fp64", "fp64", "fp64_fourier", "ozaki", "bf16x3", "bf16x3", "bf16x3", "tf32", "batch", "project"))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 24), members=rng.randint(6, 1 << 20), precision="bf16x3")
    stretch = [round(rng.uniform(1.0, 3.0), 2) for _ in range(3)]
    bc = [rng.choice(("neumann", "neumann", "dirichlet", "mixed")) for _ in range(3)]
    if kind == "project":
        n = [4 * _log_int(rng, 8, 80) for _ in range(3)]
        bc = [rng.choice(("periodic", "neumann")), "neumann", "neumann"]
        if bc[0] == "periodic":
            stretch[0] = 0.0
        return _case("project", n, stretch, bc, "bf16x3")
    if kind == "fp64_fourier":      # a uniform direction of power-of-two size takes a Fourier transform
        n = [2 ** rng.randint(4, 8), _log_int(rng, 24, 256), _log_int(rng, 24, 256)]
        bc[0] = rng.choice(("periodic", "neumann"))
        stretch[0] = 0.0
        kind = "fp64"
        if rng.random() < 0.5:
            n[1], stretch[1], bc[1] = 2 ** rng.randint(4, 8), 0.0, "neumann"
    elif kind == "fp64":
        n = [_log_int(rng, 24, 320) for _ in range(3)]
    elif kind == "ozaki":
        n = [_log_int(rng, 48, 400) for _ in range(3)]
    elif kind == "tf32":
        n = [_log_int(rng, 48, 224) for _ in range(3)]
    else:
        n = [_log_int(rng, 48, 480) for _ in range(3)]
        if rng.random() < 0.6:      # served sizes: multiples of 32
            n = [max(64, v // 32 * 32) for v in n]
    if kind == "tf32" or rng.random() < 0.4:
        return _case("solve", n, stretch, bc, kind, 1.0, -0.5 * round(rng.uniform(1e-4, 1e-2), 5))
    return _case("solve", n, stretch, bc, kind)


# ------------------------------------------------------------------ problems

def _grid(n, stretch):
    """Cell widths and centre spacings of a tanh-stretched (0: uniform) grid on [0, 1]."""
    xi = np.arange(n + 1, dtype=np.float64) / n
    xf = xi if stretch == 0.0 else 0.5 * (1.0 + np.tanh(stretch * (xi - 0.5)) / np.tanh(0.5 * stretch))
    if stretch == 0.0:
        return np.full(n, 1.0 / n), np.full(n + 1, 1.0 / n)
    dxf, xc = np.diff(xf), 0.5 * (xf[1:] + xf[:-1])
    dxc = np.empty(n + 1)
    dxc[1:n] = np.diff(xc)
    dxc[0] = dxc[n] = 0.5 * (dxf[0] + dxf[-1])
    return dxf, dxc


def _members(case):
    """The instances of a batch: half Poisson, half Helmholtz, stretching in [1, 3]; whole and odd coefficients alike."""
    rng = random.Random(case["members"])
    out = []
    for _ in range(case["count"]):
        n = rng.choice(BATCH_SIZES)
        stretch = [rng.choice((1.0, 1.5, 2.0, 2.5, 3.0)) for _ in range(3)]
        ab = (0.0, 1.0) if rng.random() < 0.5 else (1.0, -0.5 * round(rng.uniform(1e-4, 1e-2), 5))
        out.append(_case("solve", n, stretch, ("neumann",) * 3, case["precision"], *ab))
    return out


def _sizes(c):
    return c["nx"], c["ny"], c["nz"]


def _bcs(c):
    return c["bx"], c["by"], c["bz"]


def _grids(c):
    return [_grid(n, s) for n, s in zip(_sizes(c), (c["sx"], c["sy"], c["sz"]))]


def _singular(c):
    return c["alpha"] == 0.0 and all(b in ("periodic", "neumann") for b in _bcs(c))


def _volumes(c, grids):
    wx, wy, wz = (torch.from_numpy(g[0]).to(DEVICE) for g in grids)
    return wz[:, None, None] * wy[None, :, None] * wx[None, None, :]


def _rhs(c, grids, seed):
    """Uniform [-1, 1) right-hand side; the volume-weighted mean removed where the operator is singular."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    nx, ny, nz = _sizes(c)
    f = torch.rand((nz, ny, nx), generator=gen, dtype=torch.float64, device=DEVICE).mul_(2.0).sub_(1.0)
    if _singular(c):
        vol = _volumes(c, grids)
        f -= (f * vol).sum() / vol.sum()
    return f.reshape(-1)


def _velocities(c, seed):
    """A predicted face velocity: noise inside, zero on walls, equal values on the two ends of a periodic line."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    out = []
    for ax in range(3):
        shape = list(_sizes(c))
        shape[ax] += 1
        u = torch.rand(shape[::-1], generator=gen, dtype=torch.float64, device=DEVICE).mul_(2.0).sub_(1.0)
        first, last = u.select(2 - ax, 0), u.select(2 - ax, shape[ax] - 1)
        if _bcs(c)[ax] == "periodic":
            last.copy_(first)
        else:
            first.zero_()
            last.zero_()
        out.append(u.reshape(-1))
    return out


GAMMA_DT = 2e-3   # time-step factor of the projection


def _spec(c, grids):
    adaptive = c["precision"] in ("bf16x3", "tf32")
    return dict(n=_sizes(c), dxf=[g[0] for g in grids], dxc=[g[1] for g in grids], bc=[PAIRS[b] for b in _bcs(c)],
                alpha=c["alpha"], beta=c["beta"], precision=PRECISION[c["precision"]],
                rtol=1e-10 if adaptive else 0.0, max_refine=40 if adaptive else 1)


# ------------------------------------------------------------------ the measured calls

def prepare(case, seed):
    if case["kind"] == "batch":
        members = _members(case)
        grids = [_grids(c) for c in members]
        batch = tpt.Batch([_spec(c, g) for c, g in zip(members, grids)])
        fs = [_rhs(c, g, 1000 * seed + i) for i, (c, g) in enumerate(zip(members, grids))]
        phis = [torch.zeros_like(f) for f in fs]
        work = batch.new_workspace()
        batch.calibrate(fs, phis, work, rtol=1e-10, max_refine=40, spare=0)
        return dict(kind="batch", batch=batch, fs=fs, phis=phis, work=work)
    grids = _grids(case)
    plan = tpt.Plan(device=0, **_spec(case, grids))
    if case["kind"] == "project":
        vel = _velocities(case, seed)
        return dict(kind="project", plan=plan, predicted=vel, vel=[torch.empty_like(u) for u in vel],
                    phi=plan.new_field(), work=plan.project_workspace())
    work = plan.new_workspace()
    if case.get("tune"):
        plan.autotune(work)
    return dict(kind="solve", plan=plan, f=_rhs(case, grids, seed), phi=plan.new_field(), work=work)


def run(state):
    if state["kind"] == "batch":
        state["batch"].solve(state["fs"], state["phis"], state["work"], want_info=False)
        return state["phis"]
    if state["kind"] == "project":
        # the call corrects the velocity in place: each pass starts from the predicted one
        for u, p in zip(state["vel"], state["predicted"]):
            u.copy_(p)
        phi, _ = state["plan"].project(*state["vel"], GAMMA_DT, phi=state["phi"], work=state["work"])
        return dict(phi=phi, u=state["vel"][0], v=state["vel"][1], w=state["vel"][2])
    phi, _ = state["plan"].solve(state["f"], state["phi"], state["work"], want_info=False)
    return phi


def work(case):
    """One direct solve: the right-hand side read, the solution written; two transforms each along x and y, one tridiagonal
    solve along z.  A projection also reads and writes the three face velocities."""
    if case["kind"] == "batch":
        each = [work(c) for c in _members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    nx, ny, nz = _sizes(case)
    pts = nx * ny * nz
    per = 8.0
    for n, s, b in zip((nx, ny), (case["sx"], case["sy"]), _bcs(case)):
        fourier = s == 0.0 and b in ("periodic", "neumann") and n & (n - 1) == 0 and case["precision"] in ("fp64", "ozaki")
        per += 2.0 * (2.5 * math.log2(n) if fourier else 2.0 * n)
    if case["kind"] == "project":
        return {"bytes": 8.0 * 7 * pts, "flops": (per + 15.0) * pts}
    return {"bytes": 16.0 * pts, "flops": per * pts}


# ------------------------------------------------------------------ the same in plain float64

class _Direction:
    """Rows a, b, c of the 1D second difference with its boundary rows, and its eigenbasis T = Q diag(lam) Q^-1."""

    def __init__(self, grid, bc):
        dxf, dxc = grid
        n = dxf.size
        a, c, w = 1.0 / (dxf * dxc[:n]), 1.0 / (dxf * dxc[1:]), np.zeros(n)
        if bc != "periodic":
            if bc in ("dirichlet", "mixed"):
                w[0] += 2.0 / (dxf[0] * dxf[0])
            if bc == "dirichlet":
                w[-1] += 2.0 / (dxf[-1] * dxf[-1])
            a[0] = c[-1] = 0.0
        b = -((a + c) + w)
        T = np.diag(b)
        for i in range(n):          # cyclic corners of a periodic direction; zero otherwise
            T[i, (i - 1) % n] += a[i]
            T[i, (i + 1) % n] += c[i]
        s = np.sqrt(dxf)
        S = s[:, None] * T / s[None, :]
        lam, V = np.linalg.eigh(0.5 * (S + S.T))
        if bc in ("periodic", "neumann"):
            lam[np.argmax(lam)] = 0.0

        def dev(v):
            return torch.from_numpy(np.ascontiguousarray(v)).to(DEVICE)

        self.a, self.b, self.c, self.lam = dev(a), dev(b), dev(c), dev(lam)
        self.Q, self.Qinv = dev(V / s[:, None]), dev(V.T * s[None, :])


def _along(M, x, axis):
    """M applied along one axis of a (z, y, x) field."""
    if axis == 2:
        return x @ M.T
    if axis == 1:
        return torch.matmul(M, x)
    return (M @ x.reshape(x.shape[0], -1)).reshape(x.shape)


def _solve_exact(c, f):
    """(alpha + beta L) phi = f on a (z, y, x) field: all three directions diagonalised, three steps of refinement; zero
    volume-weighted mean where the operator is singular."""
    grids = _grids(c)
    dirs = [_Direction(g, b) for g, b in zip(grids, _bcs(c))][::-1]     # z, y, x, as the axes of the field
    shape = [[-1 if k == ax else 1 for k in range(3)] for ax in range(3)]
    modes = c["alpha"] + c["beta"] * sum(d.lam.reshape(shape[ax]) for ax, d in enumerate(dirs))
    vol = _volumes(c, grids) if _singular(c) else None
    if vol is not None:
        modes = torch.where(modes == 0.0, torch.inf, modes)             # the null mode's coefficient is zero

    def centred(x):
        return x if vol is None else x - (x * vol).sum() / vol.sum()

    def direct(x):
        for ax, d in enumerate(dirs):
            x = _along(d.Qinv, x, ax)
        x = x / modes
        for ax, d in enumerate(dirs):
            x = _along(d.Q, x, ax)
        return x

    def operator(x):
        y = c["alpha"] * x
        for ax, d in enumerate(dirs):
            a, b, up = (v.reshape(shape[ax]) for v in (d.a, d.b, d.c))
            y = y + c["beta"] * (b * x + a * torch.roll(x, 1, ax) + up * torch.roll(x, -1, ax))
        return y

    f = centred(f)
    phi = direct(f)
    for _ in range(3):
        phi = phi + direct(centred(f - operator(phi)))
    return centred(phi)


def _project_exact(c, vel):
    """Divergence over the time-step factor, the Poisson solve, and the gradient taken off the interior and periodic faces."""
    grids = _grids(c)
    n = _sizes(c)
    faces = []
    div = 0.0
    for ax in range(3):
        sh = list(n)
        sh[ax] += 1
        u = vel[ax].reshape(sh[::-1])
        t = 2 - ax
        faces.append(u)
        width = torch.from_numpy(grids[ax][0]).to(DEVICE).reshape([-1 if k == t else 1 for k in range(3)])
        div = div + (u.narrow(t, 1, n[ax]) - u.narrow(t, 0, n[ax])) / width
    phi = _solve_exact(c, div / GAMMA_DT)
    out = {"phi": phi.reshape(-1)}
    for ax, key in enumerate("uvw"):
        t, m = 2 - ax, n[ax]
        dxc = torch.from_numpy(grids[ax][1]).to(DEVICE).reshape([-1 if k == t else 1 for k in range(3)])
        u = faces[ax].clone()
        g = (phi.narrow(t, 1, m - 1) - phi.narrow(t, 0, m - 1)) / dxc.narrow(t, 1, m - 1)
        u.narrow(t, 1, m - 1).sub_(GAMMA_DT * g)
        if _bcs(c)[ax] == "periodic":
            wrap = GAMMA_DT * (phi.narrow(t, 0, 1) - phi.narrow(t, m - 1, 1)) / dxc.narrow(t, 0, 1)
            u.narrow(t, 0, 1).sub_(wrap)
            u.narrow(t, m, 1).sub_(wrap)
        out[key] = u.reshape(-1)
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        return [_solve_exact(c, _rhs(c, _grids(c), 1000 * seed + i).reshape(_sizes(c)[::-1])).reshape(-1)
                for i, c in enumerate(_members(case))]
    if case["kind"] == "project":
        return _project_exact(case, _velocities(case, seed))
    return _solve_exact(case, _rhs(case, _grids(case), seed).reshape(_sizes(case)[::-1])).reshape(-1)
