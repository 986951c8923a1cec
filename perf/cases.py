"""The calls whose speed matters, as a program that uses this library makes
them: operator applications, Arnoldi processes, projected exponentials,
stationary solves, frequency responses (restarted in time and in Krylov
dimension, one problem and a batch of uneven ones) and the adjoint gradient,
each through the Python entry points, over the sizes of the repository's own
configurations and their neighbours, ragged ones among them.

``listed()`` gives the cases, ``draw(rng)`` others of the same ranges,
``prepare`` the inputs and the context, ``run`` one pass, ``work`` the bytes
and operations a pass cannot do without, and ``exact`` the same outputs from
plain torch in 64 bits (its own operator and time integration).

Media are random round inclusions (permittivity 2.25 or 4 in 1) between the
absorbing layers, made from the seed; the source is the plane (3D) or line
(2D) source of the benchmark; vectors are standard normal.  Summed
intensities and Hessenberg entries of a single-precision context are handed
on in single precision, the accuracy they carry.
"""
import math

import numpy as np
import torch

from paper_1707_00023_gb300 import Batch, Context, intensity_loss

OMEGA0 = 2.0 * math.pi / 16.0
PERIODIC, PEC = 0, 1


# ---------------------------------------------------------------------------
# The cases.
def listed():
    return [
        # the smallest call: one operator application on the 2D double-precision
        # grid of the paper's test problem (launch latency)
        dict(name="apply 2d 64 f64", kind="apply", dim=2, nx=64, ny=64, prec="fp64", transpose=False),
        # one application on the largest benchmark grid (memory bandwidth)
        dict(name="apply 3d 128 f32", kind="apply", dim=3, nx=128, ny=128, nz=128, prec="fp32", transpose=False),
        # a Krylov basis of the 64^3 grid handed to the caller
        dict(name="arnoldi 3d 64 f32", kind="arnoldi", dim=3, nx=64, ny=64, nz=64, m=64, prec="fp32"),
        # the projected problem for 32 frequencies (small dense work)
        dict(name="expm phi 64 32f", kind="expm", m=64, nfreq=32, tau=10.0),
        # stationary parts of 8 frequencies on a strongly damped, ragged
        # double-precision grid
        dict(name="stationary 3d ragged f64", kind="stationary", dim=3, nx=45, ny=38, nz=52, m=64, nfreq=8,
             prec="fp64", cap=640),
        # the 2D test problem: one frequency, restarted in time, double precision
        dict(name="plain 2d 64 f64", kind="plain", dim=2, nx=64, ny=64, m=30, nfreq=1, prec="fp64", T=200.0,
             rtol=1e-11, pml=False),
        # the 64^3 problem, one frequency, restarted in time
        dict(name="plain 3d 64 f32", kind="plain", dim=3, nx=64, ny=64, nz=64, m=64, nfreq=1, prec="fp32", T=400.0,
             rtol=1e-7, pml=False),
        # the multi-frequency benchmark: 128^3, 32 frequencies on one basis a restart
        dict(name="rstdim 3d 128 32f", kind="rstdim", dim=3, nx=128, ny=128, nz=128, m=64, nfreq=32, prec="fp32",
             T=400.0, rtol=1e-7, full=False),
        # the same method on the 64^3 medium
        dict(name="rstdim 3d 64 32f", kind="rstdim", dim=3, nx=64, ny=64, nz=64, m=64, nfreq=32, prec="fp32",
             T=400.0, rtol=1e-7, full=False),
        # a small scatterer with its whole fields returned, four frequencies
        dict(name="rstdim 3d 36 4f full", kind="rstdim", dim=3, nx=36, ny=36, nz=36, m=64, nfreq=4, prec="fp32",
             T=400.0, rtol=1e-7, full=True),
        # the uneven batch: scatterer instances of 32^3 to 96^3, four frequencies each
        dict(name="batch uneven 8 4f", kind="batch", count=8, sizes=1711, nmin=32, nmax=96, m=64, nfreq=4, T=400.0,
             rtol=1e-7),
        # one gradient of the plane intensity with respect to the permittivity
        # (forward, backward and quadrature), as an optimiser takes it
        dict(name="adjoint 3d 48 2f", kind="adjoint", dim=3, nx=48, ny=48, nz=48, m=64, nfreq=2, prec="fp32", T=100.0,
             rtol=1e-7),
    ]


def _side(rng, lo, hi):
    """A size in [lo, hi], spread over its logarithm, multiples of 4 as
    often as not."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, n // 4 * 4) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["apply", "arnoldi", "expm", "stationary", "plain2", "plain3", "rstdim", "batch", "adjoint"])
    if kind == "apply":
        dim = rng.choice([2, 3])
        c = dict(kind="apply", dim=dim, prec=rng.choice(["fp32", "fp64"]), transpose=rng.random() < 0.4)
        sides = ("nx", "ny") if dim == 2 else ("nx", "ny", "nz")
        return dict(c, **{k: _side(rng, 32, 512 if dim == 2 else 128) for k in sides})
    if kind == "arnoldi":
        return dict(kind="arnoldi", dim=3, prec=rng.choice(["fp32", "fp64"]), m=rng.randint(8, 64),
                    **{k: _side(rng, 16, 72) for k in ("nx", "ny", "nz")})
    if kind == "expm":
        return dict(kind="expm", m=rng.randint(16, 64), nfreq=rng.randint(0, 32), tau=rng.uniform(1.0, 20.0))
    if kind == "stationary":
        return dict(kind="stationary", dim=3, m=rng.randint(32, 64), nfreq=rng.randint(1, 12),
                    prec="fp64", cap=320, **{k: _side(rng, 16, 52) for k in ("nx", "ny", "nz")})
    if kind == "plain2":
        n = {k: _side(rng, 32, 128) for k in ("nx", "ny")}
        return dict(kind="plain", dim=2, m=rng.randint(24, 48), nfreq=rng.randint(1, 4), prec="fp64",
                    T=rng.uniform(50.0, 200.0), rtol=1e-11, pml=rng.random() < 0.3, **n)
    if kind == "plain3":
        n = {k: _side(rng, 24, 64) for k in ("nx", "ny", "nz")}
        return dict(kind="plain", dim=3, m=rng.randint(40, 64), nfreq=rng.randint(1, 4), prec="fp32",
                    T=rng.uniform(50.0, 200.0), rtol=1e-7, pml=False, **n)
    if kind == "rstdim":
        full = rng.random() < 0.3
        n = {k: _side(rng, 24, 48 if full else 112) for k in ("nx", "ny", "nz")}
        return dict(kind="rstdim", dim=3, m=64, nfreq=rng.randint(1, 8 if full else 32), prec="fp32",
                    T=rng.uniform(100.0, 400.0), rtol=1e-7, full=full, **n)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 8), sizes=rng.randint(1, 10**6), nmin=24, nmax=80, m=64,
                    nfreq=rng.randint(1, 4), T=rng.uniform(100.0, 400.0), rtol=1e-7)
    return dict(kind="adjoint", dim=3, m=rng.randint(40, 64), nfreq=rng.randint(1, 2), prec="fp32",
                T=rng.uniform(30.0, 100.0), rtol=1e-7, **{k: _side(rng, 24, 48) for k in ("nx", "ny", "nz")})


# ---------------------------------------------------------------------------
# Grids and inputs.
class Grid:
    """What Context reads of a grid."""

    def __init__(self, dim, n, bc, layer_axis, layer_cells, sigma_max, pml=0):
        self.dim, self.n, self.bc = dim, tuple(n), bc
        self.layer_axis, self.layer_cells, self.sigma_max, self.pml = layer_axis, layer_cells, sigma_max, pml
        self.shape = tuple(reversed(self.n))
        self.ncomp = 6 if dim == 3 else 3 + pml
        self.nunk = self.ncomp * int(np.prod(self.n))


def _staggering(grid):
    """Per component, 1 along the axes where its nodes lie half a cell off
    (Hx, Hy, Ez[, P] in 2D; Hx, Hy, Hz, Ex, Ey, Ez in 3D)."""
    if grid.dim == 2:
        return [(0, 1), (1, 0), (0, 0)] + [(0, 0)] * grid.pml
    return [(0, 1, 1), (1, 0, 1), (1, 1, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]


def _layer(n):
    return (8 if n >= 48 else 6) if n >= 32 else max(2, n // 8)


def _grid(case):
    if case["dim"] == 2:
        pml = int(bool(case.get("pml")))
        return Grid(2, (case["nx"], case["ny"]), (PEC, PEC), 0, _layer(case["nx"]), 3.0 if pml else 1.0, pml)
    n = (case["nx"], case["ny"], case["nz"])
    # the stationary solves converge on strongly damped problems: there the
    # layers meet in the middle
    L = n[2] // 2 if case["kind"] == "stationary" else _layer(n[2])
    return Grid(3, n, (PERIODIC, PERIODIC, PEC), 2, L, 1.0)


def _medium(grid, rng, fill=0.3, eps=2.25):
    """Permittivity per cell: random round inclusions (radius 2-5 cells) up
    to about the volume fraction ``fill`` between the layers."""
    out = np.ones(grid.shape)
    axis, L = grid.layer_axis, _layer(grid.n[grid.layer_axis])
    lo = [0.0] * grid.dim
    hi = [float(v) for v in grid.n]
    lo[axis], hi[axis] = L + 3.0, grid.n[axis] - L - 3.0
    vol = np.prod([h - q for h, q in zip(hi, lo)])
    mean = np.pi * 12.67 if grid.dim == 2 else 4.0 / 3.0 * np.pi * 50.75   # of pi r^2, 4/3 pi r^3 over r in [2, 5]
    count = int(math.ceil(-math.log(1.0 - fill) * vol / mean))
    for _ in range(count):
        r = rng.uniform(2.0, 5.0)
        c = [rng.uniform(a, b) for a, b in zip(lo, hi)]
        box, d2 = [], 0.0
        for a in range(grid.dim):                        # x, y[, z]; the array is [z,] y, x
            i0, i1 = max(0, int(c[a] - r)), min(grid.n[a], int(c[a] + r) + 2)
            box.append(slice(i0, i1))
            shape = [1] * grid.dim
            shape[grid.dim - 1 - a] = -1
            d2 = d2 + ((np.arange(i0, i1) + 0.5 - c[a]) ** 2).reshape(shape)
        out[tuple(reversed(box))][d2 < r * r] = eps
    return out


def _source(grid, dtype):
    """Plane source on the Ex nodes behind the first layer (3D); line
    source on the Ez nodes, tapered at the walls (2D)."""
    g = torch.zeros((grid.ncomp,) + grid.shape, dtype=dtype, device="cuda")
    at = _layer(grid.n[grid.layer_axis]) + 1
    if grid.dim == 3:
        g[3, at] = 1.0
    else:
        y = torch.arange(grid.n[1], dtype=torch.float64, device="cuda")
        edge = grid.n[1] / 10.0
        g[2, :, at] = torch.clamp(torch.minimum(y, grid.n[1] - y) / edge, max=1.0).to(dtype)
    return g.reshape(-1)


def _plane(grid):
    n = grid.n[grid.layer_axis]
    return grid.layer_axis, n - _layer(n) - 2


def _freqs(nfreq, lo=0.8, hi=1.2):
    return np.array([OMEGA0]) if nfreq == 1 else OMEGA0 * np.linspace(lo, hi, nfreq)


def _dtype(case):
    return torch.float64 if case.get("prec", "fp32") == "fp64" else torch.float32


def _batch_problems(case):
    """Grid, medium parameters and frequencies of each problem of a batch:
    sizes from {nmin, nmin + 4, ..}, permittivity 2.25 or 4, fill 0.2 to 0.4."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = case["nmin"] + 4 * int(rng.integers(0, (case["nmax"] - case["nmin"]) // 4 + 1))
        eps, fill = (2.25, 4.0)[int(rng.integers(0, 2))], float(rng.uniform(0.2, 0.4))
        out.append((Grid(3, (n, n, n), (PERIODIC, PERIODIC, PEC), 2, _layer(n), 1.0), eps, fill))
    return out, np.tile(_freqs(case["nfreq"], 0.9, 1.1), (case["count"], 1))


def _vector(grid, seed, dtype):
    """Standard normal values, zero on the conducting walls (index 0 along an
    axis for the components with an integer coordinate on it)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn((grid.ncomp,) + grid.shape, generator=gen, dtype=torch.float64, device="cuda")
    for a in range(grid.dim):
        if grid.bc[a] == PEC:
            for c, off in enumerate(_staggering(grid)):
                if not off[a]:
                    v[c].narrow(-1 - a, 0, 1).zero_()
    return v.reshape(-1).to(dtype)


def _hessenberg(case, seed):
    """An upper Hessenberg matrix like those of the operator: nearly
    skew-symmetric, with a small damping on the diagonal."""
    rng = np.random.default_rng(seed)
    m = case["m"]
    H = 0.05 * np.triu(rng.standard_normal((m + 1, m)))
    i = np.arange(m)
    b = rng.uniform(0.8, 1.8, m)
    H[i + 1, i] = b
    H[i[:-1], i[1:]] -= b[:-1]
    H[i, i] += rng.uniform(0.0, 0.3, m)
    return H


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    s = {"case": case}
    if kind == "expm":
        # any context serves: the call works on the Hessenberg matrix alone
        grid = Grid(2, (16, 16), (PEC, PEC), 0, 2, 1.0)
        s["ctx"] = Context(grid, np.ones(grid.shape), precision="fp64", krylov_dim=64, max_freqs=32)
        s["H"] = _hessenberg(case, seed)
        s["omegas"] = _freqs(case["nfreq"]) if case["nfreq"] else None
        return s
    if kind == "batch":
        problems, s["omegas"] = _batch_problems(case)
        s["ctxs"] = [Context(g, _medium(g, rng, fill, eps), krylov_dim=case["m"], max_freqs=case["nfreq"], batch=2,
                             stream="own", rst_samples=4096) for g, eps, fill in problems]
        s["gs"] = [_source(g, torch.float32) for g, _, _ in problems]
        s["planes"] = np.array([_plane(g) for g, _, _ in problems])
        torch.cuda.synchronize()
        s["batch"] = Batch(s["ctxs"])
        return s
    grid, dt, nf = _grid(case), _dtype(case), case.get("nfreq", 1)
    eps = _medium(grid, rng)
    if kind == "apply" or kind == "arnoldi":
        s["ctx"] = Context(grid, eps, precision=case["prec"], krylov_dim=case.get("m", 8))
        s["v"] = _vector(grid, seed, dt)
        return s
    s["plane"], s["omegas"] = _plane(grid), _freqs(nf)
    s["g"] = _source(grid, dt)
    s["stream"] = torch.cuda.Stream()
    s["stream"].wait_stream(torch.cuda.current_stream())
    more = {"plain": dict(batch=nf), "stationary": {}, "rstdim": dict(batch=2, rst_samples=4096),
            "adjoint": dict(batch=2, max_checkpoints=128)}[kind]
    s["ctx"] = Context(grid, eps, precision=case["prec"], krylov_dim=case["m"], max_freqs=nf, stream=s["stream"], **more)
    if kind == "adjoint":
        s["eps"] = torch.tensor(eps, dtype=torch.float32, device="cuda", requires_grad=True)
        torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        return s["ctx"].apply_A(s["v"], transpose=case["transpose"])
    if kind == "expm":
        return s["ctx"].expm_phi_project(s["H"], 1.0, case["tau"], s["omegas"])
    real = np.float64 if case.get("prec", "fp32") == "fp64" else np.float32
    if kind == "arnoldi":
        V, H, beta, done = s["ctx"].arnoldi(s["v"], case["m"])
        return {"V": V, "H": H.astype(real), "beta": real(beta), "steps": done}
    if kind == "batch":
        intensity, _, restarts = s["batch"].response(s["gs"], s["omegas"], case["T"], rtol=case["rtol"],
                                                     planes=s["planes"])
        return {"intensity": intensity.astype(real), "restarts": restarts}
    with torch.cuda.stream(s["stream"]):
        if kind == "stationary":
            zr, zi, rel, products = s["ctx"].stationary_solve(s["g"], s["omegas"], rtol=1e-9, max_matvecs=case["cap"],
                                                              allow_noconv=True)
            return {"zr": zr, "zi": zi, "products": products}
        if kind == "plain":
            out = s["ctx"].response_at_freqs(s["g"], s["omegas"], case["T"], rtol=case["rtol"], method="plain",
                                             plane=s["plane"], want_full=True)
            return {"E": out["E_plane"], "Y": out["Y"], "intensity": out["intensity"].astype(real)}
        if kind == "rstdim":
            out = s["ctx"].response_restart_dim(s["g"], s["omegas"], case["T"], rtol=case["rtol"], plane=s["plane"],
                                                want_full=case["full"])
            return {"E": out["E_plane"], "Y": out["Y"], "intensity": out["intensity"].astype(real),
                    "restarts": out["restarts"]}
        s["eps"].grad = None
        loss = intensity_loss(s["ctx"], s["eps"], s["g"], s["omegas"], case["T"], rtol=case["rtol"], plane=s["plane"])
        loss.backward()
        return {"loss": loss.detach().to(torch.float32), "grad": s["eps"].grad}


# ---------------------------------------------------------------------------
# The work a pass cannot do without.
def _steps(T):
    """Krylov vectors that a response over [0, T] takes: about T times the
    operator's spectral radius."""
    return 1.1 * 3.5 * T


def _arnoldi_bytes(n, size, m):
    """An m-step process that reads the basis once a step (and the caller's
    start vector), writing each new vector."""
    return (m * m / 2.0 + 2.0 * m) * n * size


def work(case):
    kind = case["kind"]
    if kind == "expm":
        n = case["m"] + (2 if case["nfreq"] else 0)
        # about eight products of n x n matrices and a solve for each frequency
        return {"bytes": 8.0 * case["m"] * (case["m"] + max(1, case["nfreq"])),
                "flops": max(1, case["nfreq"]) * 2.0 * n ** 3 * 9.0}
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for g, _, _ in _batch_problems(case)[0]:
            one = work(dict(case, kind="rstdim", dim=3, nx=g.n[0], ny=g.n[1], nz=g.n[2], prec="fp32", full=False))
            total = {k: total[k] + one[k] for k in total}
        return total
    grid, size = _grid(case), 8 if case["prec"] == "fp64" else 4
    n, cells, nf = grid.nunk, int(np.prod(grid.n)), case.get("nfreq", 1)
    material = (3 if grid.dim == 3 else 1) * cells * size
    if kind == "apply":
        return {"bytes": 2.0 * n * size + material, "flops": 6.0 * n}
    m = case["m"]
    process = {"bytes": _arnoldi_bytes(n, size, m) + m * material, "flops": 2.0 * m * m * n}
    if kind == "arnoldi":
        return {"bytes": process["bytes"] + (m + 1.0) * n * size, "flops": process["flops"]}
    if kind == "stationary":
        k = max(1, case["cap"] // m)
        return {"bytes": k * (process["bytes"] + (m + 4.0 * nf) * n * size),
                "flops": k * (process["flops"] + 4.0 * m * nf * n)}
    times = max(1.0, _steps(case["T"]) / m)
    if kind == "rstdim":
        own = 0.0 if not case["full"] else (m + 2.0 * nf) * n * size
        return {"bytes": times * (process["bytes"] + own),
                "flops": times * (process["flops"] + (2.0 * m * nf * n if case["full"] else 0.0))}
    # restarted in time: a process and a combination of its basis for each
    # frequency and sub-step; the adjoint takes three processes and reads the
    # two bases once more
    one = {"bytes": process["bytes"] + (m + 1.0) * n * size, "flops": process["flops"] + 2.0 * m * n}
    scale = nf * times * (3.0 if kind == "adjoint" else 1.0)
    return {k: scale * v for k, v in one.items()}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits, without the library.
class _Operator:
    """A and its transpose on tensors (batch, component, [z,] y, x)."""

    def __init__(self, grid, eps):
        self.grid = g = grid
        half = _staggering(g)
        axis_of = [-1, -2, -3]                                # array axis of x, y, z
        keep, sigma, inv = [], [], []
        for off in half:
            k = torch.ones(g.shape, dtype=torch.float64, device="cuda")
            for a in range(g.dim):
                if g.bc[a] == PEC and not off[a]:
                    k.narrow(axis_of[a], 0, 1).zero_()
            keep.append(k)
            n, L = g.n[g.layer_axis], g.layer_cells
            pos = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 * off[g.layer_axis]
            d = torch.clamp(torch.maximum(L - pos, pos - (n - L)), min=0.0) / L
            shape = [1] * g.dim
            shape[axis_of[g.layer_axis]] = -1
            sigma.append((g.sigma_max * (d * d if g.pml else d)).reshape(shape))
        for off in (half[2:3] if g.dim == 2 else half[3:]):
            mean = eps
            for a in range(g.dim):
                if not off[a]:
                    mean = 0.5 * (mean + torch.roll(mean, 1, axis_of[a]))
            inv.append(1.0 / mean)
        self.keep, self.sigma, self.inv = torch.stack(keep), sigma, inv

    @staticmethod
    def _up(v, a):
        return torch.roll(v, -1, a) - v

    @staticmethod
    def _down(v, a):
        return v - torch.roll(v, 1, a)

    def __call__(self, v, transpose=False):
        up, down, s, inv = self._up, self._down, self.sigma, self.inv
        c = (v * self.keep).unbind(1)
        if self.grid.dim == 2:
            hx, hy, ez = c[:3]
            curl = down(hy, -1) - down(hx, -2)
            if self.grid.pml:
                p = c[3]
                out = [up(ez, -2), s[1] * hy - up(ez, -1), s[2] * ez - inv[0] * curl - p,
                       s[2] * inv[0] * down(hx, -2)]
            elif transpose:
                ez = ez * inv[0]
                out = [s[0] * hx - up(ez, -2), s[1] * hy + up(ez, -1), s[2] * ez + curl]
            else:
                out = [s[0] * hx + up(ez, -2), s[1] * hy - up(ez, -1), inv[0] * (s[2] * ez - curl)]
            return torch.stack(out, 1) * self.keep
        hx, hy, hz, ex, ey, ez = c
        x, y, z = -1, -2, -3
        curl = [down(hz, y) - down(hy, z), down(hx, z) - down(hz, x), down(hy, x) - down(hx, y)]
        sign = 1.0
        if transpose:
            ex, ey, ez, sign = ex * inv[0], ey * inv[1], ez * inv[2], -1.0
        out = [s[0] * hx + sign * (up(ez, y) - up(ey, z)), s[1] * hy + sign * (up(ex, z) - up(ez, x)),
               s[2] * hz + sign * (up(ey, x) - up(ex, y))]
        for k, e in enumerate((ex, ey, ez)):
            out.append(s[3 + k] * e + curl[k] if transpose else inv[k] * (s[3 + k] * e - curl[k]))
        return torch.stack(out, 1) * self.keep


def _taylor(op, y, a, b, g, omegas, dt, terms):
    """One step of y' = -A y + a g, (a, b)' = (W b, -W a), by its Taylor series."""
    ty, ta, tb = y, a, b
    wide = (-1,) + (1,) * (y.dim() - 1)
    for k in range(1, terms + 1):
        ty, ta, tb = ((ta.view(wide) * g - op(ty)) * (dt / k), tb * omegas * (dt / k), -ta * omegas * (dt / k))
        y, a, b = y + ty, a + ta, b + tb
    return y


def _response(op, g, omegas, T, length, terms, wrap=None):
    """y_j(T) of y' = -A y + sin(W_j t) g, y(0) = 0, for all frequencies."""
    W = torch.as_tensor(omegas, dtype=torch.float64, device="cuda")
    y = torch.zeros((len(omegas),) + tuple(g.shape), dtype=torch.float64, device="cuda")
    steps = int(math.ceil(T / length))
    dt = T / steps
    g = g * op.keep
    for i in range(steps):
        t = i * dt
        args = (op, y, torch.sin(W * t), torch.cos(W * t), g, W, dt, terms)
        y = _taylor(*args) if wrap is None else wrap(_taylor, *args)
    return y


def _plane_of(grid, y):
    """The output plane's E values, (frequency, component, nodes)."""
    axis, at = _plane(grid)
    first = 2 if grid.dim == 2 else 3
    e = y[:, first:first + (1 if grid.dim == 2 else 3)].select(-1 - axis, at)
    return e.reshape(e.shape[0], e.shape[1], -1)


def _arnoldi(op, v, m):
    """Orthonormal basis, Hessenberg matrix and the start vector's norm
    (orthogonalised twice)."""
    shape = v.shape
    beta = torch.linalg.vector_norm(v)
    V = torch.zeros((m + 1, v.numel()), dtype=torch.float64, device="cuda")
    H = torch.zeros((m + 1, m), dtype=torch.float64, device="cuda")
    V[0] = v.reshape(-1) / beta
    for j in range(m):
        w = op(V[j].view(shape)[None])[0].reshape(-1)
        for _ in range(2):
            h = V[:j + 1] @ w
            w = w - h @ V[:j + 1]
            H[:j + 1, j] += h
        H[j + 1, j] = torch.linalg.vector_norm(w)
        V[j + 1] = w / H[j + 1, j]
    return V, H, beta


def _exact_cost(case):
    """Field values that the time integration below updates."""
    if case["kind"] == "batch":
        return sum(g.nunk for g, _, _ in _batch_problems(case)[0]) * case["nfreq"] * case["T"]
    return _grid(case).nunk * case["nfreq"] * case["T"] * (8.0 if case["kind"] == "adjoint" else 1.0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "expm":
        H = torch.tensor(_hessenberg(case, seed)[:-1], device="cuda")
        m, nf = case["m"], case["nfreq"]
        if nf == 0:
            return torch.linalg.matrix_exp(-case["tau"] * H)[:, 0].contiguous()
        N = torch.zeros((nf, m + 2, m + 2), dtype=torch.float64, device="cuda")
        N[:, :m, :m] = -H
        N[:, 0, m] = 1.0
        W = torch.as_tensor(_freqs(nf), device="cuda")
        N[:, m, m + 1], N[:, m + 1, m] = W, -W
        return torch.linalg.matrix_exp(case["tau"] * N)[:, :m, m + 1].contiguous()
    rng = np.random.default_rng(seed)
    if kind in ("plain", "rstdim", "adjoint", "batch") and _exact_cost(case) > 3e10:
        return None
    if kind == "batch":
        problems, omegas = _batch_problems(case)
        out = []
        for (g, eps, fill), om in zip(problems, omegas):
            op = _Operator(g, torch.tensor(_medium(g, rng, fill, eps), device="cuda"))
            y = _response(op, _source(g, torch.float64).view((6,) + g.shape), om, case["T"], 4.0, 64)
            out.append((_plane_of(g, y) ** 2).sum((1, 2)))
        return {"intensity": torch.stack(out), "restarts": None}
    grid = _grid(case)
    eps = torch.tensor(_medium(grid, rng), device="cuda")
    if kind in ("apply", "arnoldi"):
        op = _Operator(grid, eps)
        v = _vector(grid, seed, _dtype(case)).double().view((grid.ncomp,) + grid.shape)
        if kind == "apply":
            return op(v[None], case["transpose"]).reshape(-1)
        V, H, beta = _arnoldi(op, v * op.keep, case["m"])
        return {"V": V, "H": H, "beta": beta, "steps": None}
    g = _source(grid, torch.float64).view((grid.ncomp,) + grid.shape)
    omegas = _freqs(case["nfreq"])
    if kind == "stationary":
        return _stationary(_Operator(grid, eps), g, omegas, case)
    if kind == "adjoint":
        from torch.utils.checkpoint import checkpoint
        eps = eps.to(torch.float32).double().requires_grad_()
        y = _response(_Operator(grid, eps), g, omegas, case["T"], 2.0, 40,
                      lambda f, *args: checkpoint(f, *args, use_reentrant=False))
        loss = (_plane_of(grid, y) ** 2).sum()
        grad, = torch.autograd.grad(loss, eps)
        return {"loss": loss.detach(), "grad": grad}
    length, terms = (1.0, 36) if case["prec"] == "fp64" else (4.0, 64)
    y = _response(_Operator(grid, eps), g, omegas, case["T"], length, terms)
    E = _plane_of(grid, y)
    out = {"E": E, "Y": y.reshape(len(omegas), -1), "intensity": (E ** 2).sum((1, 2))}
    if kind == "rstdim":
        out["restarts"] = None
        out["Y"] = out["Y"] if case["full"] else None
    return out


def _stationary(op, g, omegas, case):
    """(A + i W I)^{-1} g for all W by the restarted shifted full
    orthogonalisation method, one basis a restart, with the call's cap."""
    m, nf = case["m"], len(omegas)
    W = torch.as_tensor(omegas, device="cuda")
    start = g * op.keep
    beta = float(torch.linalg.vector_norm(start))
    rho = torch.full((nf,), beta, dtype=torch.complex128, device="cuda")
    z = torch.zeros((nf, g.numel()), dtype=torch.complex128, device="cuda")
    products = 0
    while products < case["cap"]:
        V, H, _ = _arnoldi(op, start, m)
        M = H[:m].to(torch.complex128) + 1j * W[:, None, None] * torch.eye(m, device="cuda")
        rhs = torch.zeros((nf, m, 1), dtype=torch.complex128, device="cuda")
        rhs[:, 0, 0] = rho
        c = torch.linalg.solve(M, rhs)[..., 0]
        z += torch.complex(c.real @ V[:m], c.imag @ V[:m])
        rho = -H[m, m - 1] * c[:, m - 1]
        products += m
        if float(rho.abs().max()) <= 1e-9 * beta:
            break
        start = V[m].view(g.shape)
    return {"zr": z.real.contiguous(), "zi": z.imag.contiguous(), "products": None}
