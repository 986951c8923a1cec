"""The kernels that small grids and the projected problems take, at the sizes
where their splits change, against the general kernels and the oracle.

* The cooperative two-pass Arnoldi process (one block a multiprocessor; groups
  of warps that split the columns; quads or cells) against the per-step
  launches, which kx_arnoldi_noalloc always runs, over every boundary
  condition, layer axis, model and precision that arnoldi() takes.  Both take
  the same steps in the same precision, so they differ by rounding: 1e-11 in
  double precision (as the two entry points are held to elsewhere); in single
  precision each is an FP32 Arnoldi process, and the relation A V = V H that
  both satisfy is held to 2e-6 (as for arnoldi() elsewhere).
* The chunked march of restart in dimension at sample counts around its chunk
  of 16, against the oracle's exact response; with T ||H|| / Nt <= 0.3 the
  sampling error is below 1e-11 (the rule of the default sample grid), and the
  FP64 path is held to 1e-9.
* The projected exponentials at the sizes where a cluster's rows, the series'
  degree and the squarings change, against the oracle, at 1e-11.
"""
import ctypes

import numpy as np
import pytest

import scenario as S
from oracle import exact, krylov, yee

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context, _binding  # noqa: E402

P, C = S.PERIODIC, S.PEC
# one item a thread: quads where nx % 4 == 0, else cells; (nx, ny, nz) from a
# few items to several hundred a multiprocessor, ragged everywhere
GRIDS = {
    "quads_few": S.Grid(3, (8, 3, 5), (P, P, C), 2, 2, 1.0),
    "quads_walls": S.Grid(3, (12, 9, 7), (C, C, C), 0, 2, 0.7),
    "quads_layer_y": S.Grid(3, (16, 14, 11), (P, C, P), 1, 3, 1.0),
    "quads_two_groups": S.Grid(3, (36, 35, 37), (P, P, C), 2, 4, 1.0),
    "quads_one_group": S.Grid(3, (52, 49, 50), (P, P, C), 2, 4, 1.0),
    "quads_past_256_a_block": S.Grid(3, (56, 55, 54), (P, P, C), 2, 4, 1.0),
    "quads_past_384_a_block": S.Grid(3, (64, 61, 62), (P, P, C), 2, 4, 1.0),
    "quads_past_448_a_block": S.Grid(3, (68, 63, 64), (P, P, C), 2, 4, 1.0),
    "quads_too_many": S.Grid(3, (68, 70, 66), (P, P, C), 2, 4, 1.0),
    "cells_few": S.Grid(3, (5, 3, 4), (C, P, C), 2, 1, 1.0),
    "cells_layer_x": S.Grid(3, (21, 18, 23), (C, P, P), 0, 3, 1.0),
    "cells_most": S.Grid(3, (47, 49, 50), (P, P, C), 2, 4, 1.0),
    "cells_too_many": S.Grid(3, (49, 50, 51), (P, P, C), 2, 4, 1.0),
    "2d": S.Grid(2, (37, 29), (C, C), 0, 4, 1.0),
    "2d_wide": S.Grid(2, (211, 130), (P, C), 1, 5, 2.0),
}


def dev(x, dtype):
    return torch.tensor(np.asarray(x), dtype=dtype, device="cuda")


def noalloc(ctx, eps, v0, m):
    """arnoldi() by the per-step launches."""
    lib = _binding.load_library()
    d = _binding.Desc()
    ctypes.memmove(ctypes.byref(d), ctypes.byref(ctx.desc), ctypes.sizeof(d))
    e = dev(eps.reshape(-1), torch.float64)
    V = torch.empty((m + 1, v0.numel()), dtype=v0.dtype, device="cuda")
    H = torch.empty((m, m + 1), dtype=torch.float64, device="cuda")
    beta, md = ctypes.c_double(), ctypes.c_int()
    st = lib.kx_arnoldi_noalloc(ctypes.byref(d), ctypes.c_void_p(e.data_ptr()), ctypes.c_void_p(v0.data_ptr()), m,
                                ctypes.c_void_p(V.data_ptr()), ctypes.c_void_p(H.data_ptr()), ctypes.byref(beta),
                                ctypes.byref(md), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return st, V, H.cpu().numpy().T, beta.value, md.value


@pytest.mark.parametrize("name", list(GRIDS))
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("m", [1, 9, 24])
def test_cooperative_arnoldi_matches_the_per_step_launches(name, prec, m):
    grid = GRIDS[name]
    eps = 1.0 + 3.0 * np.random.default_rng(1).random(grid.shape)
    dt = torch.float64 if prec == "fp64" else torch.float32
    # the per-step entry needs a 16-byte multiple a column: pad-free grids only
    ctx = Context(grid, eps, precision=prec, krylov_dim=max(m, 2))
    v0 = dev(S.masked_random_vector(grid, 5), dt)
    V, H, beta, md = ctx.arnoldi(v0, m)
    assert md == m
    op = yee.Operator(grid, eps)
    Vn = V.double().cpu().numpy().T
    AV = np.stack([op.apply(Vn[:, i]) for i in range(m)], 1)
    assert np.linalg.norm(AV - Vn @ H) < (1e-12 if prec == "fp64" else 2e-6) * np.linalg.norm(AV)
    if grid.nunk * v0.element_size() % 16 == 0:
        st, V2, H2, beta2, md2 = noalloc(ctx, eps, v0, m)
        assert st == 0 and md2 == m
        tol = 1e-11 if prec == "fp64" else 1e-4
        assert abs(beta - beta2) <= (1e-12 if prec == "fp64" else 1e-6) * beta2
        assert np.abs(H - H2).max() < tol * np.abs(H2).max()
        if prec == "fp64":
            assert float((V - V2).abs().max()) < 1e-10
    ctx.close()


@pytest.mark.parametrize("shape", [(8, 6, 9), (9, 6, 8)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_cooperative_arnoldi_breakdown_and_zero(shape, prec):
    """A start vector in a small invariant subspace stops the process early in
    every block alike (columns past it are zero); a non-finite one is refused."""
    grid = S.Grid(3, shape, (P, P, P), 2, 1, 0.0)
    eps = np.full(grid.shape, 2.25)
    dt = torch.float64 if prec == "fp64" else torch.float32
    v = np.zeros(grid.nunk)
    k = 2 * np.pi / shape[0]
    x = yee.node_coords(grid, 4)[0]
    v[4 * grid.ncell:5 * grid.ncell] = np.cos(k * x).reshape(-1)
    ctx = Context(grid, eps, precision=prec, krylov_dim=8)
    V, H, beta, md = ctx.arnoldi(dev(v, dt), 6)
    assert md == 2
    assert float(V[3:].abs().max()) == 0.0
    bad = dev(v, dt)
    bad[3] = float("nan")
    with pytest.raises(_binding.KxError):
        ctx.arnoldi(bad, 6)
    ctx.close()


@pytest.mark.parametrize("nt", [15, 16, 17, 31, 32, 33, 48])
def test_chunked_march_at_sample_counts_around_a_chunk(nt):
    grid = S.Grid(3, (14, 11, 13), (P, P, C), 2, 2, 1.0)
    eps = 1.0 + 3.0 * np.random.default_rng(11).random(grid.shape)
    g = S.masked_random_vector(grid, 12)
    A = yee.Operator(grid, eps).matrix()
    T = 0.04 * nt                       # T ||H|| / Nt about 0.2
    oms = S.freq_list(2)
    ctx = Context(grid, eps, precision="fp64", krylov_dim=12, max_freqs=2, batch=2, rst_samples=64)
    out = ctx.response_restart_dim(dev(g, torch.float64), oms, T, rtol=1e-11, dt_sample=T / nt, plane=(2, 9),
                                   want_full=True)
    ctx.close()
    for f, om in enumerate(oms):
        want = exact.y_plain(A, g, om, T)
        got = out["Y"][f].cpu().numpy()
        assert np.linalg.norm(got - want) < 1e-9 * np.linalg.norm(want)


@pytest.mark.parametrize("m", [2, 3, 15, 16, 17, 33, 63, 64])
@pytest.mark.parametrize("tau", [0.02, 0.3, 1.0, 3.0, 30.0])
def test_cluster_exponentials(m, tau):
    """Rows a block of the cluster from none to four, every series degree and
    up to eight squarings; beta far from one, 0 to 5 frequencies."""
    rng = np.random.default_rng(m)
    H = np.triu(rng.standard_normal((m + 1, m)), -1) * (0.8 / np.sqrt(m))
    H[np.arange(m), np.arange(m)] += 0.5
    grid = S.Grid(2, (16, 16), (C, C), 0, 2, 1.0)
    ctx = Context(grid, np.ones(grid.shape), precision="fp64", krylov_dim=64, max_freqs=5)
    u = ctx.expm_phi_project(H, 1.7e3, tau)
    want = krylov.proj_exp(H, tau, 1.7e3)
    assert np.linalg.norm(u - want) < 1e-11 * np.linalg.norm(want)
    oms = [0.0, 0.3, 0.9, 2.0, -1.1]
    u = ctx.expm_phi_project(H, 1.3e-3, tau, oms)
    for f, om in enumerate(oms):
        want = krylov.proj_sine(H, 1.3e-3, om, tau)
        assert np.linalg.norm(u[f] - want) <= 1e-11 * np.linalg.norm(want)
    ctx.close()
