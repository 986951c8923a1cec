"""Which form of the Arnoldi process a call takes, by the launches it records
with per-kernel timing on: two-pass processes on their own launches have pass_b
launches, a cooperative process is one pass_a launch alone, the single sweep has
its own class."""
import numpy as np
import pytest

import scenario as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context  # noqa: E402

P, C = S.PERIODIC, S.PEC


def launches(ctx, call):
    ctx.set_timing(True)
    ctx.kernel_times()
    call()
    kt = ctx.kernel_times()
    ctx.set_timing(False)
    return {k: v["launches"] for k, v in kt.items()}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_default_form_of_restart_in_dimension_between_the_size_lines(prec):
    """1.5e6 unknowns: the single sweep in single precision; in double
    precision, where it took twice as long as the two passes, the two passes."""
    grid = S.Grid(2, (704, 704), (C, C), 0, 8, 1.0)
    ctx = Context(grid, np.ones(grid.shape), precision=prec, krylov_dim=12, max_freqs=1, batch=2, rst_samples=256)
    g = torch.zeros(grid.nunk, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    g[2 * grid.ncell + 350 * 704 + 350] = 1.0
    k = launches(ctx, lambda: ctx.response_restart_dim(g, [0.4], 1.0, rtol=1e-6, plane=(0, 360)))
    ctx.close()
    if prec == "fp64":
        assert k["sweep"] == 0 and k["pass_a"] > 0
    else:
        assert k["sweep"] > 0 and k["pass_b"] == 0


@pytest.mark.parametrize("dim,n,prec,m", [(3, 24, "fp32", 64), (3, 36, "fp32", 40), (3, 25, "fp32", 40), (2, 64, "fp64", 30),
                                          (2, 96, "fp32", 30), (3, 16, "fp64", 30)])
def test_lockstep_batch_on_a_small_grid_shares_its_launches(dim, n, prec, m):
    """Sixteen frequencies in lockstep: a small grid's process holds nearly
    every multiprocessor, and run one slot after the other they took up to
    twice as long as by the per-step launches.  Either those run, or one
    launch serves several slots; the fields are those of one frequency at a
    time, each held to its own distance from the exact ones elsewhere (1e-6 in
    single precision, 1e-10 in double)."""
    sc = S.config_2d(n=n, ndisks=2, T=12.0) if dim == 2 else S.config_3d(n=n, fill=0.3, T=12.0)
    dt = torch.float64 if prec == "fp64" else torch.float32
    g = torch.tensor(sc.g, dtype=dt, device="cuda")
    oms = S.freq_list(16)
    rtol = 1e-11 if prec == "fp64" else 1e-7
    many = Context(sc.grid, sc.eps_cell, precision=prec, krylov_dim=m, max_freqs=16, batch=16)
    out = {}

    def call():
        out["Y"] = many.response_at_freqs(g, oms, sc.T, rtol=rtol, method="plain", plane=sc.plane, want_full=True)["Y"]

    many.reset_stats()
    k = launches(many, call)
    steps = many.stats()["substeps"]
    assert steps >= 16
    assert k["pass_b"] > 0 or k["pass_a"] <= steps / 2
    many.close()
    one = Context(sc.grid, sc.eps_cell, precision=prec, krylov_dim=m, max_freqs=1, batch=1)
    for f in (0, 7, 15):
        y = one.response_at_freqs(g, oms[f:f + 1], sc.T, rtol=rtol, method="plain", plane=sc.plane, want_full=True)["Y"][0]
        d = (out["Y"][f].double() - y.double()).norm() / y.double().norm()
        assert float(d) < (2e-10 if prec == "fp64" else 2e-6)
    one.close()


@pytest.mark.parametrize("method", ["plain", "rstdim"])
def test_threaded_driver_overlaps_the_contexts(method):
    """Eight 24^3 problems.  Alone a context's process takes launches that hold
    most of the GPU; from four threads they must leave room for the others':
    the best of three calls is then at most 0.8 times that from one thread
    (0.3 to 0.45 where they overlap, 0.95 to 1.1 where they queue).
    Intensities within the accuracy of each (fields within 1e-6, so 4e-6)."""
    import time

    from paper_1707_00023_gb300 import response_multi
    sc = S.config_3d(n=24, fill=0.3, T=30.0)
    oms = S.freq_list(2)
    g = torch.tensor(sc.g, dtype=torch.float32, device="cuda")
    ctxs = [Context(sc.grid, sc.eps_cell, precision="fp32", krylov_dim=64, max_freqs=2, batch=2, stream="own",
                    rst_samples=1024) for _ in range(8)]
    torch.cuda.synchronize()
    best, inten = {}, {}
    for threads in (1, 4):
        for _ in range(4):
            t = time.perf_counter()
            inten[threads], _ = response_multi(ctxs, [g] * 8, np.tile(oms, (8, 1)), sc.T, rtol=1e-7, method=method,
                                               planes=np.array([sc.plane] * 8), nthreads=threads)
            t = time.perf_counter() - t
            best[threads] = min(t, best.get(threads, t))
    for c in ctxs:
        c.close()
    assert np.abs(inten[4] - inten[1]).max() < 4e-6 * np.abs(inten[1]).max()
    assert best[4] < 0.8 * best[1]
