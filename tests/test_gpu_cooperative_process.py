"""The cooperative Arnoldi process at its own limits, with the route asserted:
its last size and the first one past it (from the device's multiprocessor
count), the sizes where its compiled forms change, the full Krylov dimension,
the PML model, the transposed and the augmented process.

With per-kernel timing on a cooperative process is one pass_a launch; per-step
launches have pass_b too.  A process of m steps in precision u differs from the
exact one by rounding that grows at most with the steps: A V = V H is held to
2e-6 (1e-12 in double precision) as elsewhere, V against the double-precision
process to m u = 4e-6 relative."""
import numpy as np
import pytest

import scenario as S
from oracle import pml, yee

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context, intensity_loss  # noqa: E402

P, C = S.PERIODIC, S.PEC
NSM = torch.cuda.get_device_properties(0).multi_processor_count


def run(ctx, v, m):
    """(launches by class, arnoldi())."""
    ctx.set_timing(True)
    ctx.kernel_times()
    out = ctx.arnoldi(v, m)
    k = {n: t["launches"] for n, t in ctx.kernel_times().items()}
    ctx.set_timing(False)
    return k, out


def relation(ctx, V, H, m):
    """||A V - V H|| / ||A V||, on the device in double precision of the columns."""
    a = torch.stack([ctx.apply_A(V[i]) for i in range(m)]).double()
    r = a - torch.tensor(H, device="cuda").T @ V.double()
    return float(r.norm() / a.norm())


@pytest.mark.parametrize("per_sm,extra", [(256, 0), (256, 1), (384, 0), (384, 1), (448, 0), (448, 1), (512, 0), (512, 1)])
def test_quads_a_multiprocessor_at_the_lines(per_sm, extra):
    """64 x per_sm/8 x NSM/2 cells are per_sm quads a multiprocessor exactly;
    one plane more starts the next form, past 512 the per-step launches."""
    if NSM % 2:
        pytest.skip("an even number of multiprocessors")
    grid = S.Grid(3, (64, per_sm // 8, NSM // 2 + extra), (P, P, C), 2, 4, 1.0)
    eps = 1.0 + 3.0 * np.random.default_rng(1).random(grid.shape)
    ctx = Context(grid, eps, precision="fp32", krylov_dim=12)
    v = torch.tensor(S.masked_random_vector(grid, 5), dtype=torch.float32, device="cuda")
    k, (V, H, beta, md) = run(ctx, v, 12)
    assert md == 12
    if per_sm + extra <= 512:
        assert k["pass_b"] == 0 and k["pass_a"] == 1
    else:
        assert k["pass_b"] == 12
    assert relation(ctx, V, H, 12) < 2e-6
    ctx.close()


@pytest.mark.parametrize("dim,n,bc", [(3, (24, 22, 26), (P, C, C)), (3, (40, 36, 38), (P, P, C)), (3, (25, 22, 27), (C, P, P)),
                                      (3, (52, 50, 49), (P, P, C)), (2, (64, 64), (C, C)), (2, (157, 90), (P, C))])
def test_full_krylov_dimension(dim, n, bc):
    """m = 64: columns past those in shared memory, every chunk of a group."""
    grid = S.Grid(dim, n, bc, dim - 1, 4, 1.0)
    eps = 1.0 + 3.0 * np.random.default_rng(1).random(grid.shape)
    v = S.masked_random_vector(grid, 5)
    got = {}
    for prec, dt, tol in (("fp64", torch.float64, 1e-12), ("fp32", torch.float32, 2e-6)):
        ctx = Context(grid, eps, precision=prec, krylov_dim=64)
        k, (V, H, beta, md) = run(ctx, torch.tensor(v, dtype=torch.float32, device="cuda").to(dt), 64)
        fits = prec == "fp32" or dim == 2 or grid.ncell <= 768 * NSM
        assert md == 64 and (k["pass_b"] == 0) == fits
        assert relation(ctx, V, H, 64) < tol
        got[prec] = (V.double(), H)
        ctx.close()
    a, b = got["fp32"], got["fp64"]
    assert float((a[0] - b[0]).norm() / b[0].norm()) < 4e-6
    assert np.linalg.norm(a[1] - b[1]) < 4e-6 * np.linalg.norm(b[1])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [(37, 29), (120, 85)])
def test_pml(prec, n):
    grid = S.Grid(2, n, (C, P), 0, 4, 3.0, pml=1)
    eps = 1.0 + 3.0 * np.random.default_rng(1).random(grid.shape)
    op = pml.PmlOperator(grid, eps)
    ctx = Context(grid, eps, precision=prec, krylov_dim=30)
    v = S.random_vector(grid.nunk, 3) * S.wall_keep_mask(grid)
    k, (V, H, beta, md) = run(ctx, torch.tensor(v, dtype=torch.float64 if prec == "fp64" else torch.float32,
                                                device="cuda"), 30)
    ctx.close()
    assert k["pass_b"] == 0 and k["pass_a"] == 1 and md == 30
    Vn = V.double().cpu().numpy().T
    AV = np.stack([op.apply(Vn[:, i]) for i in range(30)], 1)
    assert np.linalg.norm(AV - Vn @ H) < (1e-12 if prec == "fp64" else 2e-6) * np.linalg.norm(AV)


def test_unaligned_vectors_take_the_cells():
    """A source that is not on a sixteen-byte boundary: cells instead of quads,
    the same response."""
    sc = S.config_3d(n=24, fill=0.3, T=10.0)
    om = S.freq_list(1)
    y = []
    for shift in (0, 1, 3):
        buf = torch.zeros(sc.grid.nunk + 4, dtype=torch.float32, device="cuda")
        g = buf[shift:shift + sc.grid.nunk]
        g.copy_(torch.tensor(sc.g, dtype=torch.float32))
        ctx = Context(sc.grid, sc.eps_cell, precision="fp32", krylov_dim=40, max_freqs=1, batch=1)
        y.append(ctx.response_at_freqs(g, om, sc.T, rtol=1e-7, method="plain", plane=sc.plane, want_full=True)["Y"][0])
        ctx.close()
    ref = y[0].double()
    for x in y[1:]:
        assert float((x.double() - ref).norm() / ref.norm()) < 2e-6    # each within 1e-6 of the exact field


@pytest.mark.parametrize("n", [24, 36])
def test_gradients_of_quads_and_cells(n):
    """The augmented and the transposed process: gradients from quads in single
    precision against cells in double precision.  Both factors of the gradient
    are fields held to 1e-6; 1e-5 leaves a factor for their cancellation."""
    sc = S.config_3d(n=n, fill=0.3, T=60.0)
    got = {}
    for prec, dt in (("fp64", torch.float64), ("fp32", torch.float32)):
        ctx = Context(sc.grid, sc.eps_cell, precision=prec, krylov_dim=64, max_freqs=1, batch=2, max_checkpoints=64)
        e = torch.tensor(np.asarray(sc.eps_cell), dtype=torch.float64, device="cuda", requires_grad=True)
        g = torch.tensor(sc.g, dtype=dt, device="cuda")
        ctx.set_timing(True)
        ctx.kernel_times()
        intensity_loss(ctx, e, g, S.freq_list(1), sc.T, rtol=1e-11 if prec == "fp64" else 1e-7, plane=sc.plane).backward()
        assert ctx.kernel_times()["pass_b"]["launches"] == 0
        got[prec] = e.grad.double()
        ctx.close()
    assert float((got["fp32"] - got["fp64"]).norm() / got["fp64"].norm()) < 1e-5
