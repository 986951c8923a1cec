"""The projected work on clusters of eight blocks, the form for devices that
cannot place one of sixteen: every entry point that uses it gives the same bits
(the blocks own other rows, the operations are the same)."""
import numpy as np
import pytest

import scenario as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context, KxError, intensity_loss  # noqa: E402


@pytest.mark.parametrize("m", [1, 7, 8, 9, 16, 31, 63, 64])
def test_exponentials(m):
    rng = np.random.default_rng(m)
    H = np.triu(rng.standard_normal((m + 1, m)), -1) * (0.8 / np.sqrt(m))
    grid = S.Grid(2, (16, 16), (S.PEC, S.PEC), 0, 2, 1.0)
    ctx = Context(grid, np.ones(grid.shape), precision="fp64", krylov_dim=64, max_freqs=64)
    got = {}
    for blocks in (16, 8):
        ctx.set_cluster_blocks(blocks)
        got[blocks] = [ctx.expm_phi_project(H, 1.0, tau, om) for tau in (0.02, 1.0, 30.0)
                       for om in (None, [0.4], list(np.linspace(-2.0, 2.0, 64)))]
    for a, b in zip(got[8], got[16]):
        assert np.array_equal(a, b)
    with pytest.raises(KxError, match="KX_EINVAL"):
        ctx.set_cluster_blocks(4)
    ctx.close()


@pytest.mark.parametrize("prec,m", [("fp32", 64), ("fp64", 21)])
def test_responses_and_gradients(prec, m):
    sc = S.config_3d(n=12, fill=0.3, T=15.0)
    dt = torch.float32 if prec == "fp32" else torch.float64
    g = torch.tensor(sc.g, dtype=dt, device="cuda")
    om = S.freq_list(3)
    out = {}
    for blocks in (16, 8):
        ctx = Context(sc.grid, sc.eps_cell, precision=prec, krylov_dim=m, max_freqs=3, batch=3, rst_samples=512,
                      max_checkpoints=64)
        ctx.set_cluster_blocks(blocks)
        y = [ctx.response_at_freqs(g, om, sc.T, rtol=1e-7, method="plain", plane=sc.plane, want_full=True)["Y"],
             ctx.response_restart_dim(g, om, sc.T, rtol=1e-7, plane=sc.plane, want_full=True)["Y"]]
        e = torch.tensor(np.asarray(sc.eps_cell), dtype=dt, device="cuda", requires_grad=True)
        intensity_loss(ctx, e, g, om[:2], sc.T, rtol=1e-7, plane=sc.plane).backward()
        out[blocks] = [*y, e.grad]
        torch.cuda.synchronize()
        ctx.close()
    for a, b in zip(out[8], out[16]):
        assert torch.equal(a, b)
