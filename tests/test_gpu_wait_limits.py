"""The bounded wait of the cooperative Arnoldi process, run out without a
fault: with a limit of no polls (or of one, which the first block to arrive
uses up) every block gives up and returns, each entry point hands on
KX_ETIMEOUT with a text that says so, and the context then computes as before."""
import numpy as np
import pytest

import scenario as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context, KxError, intensity_loss  # noqa: E402

FULL = 2097152


def calls(ctx, sc, g, eps):
    om = S.freq_list(2)

    def gradient():
        e = eps.clone().requires_grad_(True)
        intensity_loss(ctx, e, g, om, sc.T, rtol=1e-6, plane=sc.plane).backward()
        return e.grad

    return {
        "arnoldi": lambda: ctx.arnoldi(g, 12)[0],
        "stationary": lambda: ctx.stationary_solve(g, om, rtol=1e-6, max_matvecs=48, allow_noconv=True)[0],
        "expm": lambda: ctx.expm_action(g, sc.T, rtol=1e-6)[0],
        "plain": lambda: ctx.response_at_freqs(g, om, sc.T, rtol=1e-6, method="plain", plane=sc.plane,
                                               want_full=True)["Y"],
        "split2": lambda: ctx.response_at_freqs(g, om, sc.T, rtol=1e-6, method="split2", plane=sc.plane,
                                                want_full=True)["Y"],
        "rstdim": lambda: ctx.response_restart_dim(g, om, sc.T, rtol=1e-6, plane=sc.plane, want_full=True)["Y"],
        "adjoint": gradient,
    }


@pytest.mark.parametrize("polls", [0, 1])
@pytest.mark.parametrize("name", ["arnoldi", "stationary", "expm", "plain", "split2", "rstdim", "adjoint"])
def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(name, polls):
    sc = S.config_3d(n=24, fill=0.3, T=6.0)
    g = torch.tensor(sc.g, dtype=torch.float32, device="cuda")
    eps = torch.tensor(np.asarray(sc.eps_cell), dtype=torch.float32, device="cuda")
    ctx = Context(sc.grid, sc.eps_cell, precision="fp32", krylov_dim=24, max_freqs=2, batch=2, rst_samples=256,
                  max_checkpoints=32)
    call = calls(ctx, sc, g, eps)[name]
    before = call().clone()
    ctx.set_wait_limit(polls)
    with pytest.raises(KxError, match="KX_ETIMEOUT") as err:
        call()
    assert "wait ran out" in str(err.value)
    ctx.set_wait_limit(FULL)
    assert torch.equal(call(), before)
    with pytest.raises(KxError, match="KX_EINVAL"):
        ctx.set_wait_limit(FULL + 1)
    ctx.close()

