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
