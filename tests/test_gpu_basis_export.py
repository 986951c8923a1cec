"""The exported basis is the stored columns times their double-precision
scales, rounded once: column 0 is v0 / ||v0||, so every one of its values has to
be float(double(v0) * (1 / beta)), as numpy rounds it.  Twelve million values: a
product that carries 48 bits of the scale instead of 53 misses a few of them."""
import numpy as np
import pytest

import scenario as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context  # noqa: E402


@pytest.mark.parametrize("size", [1.0, 3e-12, 7e14])
@pytest.mark.parametrize("shape", [(2048, 2048), (2047, 2045)])
def test_first_column_is_the_rounded_double_product(shape, size):
    grid = S.Grid(2, shape, (S.PERIODIC, S.PERIODIC), 0, 4, 1.0)
    ctx = Context(grid, np.ones(grid.shape), precision="fp32", krylov_dim=2)
    gen = torch.Generator(device="cuda").manual_seed(7)
    v0 = torch.randn(grid.nunk, generator=gen, device="cuda", dtype=torch.float64)
    # magnitudes down to denormal products, and zeros
    v0 *= size * 10.0 ** (-28.0 * (torch.rand(grid.nunk, generator=gen, device="cuda", dtype=torch.float64) < 0.01).double())
    v0[::97] = 0.0
    v0 = v0.float()
    V, H, beta, md = ctx.arnoldi(v0, 1)
    ctx.close()
    want = (v0.double().cpu().numpy() * (1.0 / beta)).astype(np.float32)
    got = V[0].cpu().numpy()
    assert np.array_equal(got, want)
