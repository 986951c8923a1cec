"""Projected solutions whose frequencies or scales lie far apart: the scaling
and squaring of one frequency is not another's, and not the source column's,
so each is as accurate as in a call of its own and in other units of time."""
import numpy as np
import pytest

import scenario as S
from oracle import krylov

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_1707_00023_gb300 import Context  # noqa: E402


def hessenberg(m):
    """Nearly skew-symmetric with a small damping, as the operator's are."""
    rng = np.random.default_rng(m)
    H = 0.05 * np.triu(rng.standard_normal((m + 1, m)))
    i = np.arange(m)
    b = rng.uniform(0.8, 1.8, m)
    H[i + 1, i] = b
    H[i[:-1], i[1:]] -= b[:-1]
    H[i, i] += rng.uniform(0.0, 0.3, m)
    return H


@pytest.fixture(scope="module")
def ctx():
    grid = S.Grid(2, (16, 16), (S.PEC, S.PEC), 0, 2, 1.0)
    c = Context(grid, np.ones(grid.shape), precision="fp64", krylov_dim=64, max_freqs=64)
    yield c
    c.close()


@pytest.mark.parametrize("m", [1, 12, 64])
@pytest.mark.parametrize("others", [(300.0,), (3e4, 20.0), tuple(np.geomspace(0.5, 5e3, 63))])
def test_a_slow_frequency_beside_fast_ones(ctx, m, others):
    H = hessenberg(m) if m > 1 else np.array([[0.4], [0.3]])
    both = ctx.expm_phi_project(H, 1.0, 10.0, [0.4, *others])
    for f in range(min(3, len(others) + 1)):
        om = [0.4, *others][f]
        alone = ctx.expm_phi_project(H, 1.0, 10.0, [om])[0]
        # a scaling of at most one squaring more than its own
        tol = 4e-15 if om < 1.0 else 1e-14 * max(1.0, om)
        assert np.linalg.norm(both[f] - alone) <= tol * np.linalg.norm(alone)
    want = krylov.proj_sine(H, 1.0, 0.4, 10.0)
    assert np.linalg.norm(both[0] - want) < 1e-13 * np.linalg.norm(want)


@pytest.mark.parametrize("k", [0, 10, 20, 30])
@pytest.mark.parametrize("beta", [1.0, 2.0 ** -12, 2.0 ** 15])
def test_other_units_of_time(ctx, k, beta):
    """H, W and 1 / tau in units 2^k smaller give 2^k times the solution: powers
    of two, so only the scaling could differ."""
    m, c = 12, 2.0 ** -k
    H = hessenberg(m)
    u = ctx.expm_phi_project(H, 1.0, 10.0, [0.4, 1.2])
    v = ctx.expm_phi_project(H * c, beta, 10.0 / c, [0.4 * c, 1.2 * c])
    for f in range(2):
        assert np.linalg.norm(v[f] * (c / beta) - u[f]) < 4e-15 * np.linalg.norm(u[f])
