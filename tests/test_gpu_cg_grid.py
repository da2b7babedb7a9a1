"""The one-kernel CG solves (FP64 and tensor cores) against the per-stage kernels where the spread of the
vectors over the grid changes: fewer elements than warps in the grid, one to seven warps a CTA, odd bonds.
Local solves run to 1e-10 of the residual, so both agree to 1e-8 of the solution after one sweep."""
import numpy as np
import pytest

from oracle import qtt_ops as Q
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mid", [1, 3, 17, 47, 64, 100])
@pytest.mark.parametrize("mode", [2, 3])
def test_cg_grid(mid, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    ctx = qtt.Context(0)
    n = 14
    bonds = [min(2 ** k, 2 ** (n - k), mid) for k in range(n + 1)]
    rng = np.random.default_rng(mid)
    ops = Q.Ops(n // 2, n // 2, 40.0, 100.0, 2e-3, "interleaved")
    A = qtt.MPO.from_cores(ctx, ops.Ap)
    b = qtt.MPS.from_cores(ctx, inputs.random_cores(n, 4, 80))
    x0 = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2.0 * bonds[k + 1]) for k in range(n)]
    out = []
    for m in (1, mode):
        ctx.set_cg_mode(m)
        x = qtt.MPS.from_cores(ctx, x0)
        info = qtt.poisson_solve(ctx, A, b, x, 1, 1e-10, 1000, 1e-10, 0.1)
        out.append((qtt.qtt_decode(ctx, x), info))
    ctx.set_cg_mode(0)
    (y, iy), (z, iz) = out
    assert (iy["sweeps"], iy["status"]) == (iz["sweeps"], iz["status"])
    assert np.linalg.norm(z - y) <= 1e-8 * np.linalg.norm(y)
