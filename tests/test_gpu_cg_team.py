"""The small-site CG kernel (one cluster, r0 r1 <= 256; the automatic mode) against the per-stage
kernels: one CTA, odd cluster sizes, several rows per CTA, both sides of the size limit, and its wait
limit.  Local solves run to 1e-10 of the residual, so both agree to 1e-8 of the solution after one
sweep (condition number of these small operators below 1e2)."""
import numpy as np
import pytest

from oracle import qtt_ops as Q
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu

BONDS = [[1] * 9, [1, 2, 2, 2, 2, 2, 2, 2, 1], [1, 2, 3, 3, 3, 3, 3, 2, 1], [1, 2, 4, 5, 5, 5, 4, 2, 1],
         [1, 2, 4, 8, 11, 8, 4, 2, 1], [1, 2, 4, 8, 13, 13, 13, 8, 4, 2, 1], [1, 2, 4, 8, 16, 16, 16, 8, 4, 2, 1],
         [1, 2, 4, 8, 16, 17, 16, 8, 4, 2, 1], [1, 2, 4, 8, 10, 18, 13, 8, 4, 2, 1]]


def solve(qtt, ctx, bonds, mode):
    n = len(bonds) - 1
    rng = np.random.default_rng(sum(bonds))
    ops = Q.Ops(n // 2, n // 2, 40.0, 100.0, 2e-3, "interleaved")
    x0 = [0.1 * rng.standard_normal((bonds[k], 2, bonds[k + 1])) for k in range(n)]
    g = qtt.MPS.from_cores(ctx, x0)
    ctx.set_cg_mode(mode)
    try:
        info = qtt.poisson_solve(ctx, qtt.MPO.from_cores(ctx, ops.Ap), qtt.MPS.from_cores(ctx, inputs.random_cores(n, 4, 80)), g,
                                 1, 1e-10, 600, 1e-10, 0.1)
    finally:
        ctx.set_cg_mode(0)
    return qtt.qtt_decode(ctx, g), info


@pytest.mark.parametrize("bonds", BONDS, ids=lambda b: "-".join(map(str, b)))
def test_cg_team(bonds):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    ctx = qtt.Context(0)
    x, ix = solve(qtt, ctx, bonds, 0)
    y, iy = solve(qtt, ctx, bonds, 1)
    assert (ix["sweeps"], ix["status"]) == (iy["sweeps"], iy["status"])
    assert np.linalg.norm(x - y) <= 1e-8 * np.linalg.norm(y)
    ctx.set_wait_limit(1e-9)                      # reported, and the context stays usable
    with pytest.raises(qtt.QttError) as e:
        solve(qtt, ctx, bonds, 0)
    assert e.value.code == -5
    ctx.set_wait_limit(2.0)
    z, _ = solve(qtt, ctx, bonds, 0)
    assert np.array_equal(x, z)
