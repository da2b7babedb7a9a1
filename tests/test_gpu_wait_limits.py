"""The wait limit (qtt_ctx_set_wait_limit) outside the solves.  Overlaps and roundings are completed
without waits when one runs out, so that their values do not depend on the limit; with a limit of 1 ns
some wait of every kernel that has grid barriers runs out."""
import numpy as np
import pytest

from oracle import tt
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    return qtt.Context(0)


@pytest.mark.parametrize("n,d,bond", [(3, 2, 33), (12, 2, 48), (20, 2, 64), (7, 4, 64)])
def test_dot_does_not_depend_on_the_limit(ctx, n, d, bond):
    """Tolerance as in test_gpu_dot: 64 n eps < 1e-12 of the norms."""
    from paper_2507_05222_gb300 import qtt
    bonds = [1] + [bond] * (n - 1) + [1]
    a = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(n, bond, 3, d=d, bonds=bonds)]
    b = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(n, bond, 4, d=d, bonds=bonds)]
    ga, gb = qtt.MPS.from_cores(ctx, a), qtt.MPS.from_cores(ctx, b)
    tol = 1e-12 * np.sqrt(tt.dot(a, a) * tt.dot(b, b))
    for limit in (1e-9, 2.0, 1e-9):
        ctx.set_wait_limit(limit)
        for _ in range(3):
            assert abs(qtt.mps_dot(ctx, ga, gb) - tt.dot(a, b)) <= tol
