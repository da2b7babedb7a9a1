"""mps_dot in one launch (contracted from both ends) against the oracle: one, two and odd numbers of
sites, different bonds of the two trains, d up to 16, both variants (16-CTA cluster up to bond 32,
cooperative grid up to 64) and the site-by-site path above.  Tolerance: sums of at most 64 d products
per entry over n sites, relative to the norms: 64 n eps < 1e-12."""
import numpy as np
import pytest

from oracle import tt
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,ba,bb", [(1, 2, 1, 1), (1, 16, 1, 1), (2, 2, 2, 1), (3, 2, 4, 2), (5, 3, 7, 9), (6, 16, 5, 3),
                                       (12, 2, 16, 16), (13, 2, 32, 31), (14, 2, 33, 8), (20, 2, 64, 64), (11, 4, 64, 37),
                                       (14, 2, 65, 65), (64, 2, 3, 4)])
def test_dot(n, d, ba, bb):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    ctx = qtt.Context(0)
    a = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(n, ba, 11 * n + ba, d=d)]
    b = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(n, bb, 13 * n + bb, d=d)]
    ga, gb = qtt.MPS.from_cores(ctx, a), qtt.MPS.from_cores(ctx, b)
    na, nb = np.sqrt(tt.dot(a, a)), np.sqrt(tt.dot(b, b))
    for _ in range(2):                           # the second call reuses the workspace
        assert abs(qtt.mps_dot(ctx, ga, gb) - tt.dot(a, b)) <= 1e-12 * na * nb
    assert abs(qtt.mps_dot(ctx, ga, ga) - na * na) <= 1e-12 * na * na


def test_dot_bounded_wait():
    """The grid variant's barrier is bounded: with a 1 ns limit the value is either right or NaN, and
    the context stays usable."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    ctx = qtt.Context(0)
    a = [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(12, 48, 3)]
    g = qtt.MPS.from_cores(ctx, a)
    ref = tt.dot(a, a)
    ctx.set_wait_limit(1e-9)
    v = qtt.mps_dot(ctx, g, g)
    assert np.isnan(v) or abs(v - ref) <= 1e-12 * ref
    ctx.set_wait_limit(2.0)
    assert abs(qtt.mps_dot(ctx, g, g) - ref) <= 1e-12 * ref
