"""The cluster QR at the edges of its work split, against LAPACK: a last panel of one column, cluster
sizes with and without split panels, both sides of 128 and 256 rows (one to eight rows a lane, then
shared memory), and columns scaled by powers of two up to 2^+-500 -- a positive column scaling leaves Q
alone and scales R's columns.  Tolerance as for well-conditioned Gaussian blocks: condition (< 1e3) x
64-bit rounding < 1e-12."""
import numpy as np
import pytest

from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(17, 16), (33, 33), (64, 61), (128, 32), (129, 65), (256, 127), (257, 100), (260, 17),
                                 (300, 64)])
@pytest.mark.parametrize("trans", [False, True])
def test_qr_cluster_edges(m, n, trans):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    ctx = qtt.Context(0)
    g = inputs.rng(31 * m + n)
    A = g.standard_normal((m, n))
    # below n = m the smallest singular value stays away from zero; shift the square block
    if m < n + 4:
        A[:n] += 2.0 * np.sqrt(n) * np.eye(n)
    Qn, Rn = np.linalg.qr(A)
    for scale in (np.ones(n), 2.0 ** np.round(g.uniform(-500, 500, n))):
        B = A * scale
        Q, R = qtt.qtt_qr(ctx, B.T.copy() if trans else B, trans=trans, path=2)
        Q = Q.T if trans else Q
        assert np.abs(Q - Qn).max() <= 1e-12
        assert np.abs(R / scale - Rn).max() <= 1e-12 * np.abs(Rn).max()


def test_scalars_over_the_reflectors_range():
    """The reciprocal and the square root that form a reflector, over what it meets: squared norms of
    columns scaled to a largest entry in [1, 2), from 2^-960 (below it the reflector is the
    identity) to 4 m, and the products of two norms.  Half an ulp from the last rounding, a quarter from the
    correction's and e^3 < 2^-57 of the series: 2 ulp = 4.5e-16 with room for the product's rounding."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import inputs, qtt
    g = inputs.rng(31)
    x = np.concatenate([2.0 ** g.uniform(-960, 12, 40000), g.uniform(0.5, 4.0, 40000), np.arange(1, 1000) ** 2.0,
                        [2.0 ** -960, 2.0 ** -959, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0)]])
    rcp, sqrt = qtt.qtt_check_recip(qtt.Context(0), x)
    assert rcp <= 4.5e-16 and sqrt <= 4.5e-16
