"""Cuts of a rounding that keep everything their matrix can hold (the whole right space, the whole
bond, every left row) take a basis from a QR or the identity instead of an eigenproblem.  The
results hold the exact value, the structural bonds and orthonormal rows, for sums, products (both
roundings), Hadamard starts and encodings, at the smallest shapes, odd bonds and d = 3.

Tolerance: a chain of n Householder factorisations and projections of matrices with at most 256
columns loses a few eps sqrt(256) per site: n * 16 * 4 eps <= 3e-13 at n = 20; 1e-12 is asserted."""
import numpy as np
import pytest

from oracle import tt
from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    return qtt.Context(0)


def cores(n, b, seed, d=2):
    return [c / np.sqrt(c.shape[1] * c.shape[2]) for c in inputs.random_cores(n, b, seed, d=d)]


def check(ctx, g, ref, bonds):
    from paper_2507_05222_gb300 import qtt
    assert g.bonds() == bonds
    v = qtt.qtt_decode(ctx, g)
    assert np.linalg.norm(v - ref) <= TOL * np.linalg.norm(ref)
    for c in g.cores()[1:]:
        m = c.reshape(c.shape[0], -1)
        assert np.abs(m @ m.T - np.eye(c.shape[0])).max() < TOL


def structural(pre, d, chi):
    m = [1]
    for k in range(1, len(pre)):
        m.append(min(pre[k], d * m[-1]))
    ob = [1] * len(pre)
    for k in range(len(pre) - 2, 0, -1):
        ob[k] = min(chi, m[k], d * ob[k + 1])
    return ob


@pytest.mark.parametrize("n,d,ba,bb", [(2, 2, 1, 1), (2, 2, 2, 2), (3, 2, 2, 1), (5, 3, 4, 3), (9, 2, 5, 12),
                                       (12, 2, 33, 20), (20, 2, 7, 16)])
def test_sum_without_truncation(ctx, n, d, ba, bb):
    from paper_2507_05222_gb300 import qtt
    x, y = cores(n, ba, 1 + n, d), cores(n, bb, 2 + n, d)
    pre = [1] + [x[k].shape[2] + y[k].shape[2] for k in range(n - 1)] + [1]
    for chi in (ba + bb, ba + bb + 9):
        info = {}
        g = qtt.mps_axpby_round(ctx, 0.7, qtt.MPS.from_cores(ctx, x), -1.3, qtt.MPS.from_cores(ctx, y), chi,
                                out_info=info)
        check(ctx, g, 0.7 * tt.full(x) - 1.3 * tt.full(y), structural(pre, d, chi))
        assert info["discarded_norm"] <= 1e-12 * info["norm"]


@pytest.mark.parametrize("apply", ["gram", "sketch"])
@pytest.mark.parametrize("n,d,b,w", [(2, 2, 2, 2), (3, 2, 1, 3), (5, 3, 3, 2), (9, 2, 7, 5), (12, 2, 12, 8), (16, 2, 5, 9)])
def test_product_without_truncation(ctx, n, d, b, w, apply):
    from paper_2507_05222_gb300 import qtt
    x, M = cores(n, b, 3 + n, d), inputs.random_mpo_cores(n, w, 4 + n, d=d)
    M = [c / np.sqrt(c.shape[2] * c.shape[3]) for c in M]
    y = tt.mpo_mps(M, x)
    pre = [1] + [c.shape[2] for c in y]
    g = qtt.mpo_apply_round(ctx, qtt.MPO.from_cores(ctx, M), qtt.MPS.from_cores(ctx, x), b * w, apply=apply)
    check(ctx, g, tt.full(y), structural(pre, d, b * w))


@pytest.mark.parametrize("n,d", [(1, 2), (2, 2), (5, 2), (9, 2), (12, 2), (14, 2), (5, 3)])
def test_encode_at_full_rank(ctx, n, d):
    from paper_2507_05222_gb300 import qtt
    v = inputs.rng(n + d).standard_normal(d ** n)
    for chi in (d ** (n // 2), d ** (n // 2) + 5):
        if d * chi > 256:
            continue
        g = qtt.qtt_encode(ctx, v, n, chi, d=d)
        check(ctx, g, v, [min(d ** k, d ** (n - k)) for k in range(n + 1)])


@pytest.mark.parametrize("n,ba,bb", [(2, 2, 2), (7, 3, 4), (11, 5, 6)])
def test_hadamard_at_the_exact_bond(ctx, n, ba, bb):
    """Zip-up start and one fit sweep at the bond of the exact product (the start alone is not exact:
    it cuts to the structural bonds without the left part)."""
    from paper_2507_05222_gb300 import qtt
    x, y = cores(n, ba, 5 + n), cores(n, bb, 6 + n)
    g = qtt.mps_hadamard_round(ctx, qtt.MPS.from_cores(ctx, x), qtt.MPS.from_cores(ctx, y), ba * bb, sweeps=1)
    ref = tt.full(x) * tt.full(y)
    assert np.linalg.norm(qtt.qtt_decode(ctx, g) - ref) <= TOL * np.linalg.norm(ref)


def test_order_above_256_stays_refused(ctx):
    """Bond 160 (order 320) is refused whether or not a cut would truncate."""
    from paper_2507_05222_gb300 import qtt
    x, M = inputs.random_cores(18, 32, 1), inputs.random_mpo_cores(18, 5, 2)
    with pytest.raises(qtt.QttError) as e:
        qtt.mpo_apply_round(ctx, qtt.MPO.from_cores(ctx, M), qtt.MPS.from_cores(ctx, x), 160)
    assert e.value.code == -7
    with pytest.raises(qtt.QttError) as e:
        qtt.qtt_encode(ctx, np.ones(2 ** 17), 17, 160)
    assert e.value.code == -7
