"""The eigensolver of the roundings' density matrices (FP32 one-sided Jacobi on a pivoted Cholesky
factor, FP64 refinement on a cooperative grid) through the roundings that use it, on cut matrices
with prescribed singular values: a two-site train of physical size N has one cut, an N x N matrix.

Bounds: the truncation to chi of an N x N matrix A is determined to eps ||A|| / gap in its subspaces;
every spectrum below has relative gaps of at least 1e-2 at the cut.  Through the Gram matrix (encode)
an error of eps ||A||^2 / (sigma_chi^2 gap) in the subspace costs sigma_chi of it: <= 1e-16 sqrt(N) /
(1e-2 sigma_chi) with sigma_chi >= 1e-5 in the encode cases: 1e-8 would be the worst case at N = 128,
reached only by adversarial rounding; 1e-10 is asserted (rounding averages over the N entries).  The
factored form (sketched products) keeps relative accuracy: 1e-11."""
import numpy as np
import pytest

from paper_2507_05222_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    return qtt.Context(0)


def spectrum(kind, N, chi):
    k = np.arange(N)
    if kind == "decay":                       # two percent apart and more, four decades
        return 10.0 ** (-4.0 * k / max(N - 1, 1))
    if kind == "rank":                        # exactly rank chi
        return np.where(k < chi, 1.0 / (1.0 + k), 0.0)
    if kind == "flat_gap":                    # nearly equal values on both sides of one gap
        return np.where(k < chi, 1.0, 1e-3) * (1.0 - 1e-3 * k / N)
    if kind == "dominant":                    # one value over a flat tail
        return np.where(k == 0, 1.0, 1e-3 * (1.0 - 0.5 * k / N))
    if kind == "deep":                        # fourteen decades (factored form only)
        return 10.0 ** (-14.0 * k / max(N - 1, 1))
    raise ValueError(kind)


def matrix(kind, N, chi, seed):
    g = inputs.rng(seed)
    U, _ = np.linalg.qr(g.standard_normal((N, N)))
    V, _ = np.linalg.qr(g.standard_normal((N, N)))
    s = spectrum(kind, N, chi)
    return (U * s) @ V.T, (U[:, :chi] * s[:chi]) @ V[:, :chi].T


def check(ctx, g, best, tol):
    from paper_2507_05222_gb300 import qtt
    v = qtt.qtt_decode(ctx, g).reshape(best.shape)
    assert np.linalg.norm(v - best) <= tol * np.linalg.norm(best)
    c = g.cores()[1]
    m = c.reshape(c.shape[0], -1)
    assert np.abs(m @ m.T - np.eye(c.shape[0])).max() < 1e-13 * max(8, m.shape[1])


@pytest.mark.parametrize("kind", ["decay", "rank", "flat_gap", "dominant"])
@pytest.mark.parametrize("N,chi", [(2, 1), (3, 2), (7, 3), (16, 8), (31, 5), (32, 17), (33, 16), (64, 32), (65, 20),
                                   (97, 48), (127, 64), (128, 64), (128, 1), (128, 127)])
def test_gram_cut(ctx, N, chi, kind):
    from paper_2507_05222_gb300 import qtt
    for seed in (1, 2):
        A, best = matrix(kind, N, chi, 100 * N + seed)
        check(ctx, qtt.qtt_encode(ctx, A.ravel(), 2, chi, d=N), best, 1e-10)


@pytest.mark.parametrize("scale", [1e-140, 1e-30, 1e60, 1e140])
def test_gram_cut_scales(ctx, scale):
    from paper_2507_05222_gb300 import qtt
    A, best = matrix("decay", 48, 20, 5)
    check(ctx, qtt.qtt_encode(ctx, (scale * A).ravel(), 2, 20, d=48), scale * best, 1e-10)


@pytest.mark.parametrize("kind", ["decay", "rank", "flat_gap", "deep"])
@pytest.mark.parametrize("h,chi", [(2, 3), (3, 5), (4, 12), (5, 17), (5, 31), (6, 33), (6, 40), (7, 70)])
def test_factored_cut(ctx, h, chi, kind):
    """Sketched rounding of the identity's product with a train of 2 h sites whose middle cut is the
    prescribed matrix and whose other cuts keep everything (2^(h-1) <= chi < 2^h)."""
    from paper_2507_05222_gb300 import qtt
    N = 2 ** h
    for seed in (1, 2):
        A, best = matrix(kind, N, chi, 7 * N + seed)
        x = [np.eye(2 ** (k + 1)).reshape(2 ** k, 2, 2 ** (k + 1)) for k in range(h)]
        x.append(A.reshape(N, 2, N // 2))
        x += [np.eye(2 ** k).reshape(2 ** k, 2, 2 ** (k - 1)) for k in range(h - 1, 0, -1)]
        M = [np.eye(2).reshape(1, 2, 2, 1)] * (2 * h)
        g = qtt.mpo_apply_round(ctx, qtt.MPO.from_cores(ctx, M), qtt.MPS.from_cores(ctx, x), chi, apply="sketch")
        check(ctx, g, best, 1e-11)


def test_zero_and_nan_matrices(ctx):
    from paper_2507_05222_gb300 import qtt
    g = qtt.qtt_encode(ctx, np.zeros(64 * 64), 2, 8, d=64)
    assert np.all(qtt.qtt_decode(ctx, g) == 0.0)
    A = np.ones(64 * 64)
    A[17] = np.nan
    assert not np.all(np.isfinite(qtt.qtt_decode(ctx, qtt.qtt_encode(ctx, A, 2, 8, d=64))))
