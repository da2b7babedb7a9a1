"""Rounding to a threshold beyond the bonds of the QR + SVD path (one CTA's shared memory: 128 x 128
cores do not fit), where the rank of a cut is chosen from its eigenvalues afterwards: every kept
vector has to be resolved then, not only the space of all of them.

The middle unfolding of a train of 14 sites is a 128 x 128 matrix with prescribed singular values, 50
in [0.9, 1] and two at 0.1 (1 +- delta) around the threshold 0.1; the other unfoldings keep all of
their singular values (asserted).  Exact result: the matrix without its singular values below 0.1.
Bound: the Gram eigenproblem determines the two vectors to the angle n eps / (4 delta 0.1^2), n = 128,
which costs 0.1 of it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = 7
N = 2 ** H


def matrices(delta, seed):
    """The matrix, its exact truncation and the train of the matrix."""
    g = np.random.default_rng(1000 + seed)
    U, _ = np.linalg.qr(g.standard_normal((N, N)))
    V, _ = np.linalg.qr(g.standard_normal((N, N)))
    s = np.zeros(N)
    s[:50] = np.linspace(1.0, 0.9, 50)
    s[50:52] = 0.1 * (1.0 + delta), 0.1 * (1.0 - delta)
    A, best = (U * s) @ V.T, (U[:, :51] * s[:51]) @ V[:, :51].T
    x = [np.eye(2 ** (k + 1)).reshape(2 ** k, 2, 2 ** (k + 1)) for k in range(H)]
    x.append(A.reshape(N, 2, N // 2))
    x += [np.eye(2 ** k).reshape(2 ** k, 2, 2 ** (k - 1)) for k in range(H - 1, 0, -1)]
    return A, best, x


@pytest.mark.parametrize("delta,seed", [(1e-1, 0), (1e-3, 1), (1e-4, 0), (1e-4, 1), (1e-5, 0), (1e-5, 1), (1e-5, 2)])
def test_threshold_between_close_singular_values(delta, seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2507_05222_gb300 import qtt
    A, best, x = matrices(delta, seed)
    for k in range(1, 2 * H):
        if k != H:
            sv = np.linalg.svd(best.reshape(2 ** k, -1), compute_uv=False)
            assert sv[-1] > 0.105 * sv[0]
    ctx = qtt.Context(0)
    g = qtt.qtt_round(ctx, qtt.MPS.from_cores(ctx, x), N, rel_tol=0.1)
    v = qtt.qtt_decode(ctx, g).reshape(N, N)
    assert g.bonds()[H] == 51
    tol = 0.1 * N * np.finfo(float).eps / (4.0 * delta * 0.01) + 1e-13
    assert np.linalg.norm(v - best, 2) <= tol
