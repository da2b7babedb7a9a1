"""The wait limit (qtt_ctx_set_wait_limit) outside the solves.  Overlaps and roundings are completed
without waits when one runs out, so that their values do not depend on the limit; with a limit of 1 ns
some wait of every kernel that has grid barriers runs out.  The waits of the cluster QR have a limit of
their own, and one that runs out is reported by the next call that reads results back."""
import numpy as np
import pytest

from oracle import qtt_ops as Q, step as S, tt
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


def matrix(N, chi, decades, seed):
    """A matrix of singular values over the given decades and its best approximation of rank chi."""
    g = inputs.rng(seed)
    U, _ = np.linalg.qr(g.standard_normal((N, N)))
    V, _ = np.linalg.qr(g.standard_normal((N, N)))
    s = 10.0 ** (-decades * np.arange(N) / max(N - 1, 1))
    return (U * s) @ V.T, (U[:, :chi] * s[:chi]) @ V[:, :chi].T


@pytest.mark.parametrize("N,chi", [(2, 1), (9, 4), (33, 16), (64, 30), (128, 64)])
def test_encode_does_not_depend_on_the_limit(ctx, N, chi):
    """One truncating cut through its density matrix; bound as in test_gpu_psd_eig (1e-10)."""
    from paper_2507_05222_gb300 import qtt
    A, best = matrix(N, chi, 4.0, N)
    for limit in (2.0, 1e-9, 2.0):
        ctx.set_wait_limit(limit)
        info = {}
        v = qtt.qtt_decode(ctx, qtt.qtt_encode(ctx, A.ravel(), 2, chi, d=N, out_info=info)).reshape(N, N)
        assert np.linalg.norm(v - best) <= 1e-10 * np.linalg.norm(best)
        assert abs(info["norm"] - np.linalg.norm(best)) <= 1e-10 * np.linalg.norm(best)


@pytest.mark.parametrize("h,chi,decades", [(4, 12, 4.0), (5, 17, 14.0), (6, 40, 14.0)])
def test_sketched_product_does_not_depend_on_the_limit(ctx, h, chi, decades):
    """The factored form, whose levels go on to the end of fourteen decades; bound as in
    test_gpu_psd_eig (1e-11)."""
    from paper_2507_05222_gb300 import qtt
    N = 2 ** h
    A, best = matrix(N, chi, decades, 7 * N)
    x = [np.eye(2 ** (k + 1)).reshape(2 ** k, 2, 2 ** (k + 1)) for k in range(h)]
    x.append(A.reshape(N, 2, N // 2))
    x += [np.eye(2 ** k).reshape(2 ** k, 2, 2 ** (k - 1)) for k in range(h - 1, 0, -1)]
    M = [np.eye(2).reshape(1, 2, 2, 1)] * (2 * h)
    gM, gx = qtt.MPO.from_cores(ctx, M), qtt.MPS.from_cores(ctx, x)
    for limit in (1e-9, 2.0):
        ctx.set_wait_limit(limit)
        v = qtt.qtt_decode(ctx, qtt.mpo_apply_round(ctx, gM, gx, chi, apply="sketch")).reshape(N, N)
        assert np.linalg.norm(v - best) <= 1e-11 * np.linalg.norm(best)


def readers(qtt, ctx):
    """Calls that read results back."""
    ne = 3
    ops = Q.Ops(ne, ne, 40.0, 100.0, 2e-3, "interleaved")
    cores = inputs.random_cores(2 * ne, 4, seed=1)
    g = qtt.MPS.from_cores(ctx, cores)
    A, b = qtt.MPO.from_cores(ctx, ops.Ap), qtt.MPS.from_cores(ctx, inputs.random_cores(2 * ne, 4, seed=80))
    def case():
        u, v = (ops.encode(f, 8) for f in (1.0 + inputs.gaussian_field(ne, ne, 1, 1e-3), inputs.gaussian_field(ne, ne, 2, 1e-3)))
        p = S.padded([np.zeros((1, 2, 1))] * (2 * ne), 8, inputs.random_cores(2 * ne, 8, 3, scale=1e-8))
        c = qtt.Case(ctx, ne, ne, 40.0, 100.0, 2e-3, 8, "interleaved")
        c.set_state(*(qtt.MPS.from_cores(ctx, x) for x in (u, v, p)))
        return c
    one, two = case(), case()
    return {"sync": ctx.sync, "dot": lambda: qtt.mps_dot(ctx, g, g), "decode": lambda: qtt.qtt_decode(ctx, g),
            "cores": g.cores, "round": lambda: qtt.qtt_round(ctx, g, 4, out_info={}),
            "threshold": lambda: qtt.qtt_round(ctx, g, 4, rel_tol=1e-3), "qr": lambda: qtt.qtt_qr(ctx, np.eye(64), path=2),
            "solve": lambda: qtt.poisson_solve(ctx, A, b, qtt.MPS.from_cores(ctx, inputs.random_cores(2 * ne, 8, seed=81)),
                                               8, 1e-9, 300, 1e-2, 0.1),
            "step": lambda: one.fractional_step(1), "forces": one.forces,
            "batch": lambda: qtt.fractional_step_batch(ctx, [one, two], 1)}


def test_expired_qr_wait_is_reported_once(ctx):
    """A cluster QR with a limit of 1 ns gives up; the next call that reads back returns
    QTT_ERR_TIMEOUT, the one after that works."""
    from paper_2507_05222_gb300 import qtt
    calls = readers(qtt, ctx)
    for f in calls.values():
        f()
    for m, n in ((64, 32), (128, 64), (256, 128), (320, 160), (16, 16)):
        qtt.qtt_check_qr_wait(ctx, m, n, 1e-9)
        with pytest.raises(qtt.QttError) as e:
            ctx.sync()
        assert e.value.code == -5 and "timed out" in str(e.value)
        qtt.qtt_check_qr_wait(ctx, m, n, 2.0)
        ctx.sync()
    for name, f in calls.items():
        qtt.qtt_check_qr_wait(ctx, 128, 64, 1e-9)
        with pytest.raises(qtt.QttError) as e:
            f()
        assert e.value.code == -5, name
        f()
    ctx.set_wait_limit(1e-9)                      # the QR's waits do not follow the limit of the solves
    A = inputs.rng(3).standard_normal((128, 64))
    q, r = qtt.qtt_qr(ctx, A, path=2)
    assert np.linalg.norm(q @ r - A) <= 1e-13 * np.linalg.norm(A)
