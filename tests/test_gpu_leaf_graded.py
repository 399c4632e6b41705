"""Spectra graded over FP64's range, as small angles give (lambda = sin theta -
cos theta): the leaf eigensolver resolves them by passes of its FP32 stage and
refinement, each a few times a well separated spectrum's one pass, and not by
the FP64 finish, which takes seconds at 1000 rows."""
import numpy as np
import pytest

from tests.gpu_util import U, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    return binding


def _spectrum(kind, n, rng):
    if kind == "powers":
        return 2.0 ** (-np.arange(n) * 40.0 / n)
    if kind == "angles":
        th = np.pi / 2 * 10.0 ** (-12 * rng.random(n))
        return np.sin(th) - np.cos(th)
    if kind == "flat":  # a few large ones over a narrow rest
        return np.concatenate([rng.uniform(0.5, 1, 5), 1e-6 * rng.uniform(-1, 1, n - 5)])
    return rng.uniform(-1, 1, n)


def _heig(ctx, kind, n, cplx):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
    Q = np.linalg.qr(X)[0]
    M = (Q * _spectrum(kind, n, rng)) @ Q.conj().T
    M = (M + M.conj().T) / 2
    d = to_dev(M)
    best = np.inf
    for _ in range(4):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        lam, V, _ = ctx.heig(d)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return M, to_host(lam), to_host(V), best


@pytest.mark.parametrize("n,cplx,tc", [(100, True, False), (250, False, False), (250, True, False), (500, False, True),
                                       (1000, False, True)])
@pytest.mark.parametrize("kind", ["powers", "angles", "flat"])
def test_graded_spectrum(B, n, cplx, tc, kind):
    """The bars, and the time: at most eight passes, each with at most eight
    looks at the refinement where the separated spectrum's only pass has three
    or more, so 8 * 8 / 3 times its time bounds it."""
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        *_, ref = _heig(ctx, "even", n, cplx)
        M, lam, V, ms = _heig(ctx, kind, n, cplx)
    finally:
        ctx.close()
    nb = np.linalg.norm(M, 2)
    assert np.max(np.abs(lam - np.linalg.eigvalsh(M))) <= 50 * n * U * nb
    assert np.linalg.norm(M @ V - V * lam) <= 50 * n * U * nb
    assert np.linalg.norm(V.conj().T @ V - np.eye(n), 2) <= 50 * n * U
    assert ms <= 8 * 8 / 3 * ref, (ms, ref)
