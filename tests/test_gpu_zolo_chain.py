"""Zolo-pd's first iteration from the chain of inverse Cholesky factors, at
the edges of its blocks (the 64- and 32-column factor, the recursion, the
joint product up to 256 columns) and down to singular inputs: the polar factor
of a matrix built from its singular value decomposition.  ||W^* W - I|| and
||W H - A|| within 50 n u as everywhere; W itself within its condition, u /
sigma_min times the same factor."""
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


def _haar(n, rng, cplx):
    X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
    Q, R = np.linalg.qr(X)
    d = np.diag(R)
    return Q * (d / np.abs(d))


@pytest.mark.parametrize("n,cplx,tc", [(1, False, False), (32, True, False), (33, True, True), (64, False, False),
                                       (65, False, False), (129, False, True), (256, False, True), (257, False, True),
                                       (450, True, True)])
@pytest.mark.parametrize("smin", [1e-3, 1e-13])
def test_polar_of_known_factors(B, n, cplx, tc, smin):
    rng = np.random.default_rng(n)
    Uo, Vo = _haar(n, rng, cplx), _haar(n, rng, cplx)
    s = np.geomspace(1.0, smin, n)
    A = (Uo * s) @ Vo.conj().T
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        W, H, info = ctx.polar(to_dev(A))
        W, H = to_host(W), to_host(H)
    finally:
        ctx.close()
    assert info["zolo_iters"] == 2
    assert np.linalg.norm(W.conj().T @ W - np.eye(n), 2) <= 50 * n * U
    assert np.linalg.norm(W @ H - A) <= 50 * n * U
    assert np.linalg.norm(W - Uo @ Vo.conj().T) <= 50 * n * U / min(smin, s[-1])
