"""The batched leaf eigensolver (leaf.cu): FP32 Jacobi, FP64 refinement and
the FP64 finish, at the sizes where its layout changes (one CTA up to 96
rows, 32- and 16-column blocks around 512 floats per column, products on the
tensor cores from 384 rows) and on spectra that FP32 cannot resolve.  The
bars are those of every eigendecomposition here: 50 n u."""
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


def _matrix(kind, n, cplx):
    rng = np.random.default_rng(n + 7 * cplx)
    X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
    if kind == "gauss":
        return X + X.conj().T
    Q = np.linalg.qr(X)[0]
    if kind == "cluster":  # half of the spectrum within 1e-8 of -1
        ev = np.where(rng.random(n) < 0.5, -1 + 1e-8 * rng.random(n), rng.uniform(-1, 1, n))
    elif kind == "scales":  # gaps over 18 orders of magnitude
        ev = np.cumsum(10.0 ** (-18 * rng.random(n)))
        ev /= ev[-1]
    else:  # three eigenvalues, each many times
        ev = rng.choice([0.25, -0.5, 0.7], n)
    M = (Q * ev) @ Q.conj().T
    return (M + M.conj().T) / 2


@pytest.mark.parametrize("n,cplx,tc", [(2, False, False), (96, False, False), (97, False, False), (520, False, False),
                                       (384, False, True), (96, True, False), (257, True, True)])
@pytest.mark.parametrize("kind", ["gauss", "cluster", "scales", "repeated"])
def test_leaf_eigendecomposition(B, n, cplx, tc, kind):
    M = _matrix(kind, n, cplx)
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        lam, V, info = ctx.heig(to_dev(M))
        lam, V = to_host(lam), to_host(V)
    finally:
        ctx.close()
    assert info["eig_leaves"] == 1  # no split: the whole matrix is one leaf
    nb = np.linalg.norm(M, 2)
    assert np.max(np.abs(lam - np.linalg.eigvalsh(M))) <= 50 * n * U * nb
    assert np.linalg.norm(M @ V - V * lam) <= 50 * n * U * nb
    assert np.linalg.norm(V.conj().T @ V - np.eye(n), 2) <= 50 * n * U


@pytest.mark.parametrize("n,cplx,tc", [(65, False, False), (150, True, False), (330, False, True), (300, True, True)])
@pytest.mark.parametrize("kind", ["gauss", "repeated"])
def test_splits_into_small_leaves(B, n, cplx, tc, kind):
    """Zolo-eig's splits on small blocks (leaves of at most 32 rows): the two
    bases from one inverse Cholesky factor, padded groups of different sizes."""
    M = _matrix(kind, n, cplx)
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        ctx.set_eig_leaf(32)
        lam, V, info = ctx.heig(to_dev(M))
        lam, V = to_host(lam), to_host(V)
    finally:
        ctx.close()
    assert info["eig_splits"] >= 1
    nb = np.linalg.norm(M, 2)
    assert np.max(np.abs(lam - np.linalg.eigvalsh(M))) <= 50 * n * U * nb
    assert np.linalg.norm(M @ V - V * lam) <= 50 * n * U * nb
    assert np.linalg.norm(V.conj().T @ V - np.eye(n), 2) <= 50 * n * U
