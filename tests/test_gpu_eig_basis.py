"""The bases of a Zolo-eig split when the random start matrix Omega is a bad
draw: the first k columns of P Omega (nearly) dependent.  Omega is the library's
own (a counter-based generator with a fixed seed, restated here), the
eigenvectors are chosen to meet it."""
import numpy as np
import pytest

from tests.gpu_util import U, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SEED = 0x5EED + 1  # depth 0, first attempt, first group


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    return binding


def _omega(n):
    M = (1 << 64) - 1
    base = np.uint64((SEED * 0x100000001B3) & M)

    def mix(z):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) + 0.5

    with np.errstate(over="ignore"):
        t = base + np.uint64(2) * np.arange(n * n, dtype=np.uint64)
        u1, u2 = mix(t) * 2.0 ** -53, mix(t + np.uint64(1)) * 2.0 ** -53
    return (np.sqrt(-2 * np.log(u1)) * np.cos(2 * np.pi * u2)).reshape(n, n).T  # column-major


@pytest.mark.parametrize("eps,width", [(0.0, 1.0), (1e-7, 1.0), (1e-7, 1e-5)])
def test_bad_draw_of_omega(B, eps, width):
    """range(P) within eps of orthogonal to a combination of the first k
    columns of Omega.  With all eigenvalues in a cluster of relative width
    1e-5 the off-block test, which is relative to ||B||, does not see an
    inaccurate basis.  Neither costs another shift, and the eigenvectors are
    orthonormal."""
    n, k = 130, 50
    rng = np.random.default_rng(1)
    y = _omega(n)[:, :k] @ rng.standard_normal(k)
    y /= np.linalg.norm(y)
    Q = np.linalg.qr(np.column_stack([y, rng.standard_normal((n, n - 1))]))[0]
    y = Q[:, 0].copy()
    r = Q[:, 1].copy()
    Q[:, 0], Q[:, 1] = np.cos(eps) * r + np.sin(eps) * y, np.cos(eps) * y - np.sin(eps) * r
    cols = np.r_[0, 2:n, 1]  # the first k of these span range(P): r (tilted by eps) and others orthogonal to y
    ev = np.concatenate([(n - k) / k + 0.2 * rng.uniform(-1, 1, k), -1 + 0.2 * rng.uniform(-1, 1, n - k)])
    if width != 1.0:
        ev = 1.0 + width * ev
    M = (Q[:, cols] * ev) @ Q[:, cols].T
    M = (M + M.T) / 2
    ctx = B.Context(0)
    try:
        ctx.set_eig_leaf(96)
        lam, V, info = ctx.heig(to_dev(M))
        lam, V = to_host(lam), to_host(V)
    finally:
        ctx.close()
    nb = np.linalg.norm(M, 2)
    assert np.linalg.norm(V.T @ V - np.eye(n), 2) <= 50 * n * U
    assert np.linalg.norm(M @ V - V * lam) <= 50 * n * U * nb
    assert np.max(np.abs(lam - np.linalg.eigvalsh(M))) <= 50 * n * U * nb
    assert info["eig_splits"] == 1 and info["eig_retries"] == 0
