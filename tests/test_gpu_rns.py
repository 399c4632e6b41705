"""The tensor-core product (tc_gemm.cu) at the edges of its tiles, stages and
moduli: 128 x 256 tiles, 64-k stages, a reduction mod p every 256 k, a 15th
modulus above 4096 terms, shared operands of a Gram product, rows and columns
of very different size.  Reference: the product of the same integers-by-scaling
bound as tests/test_gpu_control.py, here against a long-double sum on the host
(numpy longdouble or float64 where that is all there is)."""
import numpy as np
import pytest

from tests.gpu_util import U, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _tol(A, B, k):
    """Operands rounded at 2^-57 of their row / column maxima, the sum at FP64
    rounding of the reference (k u sum |a| |b|)."""
    rmax, cmax = np.max(np.abs(A), axis=1)[:, None], np.max(np.abs(B), axis=0)[None, :]
    return 2.0 ** -56 * k * rmax * cmax + (k + 4) * U * (np.abs(A) @ np.abs(B))


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 255, 63), (128, 256, 64), (129, 257, 65), (40, 300, 256),
                                   (130, 20, 257), (64, 64, 4096), (65, 33, 4800), (33, 40, 40000)])
@pytest.mark.parametrize("graded", [False, True])
def test_product_at_the_edges(ctx, m, n, k, graded):
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    if graded:
        A *= 10.0 ** rng.uniform(-150, 150, (m, 1))
        B *= 10.0 ** rng.uniform(-140, 140, (1, n))
        A[0, :] = 0.0
        B[:, n // 2] = 0.0
    got = to_host(ctx.gemm(to_dev(A), to_dev(B), engine=1))
    assert np.all(np.abs(got - A @ B) <= _tol(A, B, k))
    assert np.all(got[0, :] == 0.0) or not graded


def test_gram_product_shares_its_operand(ctx):
    rng = np.random.default_rng(5)
    A = rng.standard_normal((300, 513))
    d = to_dev(A)
    got = to_host(ctx.gemm(d, d, opA=0, opB=1, engine=1))
    assert np.all(np.abs(got - A @ A.T) <= _tol(A, A.T, 513))
    assert np.array_equal(got, got.T)


def test_extreme_integers(ctx):
    """Every entry at the rounding edge of its row maximum and of one sign: the
    sums come as close to P / 2 as they can."""
    m, n, k = 130, 260, 4096
    A = np.full((m, k), 1.0 - 2.0 ** -53)
    B = np.full((k, n), -(1.0 - 2.0 ** -53))
    got = to_host(ctx.gemm(to_dev(A), to_dev(B), engine=1))
    assert np.all(np.abs(got + k) <= k * 2.0 ** -50)
