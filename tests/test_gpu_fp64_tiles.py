"""The FP64-pipe product (blas.cu) at the edges of its tiles: 8 x 8 and 16 x 8
outputs whose k-steps are shared among groups of threads, rows and columns
beyond the edge left out, unit and other alpha.  Reference: numpy, with the
rounding of both sums."""
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


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (7, 9, 5), (8, 8, 32), (9, 17, 33), (65, 31, 15), (64, 64, 64),
                                   (97, 130, 70), (200, 201, 199), (257, 255, 40), (700, 650, 31)])
@pytest.mark.parametrize("opA,opB", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.75, 0.5)])
def test_product_at_the_tile_edges(ctx, m, n, k, opA, opB, alpha, beta):
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    A = rng.standard_normal((k, m) if opA else (m, k))
    B = rng.standard_normal((n, k) if opB else (k, n))
    C = rng.standard_normal((m, n))
    a, b = (A.T if opA else A), (B.T if opB else B)
    got = to_host(ctx.gemm(to_dev(A), to_dev(B), to_dev(C), alpha=alpha, beta=beta, opA=opA, opB=opB, engine=0))
    tol = (2 * k + 8) * U * (abs(alpha) * (np.abs(a) @ np.abs(b)) + abs(beta) * np.abs(C))
    assert np.all(np.abs(got - (alpha * (a @ b) + beta * C)) <= tol)
