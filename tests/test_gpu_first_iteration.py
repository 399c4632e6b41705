"""Zolo-pd's first iteration on the FP64 pipe on both sides of the size from
which it is taken by Householder QR of the stacked matrices (850 rows): the
polar factor of a matrix built from its singular value decomposition, within
the bars that hold everywhere (||W^* W - I||, ||W H - A|| <= 50 n u, W within its
condition)."""
import numpy as np
import pytest

from tests.gpu_util import U, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,cplx", [(849, False), (850, False), (897, False), (850, True)])
@pytest.mark.parametrize("smin", [1e-3, 1e-13])
def test_polar_of_known_factors(n, cplx, smin):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding as B
    rng = np.random.default_rng(n)

    def haar():
        X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
        return np.linalg.qr(X)[0]

    Uo, Vo, s = haar(), haar(), np.geomspace(1.0, smin, n)
    A = to_dev((Uo * s) @ Vo.conj().T)
    ctx = B.Context(0)
    try:
        W, H, info = ctx.polar(A)
    finally:
        ctx.close()
    assert info["zolo_iters"] == 2 and info["chol_fallback"] == 0
    eye = torch.eye(n, dtype=W.dtype, device=W.device)
    assert float(torch.linalg.matrix_norm(W.mH @ W - eye, 2)) <= 50 * n * U
    assert float(torch.linalg.matrix_norm(W @ H - A)) <= 50 * n * U
    assert float(torch.linalg.matrix_norm(W - to_dev(Uo @ Vo.conj().T))) <= 50 * n * U / smin
