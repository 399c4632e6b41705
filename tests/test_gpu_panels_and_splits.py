"""Paths that the default settings reach only at sizes beyond the other tests:
Householder panels of every height (a CTA below 256 rows, clusters of 4 and 8
CTAs in shared memory, a cluster of 8 on global memory above 6400 real or 3200
complex rows), and Zolo-eig's splits at 1024 rows (the default leaf is that
large) with either product engine and with fewer operand bits inside."""
import numpy as np
import pytest

from paper_1804_09002_gb300 import inputs as I
from tests.gpu_util import U, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    return binding


def _check(A1, A2, R, th, n):
    r = R["rank"]
    got = R["theta"][:r]
    assert r == len(th)
    assert float((got.cpu() - torch.from_numpy(np.sort(th))).abs().max()) <= 1e-12 * n
    c, s = torch.cos(got), torch.sin(got)
    U1, U2, V1 = (R[k][:, :r] for k in ("U1", "U2", "V1"))
    c, s = c.to(V1.dtype), s.to(V1.dtype)
    be = torch.sqrt(torch.linalg.norm(A1 - (U1 * c) @ V1.mH) ** 2 + torch.linalg.norm(A2 - (U2 * s) @ V1.mH) ** 2)
    assert float(be) / np.sqrt(r) <= 50 * n * U
    for X in (U1, U2, V1):
        assert float(torch.linalg.matrix_norm(X.mH @ X - torch.eye(r, dtype=X.dtype, device=X.device), 2)) <= 50 * n * U


@pytest.mark.parametrize("m1,m2,n,cplx", [(300, 1030, 40, False), (257, 3000, 33, False), (7000, 40, 40, False),
                                          (260, 1100, 33, True), (3500, 64, 64, True)])
def test_rectangular_blocks_of_every_panel_height(B, m1, m2, n, cplx):
    rng = np.random.default_rng(m1)

    def basis(m):
        X = rng.standard_normal((m, n)) + (1j * rng.standard_normal((m, n)) if cplx else 0)
        return np.linalg.qr(X)[0]

    th = rng.uniform(0, np.pi / 2, n)
    V = basis(n)
    A1, A2 = to_dev((basis(m1) * np.cos(th)) @ V.conj().T), to_dev((basis(m2) * np.sin(th)) @ V.conj().T)
    _check(A1, A2, B.default_context(0).csd_polar_rect(A1, A2), th, n)


@pytest.mark.parametrize("tc,slices,scope", [(False, 7, 0), (True, 7, 0), (True, 6, 3), (True, 5, 1)])
def test_csd_n1024_in_leaves_of_256(B, tc, slices, scope):
    n = 1024
    A1, A2, th = I.clustered_csd(n, seed=2)
    A1, A2 = to_dev(A1), to_dev(A2)
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        ctx.set_eig_leaf(256)
        ctx.set_mixed_precision(slices, scope)
        R = ctx.csd_polar(A1, A2)
        assert R["info"]["eig_splits"] >= 3
    finally:
        ctx.close()
    _check(A1, A2, R, th, n)
